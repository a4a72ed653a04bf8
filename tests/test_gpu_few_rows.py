"""The endpoint's few-row kernel (4..32 rows over at most 512 columns) at the
edges of its tiles, turns, rows and columns, against the oracle and, bit for
bit, against the general tensor-core kernel it takes over from (both add in
the same order over whole tiles).  Needs a GPU (marked gpu)."""
import pytest
import torch

from paper_2607_13093_gb300 import workloads as wl
from _parity import check_endpoint

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph
    c = sph.Context(0)
    yield c
    c.close()


def general(ctx, f):
    """f() on the general kernel."""
    from paper_2607_13093_gb300 import sph
    ctx.set_option(sph.SPH_OPT_FEW_ROWS, 1)
    try:
        return f()
    finally:
        ctx.set_option(sph.SPH_OPT_FEW_ROWS, 0)


def z_launches(ctx, w):
    z = torch.empty(w.rows, w.n_keep, device=DEV)
    ctx.profile_enable(True)
    ctx.fuse_sample(None, None, w.h_local, w.W_l, keep_ids=w.keep_ids, draw=False,
                    fused_logits_out=z)
    ctx.sync()
    n = ctx.profile_read()["launches"]
    ctx.profile_enable(False)
    return n


# options of other calls and kernels leave the kernel to it; those that shape
# the general one choose that (name, value, default, few-row kernel or not)
@pytest.mark.parametrize("name,value,default,few", [
    ("FEW_ROWS", 0, 0, True), ("TC_FINISH_WAIT", 0, 1 << 15, True), ("TC_MIN_ROWS", 1, 4, True),
    ("TC_MIN_ROWS", 16, 4, True), ("TC_PAIR", 2, 0, True), ("ENDPOINT_ROWS_M", 1, 0, True),
    ("ENDPOINT_Z", 1, 0, True), ("FEW_ROWS", 1, 0, False), ("TC_STAGES", 3, 0, False),
    ("TC_SCHEDULE", 1, 0, False), ("TC_BLOCK_K", 64, 0, False), ("TC_MAX_BN", 16, 0, False),
    ("TC_TILE_M", 128, 0, False), ("TC_PAIR", 1, 0, False), ("ENDPOINT_Z", 2, 0, False)])
def test_which_options_choose_the_general_kernel(ctx, name, value, default, few):
    from paper_2607_13093_gb300 import sph
    opt = getattr(sph, "SPH_OPT_" + name)
    ctx.set_option(opt, value)
    try:
        got = ctx.plan(1, 16, 12000, 256)["tile_ids"]
    finally:
        ctx.set_option(opt, default)
    # 12000 ids: 125 tiles of 96 in one turn of the SMs; the general kernel's
    # tiles have 128 or 256
    assert (got == 96) if few else got in (128, 256)
    with pytest.raises(sph.SphError):
        ctx.set_option(sph.SPH_OPT_FEW_ROWS, 2)


@pytest.mark.parametrize("rows,n,V,K,few", [
    (32, 58368, 70000, 512, True),                   # 456 tiles: three an SM
    (32, 58369, 70000, 512, False), (17, 77824, 90000, 392, False), (16, 77824, 90000, 392, True),
    (16, 77824, 77824, 392, False), (32, 77824, 77824, 384, True), (12, 45000, 45000, 512, True),
    (4, 77824, 90000, 520, False)])
def test_the_lines_over_long_hidden_dimensions(ctx, rows, n, V, K, few):
    # three turns of the 152 SMs, 16 rows, a subset or the full vocabulary
    w = wl.make_workload(V=V, d=K + 8, d_l=K, rows=rows, n_keep=n, seed=n, device=DEV)
    assert (w.keep_ids is None) == (n == V)
    g = general(ctx, lambda: ctx.plan(1, rows, n, K, gather=n < V))
    assert (z_launches(ctx, w) == 1) == (few and g["whole_tiles"] == 1)


# rows (4, both sides of 16, 32), kept ids (segments, tiles and SM turns: one
# turn of 152 tiles ends at 19456 ids), columns (atoms of 64, stages of 128)
CASES = [(4, 1, 48), (5, 31, 8), (16, 33, 64), (17, 128, 65), (32, 129, 128), (31, 700, 96),
         (8, 4864, 130), (32, 4865, 200), (12, 19456, 63), (9, 19457, 16), (32, 60000, 96),
         (6, 40001, 256), (16, 30011, 512), (32, 12000, 512)]


@pytest.mark.parametrize("rows,n,K", CASES)
@pytest.mark.parametrize("payload", [True, False])
def test_few_rows(ctx, rows, n, K, payload):
    V = max(n + n // 3, 64)
    w = wl.make_workload(V=V, d=K + 24, d_l=K, rows=rows, n_keep=n, tau=0.8, seed=900 + n + K,
                         device=DEV, run_lo=1 if n < 64 else 16, run_hi=3 if n < 64 else 256)
    if K % 8:        # weight rows of a padded stride, junk past the columns
        Wp = torch.full((V, (K + 7) // 8 * 8), float("nan"), dtype=torch.bfloat16, device=DEV)
        Wp[:, :K] = w.W_l
        w.W_l = Wp[:, :K]
    pc, ps = wl.make_payload(rows, n, seed=3, device=DEV) if payload else (None, None)

    def run():
        z = torch.full((rows, n), 7.0, device=DEV)
        t = ctx.fuse_sample(pc, ps, w.h_local, w.W_l, keep_ids=w.keep_ids, temperature=w.tau,
                            seed=w.seed, offset=5, fused_logits_out=z)
        g = ctx.fuse_sample(pc, ps, w.h_local, w.W_l, keep_ids=w.keep_ids, temperature=0.0)
        y = torch.full((rows, n), 7.0, device=DEV)
        ctx.fuse_sample(pc, ps, w.h_local, w.W_l, keep_ids=w.keep_ids, draw=False,
                        fused_logits_out=y)
        ctx.sync()
        return z, t, g, y

    # one launch for z alone on this kernel, two (operand split) on the general
    assert z_launches(ctx, w) == 1 and general(ctx, lambda: z_launches(ctx, w)) == 2
    a, b = run(), general(ctx, run)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    assert torch.equal(a[0], a[3])
    if payload and K % 8 == 0:
        check_endpoint(ctx, w, pc.cpu(), ps.cpu(), unstored=False)


@pytest.mark.parametrize("rows,n,chunk", [(19, 11987, 0), (4, 3001, 0), (32, 30000, 10000)])
def test_few_rows_one_call(ctx, rows, n, chunk):
    # the fused quantizing epilogue, and the endpoint of a block-streamed
    # payload, against the general kernel; hidden states in rows that are not
    # 16-byte aligned
    w = wl.make_workload(V=n + 999, d=640, d_l=256, rows=rows, n_keep=n, seed=31, device=DEV)
    hp = torch.zeros(rows, 641, device=DEV)
    for h in (w.h, hp[:, 1:].copy_(w.h)):
        def run():
            z = torch.empty(rows, n, device=DEV)
            c, s, t, _ = ctx.split_step(h, w.d_l, w.W_h, w.W_l, keep_ids=w.keep_ids,
                                        temperature=0.9, seed=4, chunk=chunk, fused_logits_out=z)
            ctx.sync()
            return c, s, t, z
        for x, y in zip(run(), general(ctx, run)):
            assert torch.equal(x, y)


@pytest.mark.parametrize("rows,n,K", [(4, 700, 48), (32, 30000, 256), (12, 44999, 512)])
def test_few_rows_wait_timeout_is_reported_and_context_recovers(ctx, rows, n, K):
    # with a limit of one cycle a wait is looked at once: the MMA warp's for
    # the hidden states, which are still on their way from memory, gives up
    from paper_2607_13093_gb300 import sph
    w = wl.make_workload(V=n + n // 3, d=K + 8, d_l=K, rows=rows, n_keep=n, device=DEV, seed=93)
    pc, ps = wl.make_payload(w.rows, w.n_keep, seed=3, device=DEV)
    z = torch.empty(w.rows, w.n_keep, device=DEV)

    def fuse():
        ctx.fuse_sample(pc, ps, w.h_local, w.W_l, keep_ids=w.keep_ids, draw=False,
                        fused_logits_out=z)
        ctx.sync()
        return z.clone()

    want = fuse()
    for _ in range(5):
        ctx.set_option(sph.SPH_OPT_SPIN_LIMIT, 1)
        try:
            with pytest.raises(sph.SphError) as err:
                fuse()
        finally:
            ctx.set_option(sph.SPH_OPT_SPIN_LIMIT, 1 << 34)
        assert err.value.status == 4, str(err.value)
        assert torch.equal(fuse(), want)
