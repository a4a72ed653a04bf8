"""Payloads whose rows of codes start anywhere: the transposed endpoint (rows at
even addresses) and the rows-as-M one (at any) fetch them as the aligned words
that hold them; rows at odd addresses with ids as M take the per-lane epilogue.
The same bits for every base address, and the oracle's values.  Needs a GPU
(marked gpu)."""
import pytest
import torch

from paper_2607_13093_gb300 import workloads as wl
from _parity import check_endpoint

pytestmark = pytest.mark.gpu
DEV = "cuda"


# 160 rows: ids as M, through the transpose at the even shifts (the number of
# ids is even), lane by lane at the odd ones; 250: rows as M at all of them.  Ids: whole 32-id segments, and last segments of 1, 8, 10 and 31 ids;
# divisible by 16, 8, 4, 2 and 1
@pytest.mark.parametrize("rows,n", [(160, 1024), (160, 1032), (160, 1034), (160, 1036), (250, 1024),
                                    (250, 1032), (250, 1034), (250, 1055), (250, 1025)])
def test_code_rows_at_any_address(rows, n):
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph
    ctx = sph.Context(0)
    w = wl.make_workload(V=2000, d=160, d_l=64, rows=rows, n_keep=n, seed=n, device=DEV, tau=0.9)
    pc, ps = wl.make_payload(rows, n, seed=5, device=DEV)
    check_endpoint(ctx, w, pc.cpu(), ps.cpu(), unstored=False)
    outs = []
    for shift in (0, 1, 2, 4, 6, 8, 13, 15):
        buf = torch.full((rows * n + 32,), 77, dtype=torch.int8, device=DEV)
        codes = buf[shift:shift + rows * n].view(rows, n)
        codes.copy_(pc)
        z = torch.empty(rows, n, device=DEV)
        ctx.fuse_sample(codes, ps, w.h_local, w.W_l, keep_ids=w.keep_ids, draw=False,
                        fused_logits_out=z)
        t = ctx.fuse_sample(codes, ps, w.h_local, w.W_l, keep_ids=w.keep_ids, temperature=0.9,
                            seed=3, offset=shift)
        g = ctx.fuse_sample(codes, ps, w.h_local, w.W_l, keep_ids=w.keep_ids, temperature=0.0)
        ctx.sync()
        outs.append((z, g))
        assert t.min() >= 0
    for z, g in outs[1:]:
        assert torch.equal(z, outs[0][0]) and torch.equal(g, outs[0][1])
    ctx.close()


@pytest.mark.parametrize("rows,n,K", [(250, 1034, 512), (250, 1034, 520), (250, 1034, 1024),
                                      (256, 25602, 1024), (256, 25602, 1032), (250, 1055, 2048),
                                      (4, 1034, 1024), (15, 1024, 2048), (17, 1055, 1024)])
def test_code_rows_over_long_hidden_dimensions(rows, n, K):
    # both sides of the lines at which rows off 16 bytes are fetched as words
    # (512 columns; 1024 with more tiles than CTA pairs), and the per-lane
    # epilogue's row chunks that are not full, on whole and on split tiles
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph
    ctx = sph.Context(0)
    w = wl.make_workload(V=n + 3000, d=K + 64, d_l=K, rows=rows, n_keep=n, seed=n, device=DEV,
                         tau=0.9)
    pc, ps = wl.make_payload(rows, n, seed=5, device=DEV)
    check_endpoint(ctx, w, pc.cpu(), ps.cpu(), rows=[0, rows // 2, rows - 1])
    ctx.close()
