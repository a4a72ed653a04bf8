"""The one-launch draw of short stored rows (at most 16 rows of at most 8192
ids on the GEMV endpoint) at the edges of its segments, chunks, rows and
alignments: against the oracle, and token for token against the draw through
the statistics pass, which the same rows take in a call of more than 16 rows.
Needs a GPU (marked gpu)."""
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
    c.set_option(sph.SPH_OPT_TC_MIN_ROWS, 1 << 20)     # every row count on the GEMV
    yield c
    c.close()


@pytest.mark.parametrize("rows,n", [(1, 1), (2, 31), (3, 33), (1, 1023), (2, 1025), (16, 2048),
                                    (3, 4097), (1, 8191), (3, 8190), (16, 8192), (2, 8193),
                                    (17, 700)])
@pytest.mark.parametrize("tau", [0.8, 0.0])
def test_short_draw(ctx, rows, n, tau):
    K = 64
    w = wl.make_workload(V=n + n // 3 + 64, d=K + 24, d_l=K, rows=rows, n_keep=n, tau=tau,
                         seed=500 + n, device=DEV, run_lo=1 if n < 64 else 16,
                         run_hi=3 if n < 64 else 256)
    pc, ps = wl.make_payload(rows, n, seed=3, device=DEV)
    check_endpoint(ctx, w, pc.cpu(), ps.cpu(), unstored=False)
    # the same rows among 17 and more: equal logits and equal tokens
    m = 17 + rows
    pcm, psm = wl.make_payload(m, n, seed=4, device=DEV)
    hm = torch.randn(m, K, device=DEV)
    pcm[:rows], psm[:rows], hm[:rows] = pc, ps, w.h_local
    for seed in range(8):
        out = []
        for c, s, h in ((pc, ps, w.h_local), (pcm, psm, hm)):
            z = torch.empty(len(h), n, device=DEV)
            t = ctx.fuse_sample(c, s, h, w.W_l, keep_ids=w.keep_ids, temperature=tau, seed=seed,
                                offset=9, fused_logits_out=z)
            ctx.sync()
            out.append((z[:rows].clone(), t[:rows].clone()))
        assert torch.equal(out[0][0], out[1][0])
        assert torch.equal(out[0][1], out[1][1])
