"""e4m3 weights on CTA pairs with row blocks past 128 rows (the h planes two to
a stage): the same bits as single CTAs, at ragged rows, ids and columns.
Needs a GPU (marked gpu)."""
import pytest
import torch

from paper_2607_13093_gb300 import workloads as wl
from _parity import check_cloud

pytestmark = pytest.mark.gpu
DEV = "cuda"


# one block of 160 or 192 rows, two of 160, 192 and 224, on whole tiles
@pytest.mark.parametrize("rows,four,two", [(128, 0, 0), (130, 0, 1), (160, 0, 1), (161, 1, 1),
                                           (192, 1, 1), (256, 1, 1), (257, 0, 0), (384, 0, 0),
                                           (385, 1, 1), (1024, 1, 1)])
def test_which_row_blocks_pair(rows, four, two):
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph
    ctx = sph.Context(0)
    for act, pair in ((sph.SPH_ACT_FP32, four), (sph.SPH_ACT_BF16, two)):
        p = ctx.plan(0, rows, 152064, 7168, w_dtype=sph.SPH_DTYPE_FP8_E4M3, act_mode=act,
                     gather=False)
        assert p["whole_tiles"] == 1 and p["pair"] == pair
    ctx.close()


# rows (one 256-row block short of, at and past its end), kept ids (256-id
# tiles: short, ragged, whole), hidden columns (128-column blocks, ragged)
@pytest.mark.parametrize("rows,keep,d_h", [(225, 3000, 256), (256, 2999, 1008), (250, 257, 128),
                                           (480, 700, 400), (513, 1100, 1024), (190, 1500, 528)])
@pytest.mark.parametrize("act", ["fp32", "bf16"])
def test_wide_row_blocks_on_pairs(rows, keep, d_h, act):
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph
    ctx = sph.Context(0)
    w = wl.make_workload(V=3000, d=d_h + 16, d_l=16, rows=rows, n_keep=keep, w_dtype="fp8",
                         clip=40.0, seed=61 + rows, device=DEV, with_bias=rows == 480)
    a = sph.SPH_ACT_BF16 if act == "bf16" else sph.SPH_ACT_FP32
    ctx.set_option(sph.SPH_OPT_TC_SCHEDULE, 1)          # whole tiles on both
    out = []
    for mode in (2, 1):
        ctx.set_option(sph.SPH_OPT_TC_PAIR, mode)
        p = ctx.plan(0, rows, keep, d_h, w_dtype=sph.SPH_DTYPE_FP8_E4M3, act_mode=a,
                     gather=w.keep_ids is not None)
        assert p["pair"] == (mode == 1) and (mode == 2 or p["block_rows"] > 128)
        y = torch.empty(rows, keep, device=DEV)
        c, s, _ = ctx.partial_logits(w.h_cloud, w.W_h, keep_ids=w.keep_ids, clip=w.clip,
                                     w_row_scale=w.w_scale, bias=w.bias, act_mode=a, partial_out=y)
        ctx.sync()
        out.append((y, c, s))
    for x, y in zip(*out):
        assert torch.equal(x, y)
    check_cloud(ctx, w, act_mode=act)
    ctx.close()
