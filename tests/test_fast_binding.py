"""The native argument marshalling (csrc/py_fast.cpp) takes plain calls and
leaves the rest to the Python checks: same results either way, same errors."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2607_13093_gb300 import workloads as wl


@pytest.fixture(scope="module")
def sph():
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph as m
    return m


def test_anything_not_plain_is_left_to_python(sph):
    # nothing here may reach the library: host tensors, a missing handle,
    # wrong argument counts and types
    f, no = sph._fast, sph._NOT_TAKEN
    h, W = torch.zeros(2, 16), torch.zeros(8, 16, dtype=torch.bfloat16)
    codes, scale = torch.zeros(2, 8, dtype=torch.int8), torch.zeros(2)
    tok = torch.zeros(2, dtype=torch.int32)
    for handle in (None, 0, 1, 1.5, object()):
        assert f.partial_logits(handle, h, W, None, 30.0, None, None, 0, codes, scale, None) == no
        assert f.fuse_sample(handle, codes, scale, h, W, None, 1.0, 1, 2, tok, None) == no
        assert f.split_step(handle, h, 8, W, W, None, 30.0, None, None, 0, 1.0, 1, 2, 0, 0, codes,
                            scale, tok) == no
        assert f.verify_draft(handle, h, 1, 1, tok, None, None, 1.0, 1, 2, tok, tok) == no
    for call in (f.partial_logits, f.fuse_sample, f.split_step, f.verify_draft):
        assert call() == no and call(1, h) == no and call(*[None] * 11) == no
        assert call(*[object()] * 18) == no
    with pytest.raises(RuntimeError):
        f.bind("/nonexistent/libsph.so")
    # the Python path still has the last word
    with pytest.raises(ValueError, match="CUDA tensor"):
        sph.sph_partial_logits(None, h, W, codes=codes, row_scale=scale)
    with pytest.raises(ValueError, match="CUDA tensor"):
        sph.sph_verify_draft(None, h, 1, 1, tok, n_accepted=tok, next_token=tok)


NO_STORAGE = """
import sys
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2607_13093_gb300 import sph

f, got, bf = sph._fast, [], torch.bfloat16

def call(h):          # plain CUDA tensors by type, device and shape, without storage
    W, n = h.to(bf), h.to(torch.int32)
    assert type(h) is torch.Tensor and h.is_cuda
    got.append({
        "partial": lambda: f.partial_logits(1, h, W, None, 30.0, None, None, 0, None, None, None),
        "fuse": lambda: f.fuse_sample(1, None, None, h, W, None, 1.0, 1, 2, None, None),
        "split": lambda: f.split_step(1, h, 8, W, W, None, 30.0, None, None, 0, 1.0, 1, 2, 0, 0,
                                      None, None, None),
        "verify": lambda: f.verify_draft(1, h, 1, 1, n, None, None, 1.0, 1, 2, n, n),
    }[sys.argv[1]]())
    return h

with FakeTensorMode():
    torch.vmap(call)(torch.empty(3, 2, 16, device="cuda"))
assert got == [sph._NOT_TAKEN], got
"""


@pytest.mark.parametrize("call", ["partial", "fuse", "split", "verify"])
def test_a_tensor_without_storage_is_left_to_python(sph, call):
    # (a process of its own: asking such a tensor for its address throws, and
    # an exception without the interpreter lock ends the interpreter)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", NO_STORAGE, call], cwd=root, capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr


@pytest.mark.gpu
@pytest.mark.parametrize("keep,bias,act", [(700, True, 0), (1500, False, 1)])
def test_native_and_python_marshalling_agree(sph, keep, bias, act):
    # a numpy integer is not plain, so the call goes through Python
    S, k = 4, 2
    w = wl.make_workload(V=1500, d=320, d_l=64, rows=S * (k + 1), n_keep=keep, seed=5,
                         device="cuda", sessions=S, k=k, with_bias=bias)
    ctx = sph.Context(0)
    R, n, dev = w.rows, w.n_keep, "cuda"
    out = []
    for num in (int, np.int64):
        codes = torch.empty(R, n, dtype=torch.int8, device=dev)
        scale, y, z = (torch.empty(s, device=dev) for s in ((R,), (R, n), (R, n)))
        tok, stok = (torch.empty(R, dtype=torch.int32, device=dev) for _ in range(2))
        acc, nxt = (torch.empty(S, dtype=torch.int32, device=dev) for _ in range(2))
        sc, ss = torch.empty(R * n, dtype=torch.int8, device=dev), torch.empty(3 * R, device=dev)
        r = ctx.partial_logits(w.h_cloud, w.W_h, keep_ids=w.keep_ids, clip=w.clip, bias=w.bias,
                               act_mode=num(act), codes=codes, row_scale=scale, partial_out=y)
        assert r[0] is codes and r[1] is scale and r[2] == R * n + 4 * R
        assert ctx.fuse_sample(codes, scale, w.h_local, w.W_l, keep_ids=w.keep_ids,
                               temperature=0.9, seed=num(3), offset=num(4), tokens=tok,
                               fused_logits_out=z) is tok
        ctx.verify_draft(z, S, k, w.draft_tokens, keep_ids=w.keep_ids, draft_probs=w.draft_probs,
                         temperature=0.9, seed=num(3), offset=num(5), n_accepted=acc,
                         next_token=nxt)
        r = ctx.split_step(w.h, w.d_l, w.W_h, w.W_l, keep_ids=w.keep_ids, clip=w.clip,
                           bias=w.bias, act_mode=num(act), temperature=0.9, seed=num(3),
                           offset=num(6), chunk=(n + 2) // 3, codes=sc, scales=ss, tokens=stok)
        assert r[3] == R * n + 12 * R
        ctx.sync()
        out.append([t.clone() for t in (codes, scale, y, tok, z, acc, nxt, sc, ss, stok)])
    for a, b in zip(*out):
        assert torch.equal(a, b)
    # the library's and the binding's errors come through
    codes = torch.empty(R, n, dtype=torch.int8, device=dev)
    scale = torch.empty(R, device=dev)
    with pytest.raises(sph.SphError):
        ctx.partial_logits(w.h_cloud, w.W_h, keep_ids=w.keep_ids, clip=0.0, codes=codes,
                           row_scale=scale)
    with pytest.raises(ValueError, match="elements"):
        ctx.partial_logits(w.h_cloud, w.W_h, keep_ids=w.keep_ids, codes=codes,
                           row_scale=scale[:-1])
    with pytest.raises(ValueError, match="contiguous"):
        ctx.partial_logits(w.h_cloud, w.W_h, keep_ids=w.keep_ids, codes=codes.t(),
                           row_scale=scale)
    ctx.close()
