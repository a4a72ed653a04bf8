"""A call reads what it is given -- ids and weights as well as hidden states and
payload -- only after the caller's kernel before it in the stream has written it, also where that kernel
lets its dependents start early (programmatic dependent launch), as kernels of
other libraries do.  The writer here does so and writes 50 us later; both the
old and the new contents are valid, so a call that did not wait would answer
from the old ones.  Needs a GPU (marked gpu)."""
import ctypes
import subprocess

import pytest
import torch

from paper_2607_13093_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"
SOURCE = """
__global__ void late_copy(int* dst, const int* src, long long words, long long cycles) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) { }
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < words;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = src[i];
}
extern "C" int late_copy_launch(void* dst, const void* src, long long words, void* stream) {
  late_copy<<<8, 256, 0, (cudaStream_t)stream>>>((int*)dst, (const int*)src, words, 100000);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def writer(tmp_path_factory):
    from paper_2607_13093_gb300 import build_lib
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(SOURCE)
    subprocess.run([build_lib.nvcc(), *build_lib.ARCH, "-O2", "-shared", "-cudart", "shared",
                    "-Xcompiler", "-fPIC", str(d / "late.cu"), "-o", str(d / "late.so")],
                   check=True)
    f = ctypes.CDLL(str(d / "late.so")).late_copy_launch
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p]

    def write(dst, src):
        nbytes = dst.numel() * dst.element_size()
        assert dst.is_contiguous() and src.is_contiguous() and nbytes % 4 == 0
        assert f(dst.data_ptr(), src.data_ptr(), nbytes // 4,
                 torch.cuda.current_stream().cuda_stream) == 0
    return write


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_13093_gb300 import build_lib
    build_lib.build()
    from paper_2607_13093_gb300 import sph
    c = sph.Context(0)
    yield c
    c.close()


# rows: the GEMV, the few-row endpoint kernel, the general tensor-core kernel
# on single CTAs and on pairs
@pytest.mark.parametrize("rows", [2, 16, 48, 256])
@pytest.mark.parametrize("late", ["keep_ids", "weights", "full", "hidden", "payload"])
@pytest.mark.parametrize("call", ["cloud", "endpoint", "logits", "step", "streamed", "serial",
                                  "verify"])
def test_call_reads_after_the_callers_kernel(ctx, writer, call, late, rows):
    if (call == "verify" and late != "keep_ids") or (
            late == "payload" and call not in ("endpoint", "logits")):
        pytest.skip("the call takes no such input")
    # ("full": the weights of a call over the whole vocabulary, without ids)
    V, n, k = 3000 if late == "full" else 6000, 3000, 1
    w = wl.make_workload(V=V, d=640, d_l=128, rows=rows, n_keep=n, seed=71, device=DEV, k=k,
                         sessions=rows // (k + 1))
    pc, ps = wl.make_payload(rows, n, seed=3, device=DEV)
    zt = torch.randn(rows, n, device=DEV)
    ids = None if late == "full" else w.keep_ids.clone()
    old_ids = torch.arange(n, dtype=torch.int32, device=DEV)
    codes, tok = (torch.empty(s, dtype=t, device=DEV)
                  for s, t in ((rows * n, torch.int8), (rows, torch.int32)))
    scale = torch.empty(3 * rows, device=DEV)
    z = torch.empty(rows, n, device=DEV)
    acc, nxt = (torch.empty(rows // (k + 1), dtype=torch.int32, device=DEV) for _ in range(2))
    es = torch.cuda.Stream()
    cur = torch.cuda.current_stream().cuda_stream

    def run():
        kw = dict(keep_ids=ids, temperature=0.8, seed=9, offset=2)
        if call == "cloud":
            ctx.partial_logits(w.h_cloud, w.W_h, keep_ids=ids, codes=codes.view(rows, n),
                               row_scale=scale[:rows], partial_out=z)
            return codes, scale[:rows], z
        if call == "endpoint":
            return (ctx.fuse_sample(pc, ps, w.h_local, w.W_l, tokens=tok, fused_logits_out=z,
                                    **kw), z)
        if call == "logits":
            ctx.fuse_sample(pc, ps, w.h_local, w.W_l, draw=False, fused_logits_out=z, **kw)
            return (z,)
        if call == "verify":
            ctx.verify_draft(zt, rows // (k + 1), k, w.draft_tokens, n_accepted=acc,
                             next_token=nxt, **kw)
            return acc, nxt
        ctx.split_step(w.h, w.d_l, w.W_h, w.W_l, codes=codes, scales=scale, tokens=tok,
                       fused_logits_out=z, chunk=0 if call == "step" else n // 3,
                       endpoint_stream={"streamed": es.cuda_stream, "serial": cur}.get(call),
                       **kw)
        return codes, tok, z

    def snapshot():
        out = [t.clone() for t in run()]
        torch.cuda.synchronize()
        return out

    # the weights are those of the call's last contraction (streamed: written on
    # the endpoint's own stream, which the call's endpoint half follows)
    if late == "keep_ids":
        dst, new, old = ids, w.keep_ids, old_ids
    else:
        # before the write: one row further on
        dst = {"payload": pc, "hidden": w.h}.get(late, w.W_h if call == "cloud" else w.W_l)
        new, old = dst.clone(), dst.roll(1, 0).contiguous()
    want = snapshot()
    dst.copy_(old)
    was = snapshot()
    assert any(not torch.equal(a, b) for a, b in zip(want, was))
    on_es = call == "streamed" and late in ("weights", "full")
    for _ in range(3):
        dst.copy_(old)
        torch.cuda.synchronize()
        with torch.cuda.stream(es if on_es else torch.cuda.current_stream()):
            writer(dst, new)
        got = snapshot()
        same = [torch.equal(a, b) for a, b in zip(got, want)]
        stale = [torch.equal(a, b) for a, b in zip(got, was)]
        assert all(same), (same, stale)
    ctx.sync()
