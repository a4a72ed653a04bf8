"""Performance cases of the split-head vocabulary projection.

Every case is work that a program using this package has it do through the
public entry points of `paper_2607_13093_gb300.sph`: the cloud's partial
logits and their int8 payload, the endpoint's fuse-and-sample call, the
verification of speculative drafts, and the one-call split step.  Sizes are
those of the package's workloads (its configurations) and ragged ones around
them.

`prepare` gives what such a program keeps (a context whose scratch is
reserved, weights, output buffers) and what it has in hand before a call
(hidden states, the kept ids, drafts, a payload that arrived); `run` is one
pass through the calls; `exact` is the same mathematics in 64 bits by plain
torch.
"""
from __future__ import annotations

import math

import torch

from paper_2607_13093_gb300 import sph, workloads as wl

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
# Keys (with their defaults):
#   kind     step     cloud call, then endpoint call with its draw
#            onecall  the whole split step in one call (chunk: ids per payload
#                     block, 0 = one block)
#            spec     cloud call, endpoint call that returns the fused target
#                     logits, verification of k drafts per session
#            cloud    the cloud call alone (the cloud's half, as it runs where
#                     the endpoint is another machine)
#            endpoint the endpoint call alone, on a payload that arrived,
#                     returning the fused logits beside the tokens
#            unsplit  the head that is not split: the endpoint call over the
#                     whole hidden state without a payload, returning the
#                     logits beside the tokens
#   V, n     vocabulary and kept ids (n == V: no subset)
#   d, d_l   hidden dimension and the endpoint's share of it
#   rows     hidden-state rows (spec: sessions * (k + 1))
#   act      activations of the cloud call: fp32 or bf16
#   w        cloud weights: bf16, or fp8 (e4m3 with a scale per row)
#   tau      temperature (0: greedy)
#   bias     cloud bias; logits: the cloud call also returns its unclipped
#            partial logits; sampler: cdf or gumbel; probs: drafts with their
#            distributions (else greedy drafts)
DEFAULTS = dict(kind="step", V=32000, n=12000, d=4096, d_l=256, rows=32, act="fp32", w="bf16",
                tau=1.0, clip=30.0, bias=False, logits=False, sampler="cdf", chunk=0,
                sessions=0, k=0, probs=True)


def _case(name=None, **kw):
    c = dict(DEFAULTS, **kw)
    if c["kind"] == "spec":
        c["rows"] = c["sessions"] * (c["k"] + 1)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one row of a small model: a single interactive session on a small
        # head; launches and host time are all there is
        _case("tiny_step", V=8192, n=2048, d=512, d_l=64, rows=1),
        # the everyday decode step of a served batch over a language subset
        _case("decode_step", V=32000, n=12000, d=4096, d_l=256, rows=32, tau=0.8),
        # the same service with a ragged batch, as one call, from a decoder
        # that hands over bf16 states: biased head, greedy decoding
        _case("decode_onecall_ragged", kind="onecall", V=32000, n=11987, d=4096, d_l=256,
              rows=19, act="bf16", tau=0.0, bias=True),
        # the split dimension and the language subset of the paper's own setup
        _case("dend_step", V=150000, n=60000, d=4096, d_l=96, rows=32),
        # the same setup with the payload streamed in blocks
        _case("dend_streamed", kind="onecall", V=150000, n=45000, d=4096, d_l=128, rows=32,
              chunk=15000),
        # the endpoint's machine: a few sessions' payload arrives (an odd
        # number of kept ids), the local partial is added, tokens are drawn
        _case("endpoint_ragged", kind="endpoint", V=150000, n=44999, d=4096, d_l=512, rows=12,
              tau=0.7),
        # speculative decoding: 64 sessions verify four drafts each
        _case("spec_verify", kind="spec", V=128256, n=51302, d=4096, d_l=512, sessions=64, k=4),
        # a large batch on a quantized (e4m3) head, whole vocabulary
        _case("fp8_step", V=152064, n=152064, d=8192, d_l=1024, rows=256, w="fp8", clip=40.0),
        # one row over a very large vocabulary: a weight stream
        _case("large_vocab_row", V=256000, n=256000, d=5120, d_l=512, rows=1),
        # the cloud's half for a mid-sized batch over half of a large
        # vocabulary, bf16 states, its logits kept as well (monitoring)
        _case("cloud_half_batch", kind="cloud", V=256000, n=128000, d=5120, d_l=512, rows=64,
              act="bf16", logits=True),
        # no split: the whole head for a ragged prefill batch, logits returned
        _case("unsplit_prefill", kind="unsplit", V=32000, n=32000, d=4096, d_l=4096, rows=147),
        # the largest: a thousand rows over the whole large vocabulary
        _case("large_batch_step", V=256000, n=256000, d=5120, d_l=512, rows=1024),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: rows, vocabulary, kept ids and widths over the whole
    range, ragged as often as not; no more work than the largest listed."""
    kind = rng.choice(["step", "step", "step", "onecall", "spec", "cloud", "endpoint", "unsplit"])
    d, d_l = rng.choice([(512, 64), (2048, 128), (4096, 48), (4096, 96), (4096, 256), (4096, 512),
                         (5120, 512), (8192, 1024)])
    V = max(2048, _log_uniform(rng, 4096, 256000) // 8 * 8 + rng.choice([0, 0, 1, 5]))
    keep = rng.choice([0.1, 0.3, 0.4, 0.5, 1.0, 1.0])
    n = V if keep == 1.0 else max(512, int(keep * V) + rng.randint(-9, 9))
    rows = _log_uniform(rng, 1, 1024)
    c = dict(kind=kind, V=V, n=n, d=d, d_l=d_l, rows=rows, act=rng.choice(["fp32", "fp32", "bf16"]),
             tau=rng.choice([0.0, 0.6, 0.8, 1.0, 1.0]), bias=rng.random() < 0.25)
    # (no more work than the largest listed case)
    rows = c["rows"] = max(1, min(rows, 1024 * 256000 * 5120 // (n * d)))
    if kind == "spec":
        c["k"] = rng.randint(1, 8)
        c["sessions"] = max(1, min(128, rows // (c["k"] + 1)))
        c["probs"] = rng.random() < 0.7
        c["tau"] = rng.choice([0.8, 1.0])
    elif kind == "unsplit":
        # (its outputs are fp32 logits: up to a prefill batch of 256 rows)
        c.update(d_l=d, rows=min(rows, 256), act="fp32", bias=False)
    elif kind == "endpoint":
        c.update(act="fp32", bias=False, sampler=rng.choice(["cdf", "cdf", "gumbel"]))
    elif kind == "cloud":
        c["logits"] = rng.random() < 0.3
    elif kind == "onecall" and rng.random() < 0.5:
        c["chunk"] = max(256, n // rng.randint(2, 5))
    if kind in ("step", "cloud") and rng.random() < 0.2:
        c.update(w="fp8", clip=40.0)
    return _case(**c)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _inputs(case, seed):
    """The seeded inputs of a case on the GPU: weights ~ N(0, 0.02) in bf16
    (or e4m3 with row scales), RMS-normalised hidden states, kept ids in runs
    of 16 to 256 with gaps between them, drafts drawn from their own
    distributions."""
    dev = torch.device("cuda", torch.cuda.current_device())
    c = case
    unsplit = c["kind"] == "unsplit"
    # (the unsplit head's weights are one matrix: the generator's split is
    # taken at a width beyond it, of which nothing is used)
    d = c["d"] + 16 if unsplit else c["d"]
    w = wl.make_workload("case", V=c["V"], d=d, d_l=c["d_l"], rows=c["rows"], n_keep=c["n"],
                         clip=c["clip"], tau=c["tau"], w_dtype=c["w"], seed=1000 + int(seed),
                         device=dev, sessions=c["sessions"], k=c["k"], with_bias=c["bias"])
    x = dict(w=w, h=w.h, keep=w.keep_ids)
    if c["kind"] == "endpoint":
        # a payload as a cloud sends it: codes up to 127 in every row, scales
        # of partial logits whose largest entry is a few units
        g = torch.Generator(device=dev)
        g.manual_seed(77000 + int(seed))
        codes = (torch.randn(c["rows"], c["n"], generator=g, device=dev) * 29.0)
        x["codes"] = codes.round().clamp(-127, 127).to(torch.int8).contiguous()
        x["scale"] = (torch.rand(c["rows"], generator=g, device=dev) * 0.02 + 0.03).contiguous()
    return x


def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    x = _inputs(c, seed)
    w = x["w"]
    dev = w.h.device
    ctx = sph.Context(dev.index)
    ctx.reserve(c["rows"], c["n"], c["d"])
    if c["sampler"] == "gumbel":
        ctx.set_option(sph.SPH_OPT_SAMPLER, sph.SPH_SAMPLER_GUMBEL)
    R, n = c["rows"], c["n"]
    s = dict(case=c, ctx=ctx, w=w, h=w.h, h_cloud=w.h_cloud, h_local=w.h_local,
             keep=w.keep_ids, x=x,
             tokens=torch.empty(R, dtype=torch.int32, device=dev), rng=int(seed) * 7919 + 11,
             act=sph.SPH_ACT_BF16 if c["act"] == "bf16" else sph.SPH_ACT_FP32)
    if c["kind"] in ("step", "spec", "cloud"):
        s["codes"] = torch.empty(R, n, dtype=torch.int8, device=dev)
        s["scale"] = torch.empty(R, dtype=torch.float32, device=dev)
    if c["kind"] == "onecall":
        L = n if c["chunk"] == 0 or c["chunk"] >= n else c["chunk"]
        s["codes"] = torch.empty(R * n, dtype=torch.int8, device=dev)
        s["scale"] = torch.empty(-(-n // L) * R, dtype=torch.float32, device=dev)
    if c["kind"] in ("spec", "endpoint", "unsplit"):
        s["z"] = torch.empty(R, n, dtype=torch.float32, device=dev)
    if c["logits"]:
        s["y"] = torch.empty(R, n, dtype=torch.float32, device=dev)
    if c["kind"] == "spec":
        s["n_acc"] = torch.empty(c["sessions"], dtype=torch.int32, device=dev)
        s["next"] = torch.empty(c["sessions"], dtype=torch.int32, device=dev)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c, ctx, w, kind = s["case"], s["ctx"], s["w"], s["case"]["kind"]
    if kind in ("step", "spec", "cloud"):
        ctx.partial_logits(s["h_cloud"], w.W_h, keep_ids=s["keep"], clip=c["clip"],
                           w_row_scale=w.w_scale, bias=w.bias, act_mode=s["act"],
                           codes=s["codes"], row_scale=s["scale"], partial_out=s.get("y"))
        if kind == "cloud":
            out = dict(codes=s["codes"], scale=s["scale"])
            if c["logits"]:
                out["y"] = s["y"]
            return out
    if kind == "step":
        ctx.fuse_sample(s["codes"], s["scale"], s["h_local"], w.W_l, keep_ids=s["keep"],
                        temperature=c["tau"], seed=w.seed, offset=s["rng"], tokens=s["tokens"])
        return dict(codes=s["codes"], scale=s["scale"], tokens=s["tokens"])
    if kind == "onecall":
        ctx.split_step(s["h"], c["d_l"], w.W_h, w.W_l, keep_ids=s["keep"], clip=c["clip"],
                       bias=w.bias, act_mode=s["act"], temperature=c["tau"], seed=w.seed,
                       offset=s["rng"], chunk=c["chunk"], codes=s["codes"], scales=s["scale"],
                       tokens=s["tokens"])
        return dict(codes=s["codes"], scale=s["scale"], tokens=s["tokens"])
    if kind == "spec":
        ctx.fuse_sample(s["codes"], s["scale"], s["h_local"], w.W_l, keep_ids=s["keep"],
                        temperature=c["tau"], seed=w.seed, fused_logits_out=s["z"], draw=False)
        ctx.verify_draft(s["z"], c["sessions"], c["k"], w.draft_tokens, keep_ids=s["keep"],
                         draft_probs=w.draft_probs if c["probs"] else None,
                         temperature=c["tau"], seed=w.seed, offset=s["rng"],
                         n_accepted=s["n_acc"], next_token=s["next"])
        return dict(codes=s["codes"], scale=s["scale"], z=s["z"], n_acc=s["n_acc"],
                    next=s["next"])
    if kind == "endpoint":
        ctx.fuse_sample(s["x"]["codes"], s["x"]["scale"], s["h_local"], w.W_l, keep_ids=s["keep"],
                        temperature=c["tau"], seed=w.seed, offset=s["rng"], tokens=s["tokens"],
                        fused_logits_out=s["z"])
        return dict(z=s["z"], tokens=s["tokens"])
    ctx.fuse_sample(None, None, s["h_local"], w.W_l, keep_ids=s["keep"], temperature=c["tau"],
                    seed=w.seed, offset=s["rng"], tokens=s["tokens"], fused_logits_out=s["z"])
    return dict(z=s["z"], tokens=s["tokens"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    c = dict(DEFAULTS, **case)
    R, n, d, d_l, kind = c["rows"], c["n"], c["d"], c["d_l"], c["kind"]
    wb = 1 if c["w"] == "fp8" else 2
    d_h = d - d_l
    ids = 4 * n if n != c["V"] else 0
    payload = R * n + 4 * R
    flops = 2 * R * n * d
    if kind == "cloud":
        b = n * d_h * wb + 4 * R * d_h + ids + payload
        flops = 2 * R * n * d_h
    elif kind == "endpoint":
        b = n * d_l * 2 + 4 * R * d_l + ids + payload + 4 * R * n + 4 * R
        flops = 2 * R * n * d_l
    elif kind == "unsplit":
        b = n * d * 2 + 4 * R * d + ids + 4 * R * n + 4 * R
    else:
        b = n * d_h * wb + n * d_l * 2 + 4 * R * d + ids + payload + 4 * R
    if c["w"] == "fp8":
        b += 4 * n
    if c["bias"]:
        b += 4 * n
    if c["logits"]:
        b += 4 * R * n
    if kind == "spec":
        S, k = c["sessions"], c["k"]
        # the fused target logits (an output) and the drafts: ids, and where
        # given the distribution of the one position a rejection can land on
        b += 4 * R * n + 4 * S * k + 8 * S + (4 * S * n if c["probs"] else 0)
    return {"bytes": float(b), "flops": float(flops)}


# ---------------------------------------------------------------------------
# how close another correct implementation comes
# ---------------------------------------------------------------------------
def tolerance(case):
    """About four times what `run` was measured to be off `exact`: fp32 sums
    over up to 8192 products on the tensor cores, 1.3e-5 of the logits and row
    scales (largest entry 3e-5), which rounds one code in 7000 (e4m3 weights:
    one in 3000) to its neighbour; z, where a payload made in the same pass is
    fused, moves by one code step there (3.4e-4, largest 4e-2)."""
    c = dict(DEFAULTS, **case)
    if c["kind"] == "spec":
        return {"rel": 1e-3, "max": 0.15, "differ": 1e-3}
    return {"rel": 5e-5, "max": 2e-4, "differ": 2e-3 if c["w"] == "fp8" else 1e-3}


# ---------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------
def _logits64(h, W, keep, n, scale=None, bias=None):
    """h [R, K] fp64 times the kept rows of W [V, K], over blocks of ids."""
    R, K = h.shape
    y = torch.empty(R, n, dtype=torch.float64, device=h.device)
    step = max(1024, (1 << 28) // K)
    for j in range(0, n, step):
        e = min(n, j + step)
        rows = W[j:e] if keep is None else W[keep[j:e].long()]
        y[:, j:e] = h @ rows.to(torch.float32).double().t()
    if scale is not None:
        y *= (scale if keep is None else scale[keep.long()]).double()
    if bias is not None:
        y += (bias if keep is None else bias[keep.long()]).double()
    return y


def exact(case, seed):
    c = dict(DEFAULTS, **case)
    x = _inputs(c, seed)
    w = x["w"]
    R, n, kind = c["rows"], c["n"], c["kind"]
    h = w.h.double()
    h_l = h[:, :c["d_l"]]
    if kind == "unsplit":
        return dict(z=_logits64(h_l, w.W_l, w.keep_ids, n), tokens=None)
    if kind == "endpoint":
        z = _logits64(h_l, w.W_l, w.keep_ids, n)
        return dict(z=z + x["codes"].double() * x["scale"].double()[:, None], tokens=None)
    h_c = h[:, c["d_l"]:]
    if c["act"] == "bf16":
        h_c = w.h[:, c["d_l"]:].bfloat16().double()
    y = _logits64(h_c, w.W_h, w.keep_ids, n, w.w_scale, w.bias)
    yc = y.clamp(-c["clip"], c["clip"])
    L = n if c["chunk"] == 0 or c["chunk"] >= n else c["chunk"]
    codes, scales = [], []
    for j in range(0, n, L):                       # a scale per row and payload block
        blk = yc[:, j:j + L]
        sc = blk.abs().amax(dim=1) / 127.0
        q = torch.where(sc[:, None] > 0, blk / sc[:, None], torch.zeros_like(blk)).round()
        codes.append(q.clamp(-127, 127).to(torch.int8).reshape(-1))
        scales.append(sc)
    out = dict(codes=torch.cat(codes), scale=torch.cat(scales), tokens=None)
    if kind == "cloud":
        out.pop("tokens")
        if c["logits"]:
            out["y"] = y
    if kind == "spec":
        out.pop("tokens")
        z = _logits64(h_l, w.W_l, w.keep_ids, n)
        z += out["codes"].view(R, n).double() * out["scale"].float().double()[:, None]
        out.update(z=z, n_acc=None, next=None)
    return out
