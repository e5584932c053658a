"""The work this framework is used for, as cases that can be timed.

Every case is one call sequence of ``DemoTransform`` on a set of parameter tensors: a whole optimizer step (every
worker's ``compress``, then ``decode_apply``), the decode alone at a large fan-in, or the parameter-server form
(``decode_signs`` + ``apply_signs``).  Tensor sets, chunk sizes, k, worker counts and value distributions are those of the
benchmark configurations and tests of this repository; ``draw`` spreads them over the ranges that these stand for.

Outputs of a step are the new momentum of every worker, the record indices of every worker and the new parameters.
The record values are not listed beside them because the momentum holds them (m_new = B - IDCT(records)), and
because a tie at rounding level between the k-th and the next magnitude moves the later records of that chunk by one place.
"""
from __future__ import annotations

import math

import torch

from paper_2411_19870_b200 import (
    DEMO_AGG_COUNT_MEAN,
    DEMO_AGG_MEAN,
    DEMO_AGG_SUM,
    DEMO_BF16,
    DEMO_F32,
    DEMO_MOMENTUM_DCT,
    DEMO_PHI_IDENTITY,
    DEMO_PHI_SIGN,
    DemoTransform,
)
from paper_2411_19870_b200.chunking import divisor_chunk_shape

BETA, LR, WD = 0.999, 1e-3, 0.1
AGG = {"sum": DEMO_AGG_SUM, "mean": DEMO_AGG_MEAN, "count": DEMO_AGG_COUNT_MEAN}
PHI = {"sign": DEMO_PHI_SIGN, "identity": DEMO_PHI_IDENTITY}


def _case(op, tensors, **kw):
    c = {"op": op, "tensors": tensors, "chunk": 64, "topk": 32, "workers": 1, "grad": "bf16", "values": "normal",
         "basis": "dct", "domain": "spatial", "agg": "sum", "phi": "sign"}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call: one fp32 weight and one bias in 8 x 8 chunks (the "tiny" configuration).  Latency and launches.
        _case("step", "matrix", name="tiny", rows=256, cols=512, bias=512, chunk=8, topk=4, workers=2, grad="f32"),
        # A scaled-down decoder set, as in quick runs: many small tensors, 1-D norm vectors among them.  Latency again.
        _case("step", "decoder", name="small_decoder", d_model=256, layers=2, d_ff=1024, vocab=1024, untied=True, workers=4),
        # One large matrix, one worker, row-wise scaled gradients (the single-matrix configuration).
        _case("step", "matrix", name="matrix_8192", rows=8192, cols=8192, values="rows"),
        # The 300M-class decoder set with its eight workers.
        _case("step", "decoder", name="decoder_300m", d_model=1024, layers=24, d_ff=4096, vocab=50304, untied=False,
              workers=8),
        # The 1B-class decoder set, the largest: four of its sixteen workers, so that a few sets of inputs fit one GPU.
        _case("step", "decoder", name="decoder_1b", d_model=2048, layers=16, d_ff=8192, vocab=50304, untied=True,
              workers=4),
        # The stress matrix in 32 x 32 chunks: heavy-tailed gradients, some rows of chunks untouched.
        _case("step", "matrix", name="stress_s32", rows=4096, cols=4096, chunk=32, topk=8, workers=8, values="heavy"),
        # One decoder layer of the 1B class in 128 x 128 chunks, the paper's second chunk size.
        _case("step", "decoder", name="layer_s128", d_model=2048, layers=1, d_ff=8192, vocab=0, untied=False, chunk=128,
              workers=4),
        # The stress matrix with more coefficients kept than a chunk has rows.
        _case("step", "matrix", name="stress_k128", rows=4096, cols=4096, topk=128, workers=8, values="heavy"),
        # The receiving side of 64 workers: decode and update alone.
        _case("decode", "matrix", name="fan_in_64", rows=4096, cols=4096, workers=64),
        # The parameter server's side and the workers' update on the 300M-class set.
        _case("server", "decoder", name="server_300m", d_model=1024, layers=24, d_ff=4096, vocab=50304, untied=False,
              workers=8),
        # A random orthonormal projection, redrawn every step (the paper's choice-of-projection experiment).
        _case("step", "matrix", name="random_basis", rows=4096, cols=8192, workers=2, basis="random"),
        # Convolution weights in 32 x 32 x 3 x 3 chunks, a 7 x 7 stem and a table whose row count 64 does not divide.
        _case("step", "conv", name="conv_ragged", layers=4, out_ch=512, in_ch=512, kernel=3, stem=7, table_rows=7511,
              table_extent=29, table_cols=512, target=32, workers=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(v, s):
    return max(1, int(round(v / s))) * s


def draw(rng):
    """Matrices from one chunk to 8192 x 8192, decoder sets up to a few hundred million parameters, every chunk size and
    gradient type, k from 1 to 128, one to eight workers in a step and up to 64 in a decode."""
    kind = rng.choice(["matrix"] * 5 + ["decoder"] * 5 + ["decode"] * 2 + ["server", "basis", "host"] + ["conv"] * 2)
    s = rng.choice([64] * 6 + [128] * 3 + [32] * 2 + [16, 8])
    grad = rng.choice(["bf16", "bf16", "bf16", "f32"])
    values = rng.choice(["normal", "rows", "heavy"])
    k = min(_log_int(rng, 1, 128), s * s)
    workers = _log_int(rng, 1, 8)
    side = 8192 if s >= 32 else 1024  # the small chunk sizes serve small tensors
    rows, cols = _mult(_log_int(rng, s, side), s), _mult(_log_int(rng, s, side), s)
    if kind == "decoder":
        d = _mult(_log_int(rng, 128, 1024), 128)
        layers, vocab = _log_int(rng, 1, 12), _mult(_log_int(rng, 512, 16384), 128)
        if s < 32:
            d, layers, vocab = 128, min(layers, 3), 512
        return _case("step", "decoder", d_model=d, layers=layers, d_ff=4 * d, vocab=vocab, untied=rng.random() < 0.5,
                     chunk=s, topk=k, workers=workers, grad=grad,
                     domain="dct" if s == 64 and rng.random() < 0.2 else "spatial")
    if kind == "decode":
        rows, cols = min(rows, 4096), min(cols, 4096)
        return _case("decode", "matrix", rows=rows, cols=cols, chunk=s, topk=k, workers=_log_int(rng, 1, 64),
                     agg=rng.choice(["sum", "sum", "mean", "count"]), phi=rng.choice(["sign", "sign", "identity"]))
    if kind == "server":
        return _case("server", "matrix", rows=rows, cols=cols, chunk=s, topk=k, workers=_log_int(rng, 1, 16))
    if kind == "basis":
        return _case("step", "matrix", rows=_mult(min(rows, 4096), 64), cols=_mult(min(cols, 4096), 64), topk=k,
                     workers=min(workers, 4), grad=grad, basis="random")
    if kind == "host":
        return _case("host", "matrix", rows=min(rows, 2048), cols=min(cols, 2048), chunk=s, topk=k,
                     workers=min(workers, 4), grad=grad)
    if kind == "conv":
        return _case("step", "conv", layers=rng.randint(1, 4), out_ch=_mult(_log_int(rng, 32, 512), 32),
                     in_ch=_mult(_log_int(rng, 32, 512), 32), kernel=rng.choice([1, 3, 5]), stem=rng.choice([0, 7]),
                     table_rows=_log_int(rng, 16, 2048), table_extent=rng.choice([13, 29, 31, 48, 57]),
                     table_cols=_mult(_log_int(rng, 32, 512), 32), target=rng.choice([16, 32, 64]), topk=k,
                     workers=min(workers, 4), grad=grad)
    return _case("step", "matrix", rows=rows, cols=cols, bias=rng.choice([0, cols]), chunk=s, topk=k, workers=workers,
                 grad=grad, values=values)


def _shapes(c):
    """(shapes, chunk shapes or None) of the case's tensors; a conv set's table has table_rows blocks of table_extent rows."""
    if c["tensors"] == "matrix":
        return [(c["rows"], c["cols"])] + ([(c["bias"],)] if c.get("bias") else []), None
    if c["tensors"] == "decoder":
        d, ff = c["d_model"], c["d_ff"]
        shapes = ([(d, d)] * 4 + [(ff, d)] * 2 + [(d, ff)] + [(d,)] * 2) * c["layers"]
        if c["vocab"]:
            shapes = shapes + [(c["vocab"], d)] + ([(d, c["vocab"])] if c["untied"] else [])
        return shapes, None
    shapes = [(c["out_ch"], c["in_ch"], c["kernel"], c["kernel"])] * c["layers"]
    if c["stem"]:
        shapes = shapes + [(64, 3, c["stem"], c["stem"])]
    shapes = shapes + [(c["table_extent"] * max(1, c["table_rows"] // c["table_extent"]), c["table_cols"]), (c["out_ch"],)]
    chunks = [divisor_chunk_shape(shp, c["target"]) for shp in shapes]
    # (the table keeps the extent that divides its rows, whatever the target)
    chunks[-2] = (c["table_extent"], divisor_chunk_shape((c["table_cols"],), 64)[0])
    return shapes, chunks


def _chunk_elems(c):
    """[(elements per chunk, chunks)] per tensor."""
    shapes, chunks = _shapes(c)
    if chunks is None:
        chunks = [(c["chunk"],) * len(shp) for shp in shapes]
    return [(math.prod(ch), math.prod(shp) // math.prod(ch)) for shp, ch in zip(shapes, chunks)]


def _views(flat, shapes, offsets):
    return [flat[o:o + math.prod(s)].view(*s) for s, o in zip(shapes, offsets)]


def prepare(case, seed):
    c = case
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    shapes, chunks = _shapes(c)
    W = c["workers"]
    gdtype = torch.bfloat16 if c["grad"] == "bf16" else torch.float32
    tr = DemoTransform(shapes, chunk=c["chunk"] if chunks is None else 0, topk=c["topk"], beta=BETA, lr=LR, weight_decay=WD,
                       num_workers=W, grad_dtype=DEMO_BF16 if c["grad"] == "bf16" else DEMO_F32, device=dev.index,
                       chunk_shapes=chunks)
    tr.set_decode_mode(AGG[c["agg"]], PHI[c["phi"]])
    if c["domain"] == "dct":
        tr.set_momentum_domain(DEMO_MOMENTUM_DCT)
    offsets, total = [], 0
    for s in shapes:  # every tensor starts on a 16-byte boundary of its flat buffer
        offsets.append(total)
        total += (math.prod(s) + 63) // 64 * 64
    records = tr.payload_bytes // 8

    st = {"case": c, "tr": tr, "gauss": None}
    flat_x = torch.empty(total, device=dev).normal_(0.0, 0.02, generator=gen)
    st["x"] = _views(flat_x, shapes, offsets)
    payloads = [torch.zeros(tr.payload_bytes, dtype=torch.uint8, device=dev) for _ in range(W)]
    st["payloads"] = payloads
    out = {"x": flat_x}

    if c["op"] in ("decode", "server"):
        # records as workers send them: k distinct ascending indices per chunk, values of both signs
        for p in payloads:
            rec = p.view(torch.int32).view(records, 2)
            at = 0
            for M, n in _chunk_elems(c):
                k = min(c["topk"], M)
                step = M // k
                idx = torch.arange(k, device=dev) * step + torch.randint(0, step, (n, k), generator=gen, device=dev)
                rec[at:at + n * k, 0] = idx.reshape(-1).to(torch.int32)
                at += n * k
            p.view(torch.float32).view(records, 2)[:, 1].normal_(0.0, 1e-2, generator=gen)
        if c["op"] == "server":
            flat_s = torch.zeros(total, dtype=torch.int8, device=dev)
            st["signs"] = _views(flat_s, shapes, offsets)
            out["signs"] = flat_s
        st["out"] = out
        return st

    # per-tensor gradient scale, log-uniform over two decades; the momentum a few gradients large
    scales = [10.0 ** (2.0 * float(u) - 4.0) for u in torch.rand(len(shapes), generator=gen, device=dev).cpu()]
    st["g"], st["m"], st["host_g"] = [], [], []
    for w in range(W):
        g = torch.empty(total, device=dev, dtype=gdtype).normal_(generator=gen)
        m = torch.empty(total, device=dev).normal_(0.0, 3.0, generator=gen)
        gv, mv = _views(g, shapes, offsets), _views(m, shapes, offsets)
        for t, s in enumerate(shapes):
            if c["values"] == "rows" and len(s) == 2:
                f = torch.exp(torch.randn((s[0], 1), generator=gen, device=dev))
                gv[t].mul_(f.to(gdtype))
                mv[t].mul_(f)
            if c["values"] == "heavy" and len(s) == 2:
                # Student-t with three degrees of freedom; one block of chunk rows in twenty is untouched (exactly zero)
                for v in (gv[t], mv[t]):
                    chi = torch.zeros(s, device=dev)
                    for _ in range(3):
                        chi.add_(torch.randn(s, generator=gen, device=dev).square_())
                    v.mul_(chi.div_(3.0).rsqrt_().to(v.dtype))
                blocks = torch.rand((s[0] // c["chunk"], 1), generator=gen, device=dev).ge(0.05)
                keep = blocks.repeat_interleave(c["chunk"], dim=0)
                gv[t].mul_(keep.to(gdtype))
                mv[t].mul_(keep.to(torch.float32))
            gv[t].mul_(scales[t])
            mv[t].mul_(scales[t])
        st["g"].append(gv)
        st["m"].append(mv)
        out["m%d" % w] = m
        out["idx%d" % w] = payloads[w].view(torch.int32).view(records, 2)[:, 0]
        if c["op"] == "host":
            st["host_g"].append([v.cpu().pin_memory() for v in gv])
    if c["op"] == "host":
        st["host_out"] = torch.zeros(W * tr.payload_bytes, dtype=torch.uint8).pin_memory()
        out["host_idx"] = st["host_out"].view(torch.int32).view(W * records, 2)[:, 0]
    if c["basis"] == "random":
        st["gauss"] = torch.randn((64, 64), generator=gen, device=dev).cpu()
    st["out"] = out
    return st


def run(state):
    tr, op = state["tr"], state["case"]["op"]
    if op == "decode":
        tr.decode_apply(state["payloads"], state["x"])
    elif op == "server":
        tr.decode_signs(state["payloads"], state["signs"])
        tr.apply_signs(state["signs"], state["x"])
    elif op == "host":
        tr.step_host(state["host_g"], state["g"], state["m"], state["payloads"], state["x"], state["host_out"])
    else:
        if state["gauss"] is not None:
            tr.set_basis_gaussian(state["gauss"])
        for w in range(state["case"]["workers"]):
            tr.compress(w, state["g"][w], state["m"][w], state["payloads"][w])
        tr.decode_apply(state["payloads"], state["x"])
    return state["out"]


def work(case):
    c = case
    W, gb = c["workers"], 2 if c["grad"] == "bf16" else 4
    per = _chunk_elems(c)
    P = sum(M * n for M, n in per)
    R = sum(min(c["topk"], M) * n for M, n in per)
    # additions and multiplications of a fast transform, about 4 log2(M) per element; a caller-supplied basis has none:
    # two dense products of length s
    one = sum((4 * 64 if c["basis"] == "random" else 4 * math.log2(max(2, M))) * M * n for M, n in per)
    decode = {"bytes": W * 8 * R + 8 * P, "flops": one + 3 * P}
    if c["op"] == "decode":
        return decode
    if c["op"] == "server":  # the signs are written by one call and read by the other
        return {"bytes": W * 8 * R + 10 * P, "flops": one + 3 * P}
    step = {"bytes": W * ((gb + 8) * P + 8 * R) + decode["bytes"], "flops": W * (2 * one + 3 * P) + decode["flops"]}
    if c["op"] == "host":  # the gradients cross to the device first, the records back to the host
        step["bytes"] += W * (2 * gb * P + 2 * 8 * R)
    return step


def tolerance(case):
    """Between the two kernel families of the library (DEMO_PATH_AUTO / DEMO_PATH_GENERIC: other summation orders) the
    momentum differs by 5e-8 ... 2e-7 (relative 2-norm) and the parameters by 4e-8, as fp32 gives.  Beside that there are
    two discrete effects.  A chunk whose k-th and next magnitude differ by less than the rounding may keep either: measured
    for up to one chunk in 8000 of a worker (more under a dense basis product), and then the momentum of that chunk
    differs by one coefficient (about 2.5 * 2 ** 0.5 / s of the chunk's norm; measured 6e-4 ... 9e-4 over all chunks) and a
    third of its record places move.  And a parameter whose reconstructed momentum is zero to rounding takes another sign,
    a step of 2 lr at parameters of size 0.02 (about one in a million; measured 3e-5 ... 4e-4 for the parameters)."""
    c = case
    if c["op"] in ("decode", "server"):
        return {"rel": 3e-4, "max": 0.3, "differ": 1e-5}
    M, n = max(_chunk_elems(c), key=lambda v: v[0] * v[1])
    share = max(5e-4, 3.0 / n)
    return {"rel": min(0.03, 1.5 * 3.5 / math.sqrt(M) * math.sqrt(share)), "max": min(0.9, 40.0 / math.sqrt(M)),
            "differ": min(0.01, share)}
