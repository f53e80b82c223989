"""The work a training program has this framework do, as measurable cases.

A case is one pass of such a program through the public entry points: a whole layer step (split and quantize the
activation, the weight and the output gradient, then forward, input gradient and weight gradient), the same with stored
weight factors, a decoder block with its layers spread over streams, a forward-only pass, or plain quantization.
Sizes are those of the repository's workloads (LLaMA-3 8B and 70B projections, the small configuration) and ragged ones
between them.  Inputs are the repository's planted-spectrum tensors.
"""
import functools
import math

import torch

from paper_2509_00404_b200 import binding as B
from paper_2509_00404_b200 import synth

SIGMA_X, SIGMA_W, SIGMA_D = 1.0, 0.02, 1e-4        # bulk widths of activations, weights and output gradients


def _step(name, tokens, d_in, d_out, k, p=8, **more):
    return {"name": name, "op": "step", "tokens": tokens, "d_in": d_in, "d_out": d_out, "k": k, "p": p if k else 0, "weights": "split",
            "act_sketch": "sampled", "out": "bf16", **more}


def listed():
    return [
        # the smallest call: forward of the small configuration, weight operand kept (latency and launches)
        {"name": "forward_128tok_256", "op": "forward", "tokens": 128, "d_in": 256, "d_out": 256, "k": 4, "p": 4, "out": "fp32"},
        # evaluation of a q_proj-shaped layer on a short batch, weight operand kept
        {"name": "forward_1024tok_4096", "op": "forward", "tokens": 1024, "d_in": 4096, "d_out": 4096, "k": 32, "p": 8, "out": "bf16"},
        # plain NVFP4 quantization of an FP32 master weight that is a strided view, ragged against the 128-element tiles
        {"name": "quantize_fp32_ragged", "op": "quantize", "rows": 4160, "cols": 2752, "pad": 64, "dtype": "fp32", "rounding": "rne", "axes": "both"},
        # plain quantization of the largest output gradient of a decoder block, stochastic rounding, both orientations
        {"name": "quantize_sr_16384x14336", "op": "quantize", "rows": 16384, "cols": 14336, "pad": 0, "dtype": "bf16", "rounding": "sr", "axes": "both"},
        # a layer step whose extents are no multiple of any tile
        _step("step_ragged_1088tok", 1088, 2112, 1472, 24),
        # LLaMA-3-8B q_proj, two sequences of 2048 tokens
        _step("step_q_4096tok", 4096, 4096, 4096, 32),
        # grouped-query k / v projection at a full batch (tall and narrow), every operand decomposed from all of its rows
        _step("step_kv_full_16384tok", 16384, 4096, 1024, 32, act_sketch="full"),
        # LLaMA-3-8B up projection in the paper's training form: stored factors and residual re-quantized, factor gradients
        _step("step_stored_up_8192tok", 8192, 4096, 14336, 32, weights="stored", out="fp32"),
        # a rank above 64 (the wide decomposition)
        _step("step_rank128_4096tok", 4096, 2048, 7168, 128),
        # LLaMA-3-70B-shaped projection without a low-rank part (plain NVFP4 training step)
        _step("step_70b_plain_16384tok", 16384, 8192, 28672, 0),
        # the same projection at rank 64: the largest step
        _step("step_70b_rank64_16384tok", 16384, 8192, 28672, 64),
        # all seven linear layers of a LLaMA-3-8B decoder block, decompositions and products spread over streams
        {"name": "block_16384tok", "op": "block", "tokens": 16384, "d_model": 4096, "d_kv": 1024, "d_ff": 14336, "k": 32, "p": 8},
    ]


def _log_size(rng, lo, hi, multiple=64):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple))


def draw(rng):
    op = rng.choice(["step", "step", "step", "forward", "quantize", "block"])
    if op == "quantize":
        dtype = rng.choice(["bf16", "fp32"])
        return {"op": op, "rows": _log_size(rng, 128, 16384), "cols": _log_size(rng, 256, 14336), "pad": rng.choice([0, 64]), "dtype": dtype,
                "rounding": rng.choice(["rne", "sr"]), "axes": rng.choice(["both", "cols", "rows"])}
    if op == "block":
        d = _log_size(rng, 1024, 4096, 128)
        return {"op": op, "tokens": _log_size(rng, 1024, 16384), "d_model": d, "d_kv": d // 4 // 64 * 64, "d_ff": d * 7 // 2 // 64 * 64,
                "k": rng.choice([16, 24, 32]), "p": 8}
    tokens, d_in, d_out = _log_size(rng, 128, 16384), _log_size(rng, 256, 8192), _log_size(rng, 256, 28672)
    most = min(tokens, d_in, d_out)
    ranks = [k for k in (4, 8, 16, 24, 32, 48, 64) if 8 * k <= most]
    if most >= 1024:
        ranks += [k for k in (96, 128) if 8 * k <= most]
    k = rng.choice(ranks + [0]) if op == "step" else rng.choice(ranks)
    p = rng.choice([4, 8]) if k <= 32 else 8
    out = rng.choice(["bf16", "fp32"])
    if op == "forward":
        return {"op": op, "tokens": tokens, "d_in": d_in, "d_out": d_out, "k": k, "p": p, "out": out}
    c = _step("", tokens, d_in, d_out, k, p, weights=rng.choice(["split", "stored"]) if k else "split",
              act_sketch=rng.choice(["sampled", "sampled", "full"]), out=out)
    del c["name"]
    return c


@functools.lru_cache(maxsize=None)
def _handle(i):
    """One library handle per stream, kept for the life of the program; handle 0 serves the current stream."""
    return B.Handle(torch.cuda.current_device())


@functools.lru_cache(maxsize=None)
def _stream(i):
    return torch.cuda.Stream()


def _dtype(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


def _planted(rows, cols, k, sigma, seed):
    return synth.planted_device(rows, cols, max(k, 8), sigma, seed)


BLOCK_X = (0, 0, 0, 1, 2, 2, 3)                    # which activation each layer of the block reads (q, k, v | o | gate, up | down)


def _block_dims(c):
    d, kv, ff = c["d_model"], c["d_kv"], c["d_ff"]
    return [(d, d), (d, kv), (d, kv), (d, d), (d, ff), (d, ff), (ff, d)]


def prepare(case, seed):
    c, h = dict(case), _handle(0)
    seed = 1000 * (seed % 1000003)
    st = {"case": c, "seed": seed % 65521}
    if c["op"] == "quantize":
        x = _planted(c["rows"], c["cols"] + c["pad"], 8, SIGMA_D if c["rounding"] == "sr" else SIGMA_W, seed + 1).to(_dtype(c["dtype"]))
        st["x"] = x[:, : c["cols"]]
        st["out"] = (B.NvFp4(c["rows"], c["cols"]) if c["axes"] != "rows" else None, B.NvFp4(c["cols"], c["rows"]) if c["axes"] != "cols" else None)
        return st
    k, p, l = c["k"], c["p"], c["tokens"]
    if c["op"] == "block":
        dims = _block_dims(c)
        xs = [_planted(l, dims[BLOCK_X.index(g)][0], k, SIGMA_X, seed + g) for g in range(4)]
        st["layers"] = [{"x": BLOCK_X[j], "w": _planted(n, m, k, SIGMA_W, seed + 11 + j), "d": _planted(l, n, k, SIGMA_D, seed + 31 + j),
                         "wo": B.Operand(n, m, k), "do": B.Operand(l, n, k), "y": torch.empty((l, n), dtype=torch.bfloat16, device="cuda"),
                         "dx": torch.empty((l, m), dtype=torch.bfloat16, device="cuda"), "dw": torch.empty((n, m), dtype=torch.bfloat16, device="cuda")}
                        for j, (m, n) in enumerate(dims)]
        st["xs"], st["xo"] = xs, [B.Operand(l, x.shape[1], k) for x in xs]
        # every handle's scratch memory is sized for its largest layer before the first pass
        big = max(max(d) for d in dims + [(l, l)])
        need = [max(B.workspace_bytes(1, n, m, k, p) for m, n in dims), max(B.workspace_bytes(1, l, n, k, p) for n in set(sum(dims, ())))]
        need = [need[0]] + [max(need[1], B.workspace_bytes(3, big, big, k, 0), B.workspace_bytes(2, big, big, k, 0))]
        for i in range(9):
            _handle(i).workspace(need[0] if 1 <= i <= 4 else need[1])
        return st
    m, n = c["d_in"], c["d_out"]
    st["x"] = _planted(l, m, k, SIGMA_X, seed + 1)
    w = _planted(n, m, k, SIGMA_W, seed + 2)
    if c["op"] == "forward":
        st["xo"] = B.Operand(l, m, k, axes=B.BLOCKS_ALONG_COLS)
        st["wo"] = h.split(w, k, p, sketch=B.SKETCH_FULL, seed=st["seed"] + 2, axes=B.BLOCKS_ALONG_COLS)
        return st
    st["d"] = _planted(l, n, k, SIGMA_D, seed + 3)
    st["xo"], st["do"] = B.Operand(l, m, k), B.Operand(l, n, k)
    if c["weights"] == "stored":
        st["wo"], st["w_res"] = h.split(w, k, p, sketch=B.SKETCH_FULL, seed=st["seed"] + 2, want_residual=True)
    else:
        st["w"], st["wo"] = w, B.Operand(n, m, k)
    return st


def _run_block(st):
    """Layer j's weight is split on one of four weight streams, its gradient is split and its backward products run on one of
    four gradient streams; activations and forward products stay on the current stream."""
    c, seed = st["case"], st["seed"]
    k, p, main = c["k"], c["p"], torch.cuda.current_stream()
    start = main.record_event()
    w_done, x_done, used = [], {}, set()
    for j, ly in enumerate(st["layers"]):
        i = 1 + j % 4
        sw = _stream(i)
        sw.wait_event(start)
        _handle(i).split(ly["w"], k, p, sketch=B.SKETCH_FULL, seed=seed + 2, out=ly["wo"], stream=sw)
        w_done.append(sw.record_event())
    for j, ly in enumerate(st["layers"]):
        g = ly["x"]
        if g not in x_done:
            _handle(0).split(st["xs"][g], k, p, seed=seed + 1, out=st["xo"][g])
            x_done[g] = main.record_event()
        main.wait_event(w_done[j])
        _handle(0).linear_fwd(st["xo"][g], ly["wo"], out=ly["y"])
        i = 5 + j % 4
        sd = _stream(i)
        sd.wait_event(start)
        _handle(i).split(ly["d"], k, p, seed=seed + 3, rounding=B.ROUND_SR, out=ly["do"], stream=sd)
        sd.wait_event(x_done[g])
        sd.wait_event(w_done[j])
        _handle(i).linear_bwd(ly["do"], st["xo"][g], ly["wo"], out=(ly["dx"], ly["dw"]), stream=sd)
        used.add(i)
    for i in used:
        main.wait_event(_stream(i).record_event())
    return [(ly["y"], ly["dx"], ly["dw"]) for ly in st["layers"]]


def run(st):
    c, h, seed = st["case"], _handle(0), st["seed"]
    if c["op"] == "quantize":
        axes = {"both": B.BLOCKS_BOTH, "cols": B.BLOCKS_ALONG_COLS, "rows": B.BLOCKS_ALONG_ROWS}[c["axes"]]
        h.quantize_nvfp4(st["x"], axes=axes, rounding=B.ROUND_SR if c["rounding"] == "sr" else B.ROUND_RNE, seed=seed, out=st["out"])
        return [(o.codes, o.scales, o.tensor_scale) for o in st["out"] if o is not None]
    if c["op"] == "block":
        return _run_block(st)
    k, p, out = c["k"], c["p"], _dtype(c["out"])
    if c["op"] == "forward":
        h.split(st["x"], k, p, seed=seed + 1, axes=B.BLOCKS_ALONG_COLS, out=st["xo"])
        return h.linear_fwd(st["xo"], st["wo"], out_dtype=out)
    act = B.SKETCH_FULL if c["act_sketch"] == "full" else B.SKETCH_SAMPLED
    wo, grads = st["wo"], None
    h.split(st["x"], k, p, sketch=act, seed=seed + 1, out=st["xo"])
    if c["weights"] == "stored":
        h.requantize_operand(wo, st["w_res"], seed=seed + 2)
        grads = tuple(torch.empty(s, dtype=torch.float32, device="cuda") for s in ((k, c["d_out"]), (k,), (k, c["d_in"])))
    else:
        h.split(st["w"], k, p, sketch=B.SKETCH_FULL, seed=seed + 2, out=wo)
    y = h.linear_fwd(st["xo"], wo, out_dtype=out)
    h.split(st["d"], k, p, sketch=act, seed=seed + 3, rounding=B.ROUND_SR, out=st["do"])
    dx, dw = h.linear_bwd(st["do"], st["xo"], wo, out_dtype=out, factor_grads=grads)
    return [y, dx, dw] + list(grads or ())


def work(case):
    """Bytes: every tensor handed in once and every tensor handed back once.  Flops: the products (three of 2 l m n in a step)."""
    c = case
    if c["op"] == "quantize":
        e, each = c["rows"] * c["cols"], 2 if c["axes"] == "both" else 1
        return {"bytes": e * ((2 if c["dtype"] == "bf16" else 4) + each * 0.5625), "flops": 0}
    l = c["tokens"]
    if c["op"] == "block":
        dims = _block_dims(c)
        x = sum(l * dims[BLOCK_X.index(g)][0] for g in range(4))
        return {"bytes": 2 * (x + sum(2 * m * n + 2 * l * n + l * m for m, n in dims)), "flops": sum(6 * l * m * n for m, n in dims)}
    m, n, es = c["d_in"], c["d_out"], 2 if c["out"] == "bf16" else 4
    if c["op"] == "forward":                       # the kept weight operand is read as codes and scales
        return {"bytes": 2 * l * m + 0.5625 * n * m + es * l * n, "flops": 2 * l * m * n}
    w_in = 4 * (n * m + c["k"] * (n + m)) if c["weights"] == "stored" else 2 * n * m
    grads = 4 * c["k"] * (n + m + 1) if c["weights"] == "stored" else 0
    return {"bytes": 2 * (l * m + l * n) + w_in + es * (l * n + l * m + n * m) + grads, "flops": 6 * l * m * n}


def tolerance(case):
    c = case
    if c["op"] == "quantize":
        return "exact"                             # defined in binary32, operation by operation
    if c["k"] == 0:
        # exact codes, FP32 accumulation (3e-8 of a float64 product; the order of the sum changed nothing), output rounding
        return {"rel": 2e-4, "max": 8e-3} if c["out"] == "bf16" else {"rel": 1e-6, "max": 1e-5}
    # A factor entry on a rounding midpoint becomes another FP4 code when the decomposition's FP32 sums are taken in another
    # order.  Full decompositions of a token batch and of the same batch with its 128-row tiles permuted, k = 4 ... 128: the
    # outputs differ by up to 3.0e-3 in norm and 0.44 in the largest entry (against float64: 2e-4 and 0.01 at 1088 tokens).
    return {"rel": 1.2e-2, "max": 0.95}
