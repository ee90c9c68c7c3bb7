"""Performance cases: the work that a user of this library has it do, through its public calls.

Three directions: products from compressed weights (decode-phase matrix-vector and small-batch products, alone and as the
launches of a decoder layer), decompression of a whole tensor, and compression on the device of a tensor being loaded.

Weights and activations are synthetic (no checkpoints here): N(0, std^2) times a per-row scale U(0.5, 2), rounded to the
stored type, which compresses like trained LLM weights do (11.7 .. 11.8 payload bits per BF16 weight); activations N(0, 1).
"fp16_from_bf16" are BF16-trained weights stored as FP16 (low mantissa bits mostly zero), "fp16" FP16-trained ones.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_2502_00922_b200 as hl

_FP16 = ("fp16", "fp16_from_bf16")


def _product(name, rows, cols, batch, dtype="bf16", chunk=4096, limit=0):
    return {"name": name, "kind": "product", "rows": rows, "cols": cols, "batch": batch, "dtype": dtype, "chunk": chunk, "limit": limit}


def _layer(name, hidden, kv, ffn, batch, dtype="bf16", chunk=4096):
    return {"name": name, "kind": "layer", "hidden": hidden, "kv": kv, "ffn": ffn, "batch": batch, "dtype": dtype, "chunk": chunk, "limit": 0}


def listed():
    return [
        # one k or v projection of the 8B-shaped layer, one token: the smallest call, where latency counts
        _product("gemv_kv_8b", 1024, 4096, 1),
        # the Llama-7B-shaped layer, one token: q+k+v | o | gate+up | down, the four launches its data dependencies allow
        _layer("layer_7b_b1", 4096, 4096, 11008, 1),
        # one matrix of the 70B-shaped FFN, one token: the largest matrix-vector product
        _product("gemv_up_70b", 28672, 8192, 1),
        # the 8B-shaped layer (grouped-query attention) for a handful of sequences
        _layer("layer_8b_b4", 4096, 1024, 14336, 4),
        # the 8B-shaped down projection for 16 sequences
        _product("gemm_down_8b_b16", 4096, 14336, 16),
        # the 7B-shaped layer served at 32 sequences
        _layer("layer_7b_b32", 4096, 4096, 11008, 32),
        # the 70B-shaped down projection at the widest batch
        _product("gemm_down_70b_b64", 8192, 28672, 64),
        # FP16-trained weights, one token (the 7B-shaped gate)
        _product("gemv_fp16_gate_7b", 11008, 4096, 1, "fp16", 2048),
        # BF16-trained weights stored as FP16, a batch of 24
        _product("gemm_fp16_down_7b_b24", 4096, 11008, 24, "fp16_from_bf16", 2048),
        # the paper's quoted codeword bound, L_max = 12
        _product("gemv_lmax12_gate_7b", 11008, 4096, 1, limit=12),
        # a whole tensor back to its 16-bit weights; odd sizes
        {"name": "decode_odd", "kind": "decode", "rows": 11007, "cols": 4099, "dtype": "bf16", "chunk": 4096, "limit": 0},
        # a 7B-shaped gate matrix compressed while a model is being loaded: field counts, codebook, encoder
        {"name": "compress_gate_7b", "kind": "compress", "rows": 11008, "cols": 4096, "dtype": "bf16", "chunk": 4096, "limit": 0},
    ]


def _log_size(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choices(["product", "layer", "decode", "compress"], [45, 20, 15, 20])[0]
    dtype = rng.choices(["bf16", "fp16", "fp16_from_bf16"], [70, 15, 15])[0]
    chunk = rng.choice([2048, 4096, 4096, 4096, 8192]) if dtype == "bf16" else rng.choice([1024, 2048, 2048, 4096])
    batch = rng.choice([1, _log_size(rng, 1, 64)])
    if kind == "layer":
        hidden = 128 * _log_size(rng, 8, 40)                         # 1024 .. 5120
        kv = hidden if rng.random() < 0.5 else max(256, hidden // 4)
        ffn = 32 * round(hidden * rng.uniform(2.5, 3.5) / 32)
        if dtype in _FP16 and 8 < batch <= 16:                       # launches over several FP16 matrices take 1..8 and 17..64
            batch = 8
        return {"kind": kind, "hidden": hidden, "kv": kv, "ffn": ffn, "batch": batch, "dtype": dtype, "chunk": chunk, "limit": 0}
    limit = rng.choice([0, 0, 0, 0, 9, 10, 12]) if dtype == "bf16" and chunk <= 4096 else rng.choice([0, 0, 0, 7]) if dtype in _FP16 else 0
    most = 11008 * 4096 if kind == "compress" else 4096 * 28672
    rows = _log_size(rng, 250, 28672)                                # odd as often as not
    cols = _log_size(rng, 1000, max(1001, min(28672, most // rows)))
    if kind == "product":
        cols = (cols + 31) // 32 * 32                                # what the fused products take
        return {"kind": kind, "rows": rows, "cols": cols, "batch": batch, "dtype": dtype, "chunk": chunk, "limit": limit}
    return {"kind": kind, "rows": rows, "cols": cols, "dtype": dtype, "chunk": chunk, "limit": limit}


# ------------------------------------------------------------------------------------------------ inputs

def _weights(rows, cols, dtype, gen):
    """16-bit patterns of one matrix, on the GPU (torch.int16)."""
    w = torch.randn((rows, cols), generator=gen, device="cuda", dtype=torch.float32)
    scale = torch.rand((rows, 1), generator=gen, device="cuda", dtype=torch.float32) * 1.5 + 0.5
    w *= scale * 0.02
    if dtype == "bf16":
        return w.to(torch.bfloat16).view(torch.int16)
    if dtype == "fp16":
        return w.to(torch.float16).view(torch.int16)
    return w.to(torch.bfloat16).to(torch.float16).view(torch.int16)


def _activations(batch, cols, dtype, gen):
    x = torch.randn((batch, cols), generator=gen, device="cuda", dtype=torch.float32)
    return x.to(torch.float16 if dtype in _FP16 else torch.bfloat16).view(torch.int16)


def _dtype(case):
    return hl.FP16 if case["dtype"] in _FP16 else hl.BF16


def _split(case):
    return [1, 5, 5, 5] if case["dtype"] in _FP16 else [1, 8, 7]


def _compress(w, case, counts, blob, scratch):
    """What a loader does with one tensor: count its fields, build the codebook from the counts, encode."""
    rows, cols = w.shape
    hl.split_histogram(w, rows * cols, _split(case), counts)
    c = counts.cpu().numpy().view(np.uint64)
    cb = hl.build_codebook_from_counts(c[2:] if case["dtype"] in _FP16 else c[2:258], _dtype(case), case["limit"])
    desc = hl.encode_device(cb, w, rows, cols, case["chunk"], blob, blob.numel(), scratch, scratch.numel())
    cb.free()
    return desc


def _buffers(rows, cols, case):
    counts = torch.zeros(hl.split_counts_size(_split(case)), dtype=torch.int64, device="cuda")
    blob = torch.zeros(hl.encode_bound(rows, cols, _dtype(case), case["chunk"]), dtype=torch.uint8, device="cuda")
    scratch = torch.zeros(hl.encode_device_scratch_bytes(rows, cols, case["chunk"]), dtype=torch.uint8, device="cuda")
    return counts, blob, scratch


def _encoded(rows, cols, case, gen):
    """(descriptor, blob on the device trimmed to its size) of one matrix."""
    w = _weights(rows, cols, case["dtype"], gen)
    counts, blob, scratch = _buffers(rows, cols, case)
    desc = _compress(w, case, counts, blob, scratch)
    return desc, blob[:desc.blob_bytes].clone()


def _layer_groups(case):
    h, kv, f = case["hidden"], case["kv"], case["ffn"]
    return [[(h, h), (kv, h), (kv, h)], [(h, h)], [(f, h), (f, h)], [(h, f)]]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    state = {"case": case, "err": err}
    if case["kind"] == "compress":
        rows, cols = case["rows"], case["cols"]
        state["w"] = _weights(rows, cols, case["dtype"], gen)
        state["buffers"] = _buffers(rows, cols, case)
        return state
    if case["kind"] == "decode":
        rows, cols = case["rows"], case["cols"]
        state["desc"], state["blob"] = _encoded(rows, cols, case, gen)
        state["out"] = torch.zeros((rows, cols), dtype=torch.int16, device="cuda")
        return state
    batch = case["batch"]
    groups = _layer_groups(case) if case["kind"] == "layer" else [[(case["rows"], case["cols"])]]
    state["ys"], state["calls"] = [], []
    for shapes in groups:
        descs, blobs, xs, ys = [], [], [], []
        x = _activations(batch, shapes[0][1], case["dtype"], gen)     # the matrices of a launch share their input
        for rows, cols in shapes:
            desc, blob = _encoded(rows, cols, case, gen)
            descs.append(desc)
            blobs.append(blob)
            xs.append(x)
            ys.append(torch.zeros((batch, rows), dtype=torch.float32, device="cuda"))
        ws_bytes = max(hl.workspace_bytes(d, batch) for d in descs)
        wss = [torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda") for _ in descs]
        state["ys"] += ys
        if case["kind"] == "layer":
            state["calls"].append(hl.PreparedMulti(descs, blobs, xs, batch, ys, wss, ws_bytes, err))
        else:
            state["single"] = (descs[0], blobs[0], x, ys[0], wss[0], ws_bytes)
    return state


# ------------------------------------------------------------------------------------------------ one pass

def run(state):
    case, err = state["case"], state["err"]
    if case["kind"] == "layer":
        stream = torch.cuda.current_stream().cuda_stream
        for call in state["calls"]:
            call.run(stream)
        return state["ys"] + [err]
    if case["kind"] == "product":
        desc, blob, x, y, ws, ws_bytes = state["single"]
        if case["batch"] == 1:
            hl.decode_gemv(desc, blob, x, y, ws, ws_bytes, err)
        else:
            hl.decode_gemm(desc, blob, x, case["batch"], y, ws, ws_bytes, err)
        return [y, err]
    if case["kind"] == "decode":
        hl.decode(state["desc"], state["blob"], state["out"], err)
        return [state["out"], err]
    counts, blob, scratch = state["buffers"]
    desc = _compress(state["w"], case, counts, blob, scratch)
    return [counts, blob, np.frombuffer(bytes(desc), dtype=np.uint8)]      # (the buffer behind the blob stays as it was)


# ------------------------------------------------------------------------------------------------ what a pass cannot do without

def _blob_bytes_per_weight(case):
    """Raw and coded bits of these weights (the blob's payload without padding, index and table)."""
    if case["dtype"] == "fp16":
        return 13.72 / 8
    if case["dtype"] == "fp16_from_bf16":
        return 10.98 / 8
    return 11.75 / 8


def work(case):
    per = _blob_bytes_per_weight(case)
    if case["kind"] in ("decode", "compress"):
        n = case["rows"] * case["cols"]
        return {"bytes": n * (2 + per), "flops": 0}
    groups = _layer_groups(case) if case["kind"] == "layer" else [[(case["rows"], case["cols"])]]
    n = sum(r * c for g in groups for r, c in g)
    xs, ys = sum(g[0][1] for g in groups), sum(r for g in groups for r, _ in g)
    return {"bytes": n * per + case["batch"] * (2 * xs + 4 * ys), "flops": 2 * n * case["batch"]}


def tolerance(case):
    if case["kind"] in ("decode", "compress"):
        return "exact"
    # Products of 16-bit values are exact in fp32, sums are taken in fp32 in an order of the implementation's choosing.
    # Against the same product in 64 bits: one vector (multiply-adds, each rounded) 0.9e-7 .. 2.3e-7 over the listed shapes;
    # more vectors (the tensor cores' fp32 accumulators) 2.3e-7 .. 3.8e-6, growing with the columns.  About four times that.
    return {"rel": 2e-6 if case["batch"] == 1 else 1.5e-5}


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits: the weights as they were before compression times the activations."""
    if case["kind"] in ("decode", "compress"):
        return None
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = torch.float16 if case["dtype"] in _FP16 else torch.bfloat16
    groups = _layer_groups(case) if case["kind"] == "layer" else [[(case["rows"], case["cols"])]]
    ys = []
    for shapes in groups:                                            # (drawn from the generator in prepare()'s order)
        x = _activations(case["batch"], shapes[0][1], case["dtype"], gen).view(kind).double()
        for rows, cols in shapes:
            w = _weights(rows, cols, case["dtype"], gen).view(kind).double()
            ys.append(x @ w.T)
            del w
    return ys + [None]                                               # (the error flag has no such value)
