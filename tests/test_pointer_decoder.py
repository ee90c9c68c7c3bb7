"""The decoders that keep nothing of a bit sequence but its pointer: how far a damaged blob can move them (CPU), and the
FP16 decoders that read flat mantissa codes without tables (GPU)."""
import numpy as np
import pytest

import workloads as wl
from oracle import oracle as orc

# decoder: (dtype, limit, flat bits per weight, fields looked up in a table, window rows read behind the pointer's)
DECODERS = [("bf16", 8, 0, 1, 1), ("bf16", 9, 0, 1, 2), ("bf16", 12, 0, 1, 2), ("fp16", 8, 0, 3, 2), ("fp16", 7, 0, 3, 2),
            ("fp16", 12, 0, 3, 2), ("fp16", 8, 10, 1, 2), ("fp16", 8, 5, 2, 2)]


@pytest.mark.parametrize("dtype,limit,flat,fields,ahead", DECODERS)
@pytest.mark.parametrize("chunk_elems", [512, 4096, 16384])
def test_no_table_can_move_a_pointer_past_the_guard(dtype, limit, flat, fields, ahead, chunk_elems):
    """The tables in shared memory hold no length above the limit, so after n weights a sequence stands at most
    lag + n * (fields * limit + flat) bits into its rows; the furthest row a window reads from there must lie inside the
    smallest slot (one row) and the guard area behind it."""
    import paper_2502_00922_b200 as hl
    w = wl.gaussian_weights(16, chunk_elems // 16, 0.02, 3, "fp16") if dtype == "fp16" else wl.skewed_exponent_weights(16, chunk_elems // 16, 3)
    cb = hl.build_codebook(w, hl.FP16 if dtype == "fp16" else hl.BF16, limit)
    _, desc = hl.encode(cb, w, chunk_elems)
    cb.free()
    weights = desc.chunk_cols // 32 * 8
    last_window = 4 if dtype == "bf16" else 1 if limit == 12 else 2            # weights of the last window taken
    bits = desc.lag_bits + (weights - last_window) * (fields * limit + flat)
    assert (bits // 32 + ahead + 1) * 256 <= 256 + hl.decode_smem_plan(desc)["guard_bytes"]


@pytest.fixture(scope="module")
def hl():
    import paper_2502_00922_b200 as m
    m.lib()
    return m


def weights(kind, rows, cols, seed):
    if kind == "no field flat":
        return wl.all_patterns_weights(rows, cols, seed) & np.uint16(0xFDF7)     # mantissa halves of 16 symbols each
    return wl.gaussian_weights(rows, cols, 0.02, seed, "fp16" if kind == "both flat" else "fp16_from_bf16")


@pytest.mark.gpu
@pytest.mark.parametrize("kind,flat", [("both flat", 6), ("upper flat", 2), ("no field flat", None)])
@pytest.mark.parametrize("limit", [7, 8, 12])
@pytest.mark.parametrize("rows,cols,chunk", [(16, 32, 512), (250, 1024, 1024), (37, 4128, 2048), (129, 2080, 4096)])
def test_fp16_decoders_by_their_flat_codes(hl, kind, flat, limit, rows, cols, chunk):
    """One block, ragged rows, a last column chunk of one block, odd block counts; tables of 7 bits serve the decoders of flat
    codes as tables of 8.  Products against the oracle; the bound is the rounding of fp32 sums of cols terms."""
    import torch
    w = weights(kind, rows, cols, rows + cols)
    cb = hl.build_codebook(w, hl.FP16, limit)
    blob, desc = hl.encode(cb, w, chunk)
    cb.free()
    if rows * cols > 100000:
        assert desc.flat_fields & 6 == flat if flat is not None else desc.flat_fields & 2 == 0
    dev, err = torch.from_numpy(blob).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.zeros(rows * cols, dtype=torch.int16, device="cuda")
    hl.decode(desc, dev, out, err)
    assert np.array_equal(out.cpu().numpy().view(np.uint16).reshape(rows, cols), w)
    if kind == "no field flat":                                       # (infinities and NaN among them)
        return
    for batch in (1, 3, 24):
        x = wl.activations(batch, cols, 7, "fp16")
        xd, y = torch.from_numpy(x.view(np.int16)).cuda(), torch.zeros((batch, rows), dtype=torch.float32, device="cuda")
        n = hl.workspace_bytes(desc, batch)
        ws = torch.zeros(n, dtype=torch.uint8, device="cuda")
        hl.decode_gemm(desc, dev, xd, batch, y, ws, n, err) if batch > 1 else hl.decode_gemv(desc, dev, xd, y, ws, n, err)
        want, size = orc.matmul(w, x, orc.FP16)
        assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - want) <= cols * 2.0**-23 * size)
    assert int(err.item()) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("limit", [7, 8, 12])
@pytest.mark.parametrize("rows,cols,chunk", [(250, 1024, 512), (129, 2080, 1024), (37, 4128, 2048)])
def test_fp16_products_through_three_tables(hl, limit, rows, cols, chunk):
    """Fields none of which is flat: every product goes through the tables of all three, on the register path and the tensor cores."""
    import torch
    w = wl.skewed_exponent_weights(rows, cols, rows + limit, dtype="fp16")
    cb = hl.build_codebook(w, hl.FP16, limit)
    blob, desc = hl.encode(cb, w, chunk)
    cb.free()
    assert desc.flat_fields & 6 == 0 and desc.lut_bits == limit
    dev, err = torch.from_numpy(blob).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    for batch in (1, 3, 8, 12, 24, 40):
        x = wl.activations(batch, cols, 7, "fp16")
        xd, y = torch.from_numpy(x.view(np.int16)).cuda(), torch.zeros((batch, rows), dtype=torch.float32, device="cuda")
        n = hl.workspace_bytes(desc, batch)
        ws = torch.zeros(n, dtype=torch.uint8, device="cuda")
        hl.decode_gemm(desc, dev, xd, batch, y, ws, n, err) if batch > 1 else hl.decode_gemv(desc, dev, xd, y, ws, n, err)
        want, size = orc.matmul(w, x, orc.FP16)
        assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - want) <= cols * 2.0**-23 * size)
    assert int(err.item()) == 0


@pytest.mark.gpu
def test_a_launch_reads_without_tables_what_all_its_matrices_allow(hl):
    """A matrix of two flat mantissa halves beside one of which only the upper half is flat."""
    import torch
    rows, cols, descs, blobs, ws = 144, 1024, [], [], []
    mats = [weights(k, rows, cols, 5) for k in ("both flat", "upper flat")]
    for w in mats:
        cb = hl.build_codebook(w, hl.FP16, 8)
        blob, d = hl.encode(cb, w, 2048)
        cb.free()
        descs.append(d)
        blobs.append(torch.from_numpy(blob).cuda())
    assert [d.flat_fields & 6 for d in descs] == [6, 2]
    for batch in (1, 32):
        x = wl.activations(batch, cols, 7, "fp16")
        xd = torch.from_numpy(x.view(np.int16)).cuda()
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        ys = [torch.zeros((batch, rows), dtype=torch.float32, device="cuda") for _ in mats]
        n = max(hl.workspace_bytes(d, batch) for d in descs)
        ws = [torch.zeros(n, dtype=torch.uint8, device="cuda") for _ in mats]
        hl.decode_gemm_multi(descs, blobs, [xd, xd], batch, ys, ws, n, err)
        assert int(err.item()) == 0
        for w, y in zip(mats, ys):
            want, size = orc.matmul(w, x, orc.FP16)
            assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - want) <= cols * 2.0**-23 * size)
