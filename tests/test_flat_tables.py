"""FP16 blobs whose mantissa halves are both flat keep one table, with sixteen copies of an entry or with one per lane: the plans
that choose (CPU) and both layouts in every kernel that has them (GPU)."""
import numpy as np
import pytest

import workloads as wl
from oracle import oracle as orc


@pytest.fixture(scope="module")
def hl():
    import paper_2502_00922_b200 as m
    m.lib()
    return m


def flat_blob(hl, rows, cols, chunk):
    w = wl.gaussian_weights(rows, cols, 0.02, rows + cols, "fp16")
    cb = hl.build_codebook(w, hl.FP16, 0)
    blob, d = hl.encode(cb, w, chunk)
    cb.free()
    assert d.flat_fields & 6 == 6
    return w, blob, d


def planned(hl, rows, cols, chunk, words):
    """The descriptor of a rows x cols matrix whose largest record has `words` rows, without the matrix."""
    d = flat_blob(hl, 256, 2048, chunk)[2]
    d.rows, d.cols, d.row_groups, d.max_words = rows, cols, (rows + 15) // 16, words
    d.col_chunks = (cols + d.chunk_cols - 1) // d.chunk_cols
    d.n_chunks = d.row_groups * d.col_chunks
    d.off_payload = (d.off_index + 4 * (d.n_chunks + 1) + 255) // 256 * 256
    d.payload_bytes, d.blob_bytes = 128 * d.n_chunks, d.off_payload + 128 * d.n_chunks + 4096
    return d


@pytest.mark.parametrize("rows,cols,most", [(12288, 12288, 11), (8192, 28672, 18), (4096, 14336, 9), (4096, 11008, 7), (11008, 4096, 7),
                                            (28672, 8192, 10), (14336, 4096, 11)])
@pytest.mark.parametrize("batch", [9, 16, 24, 32, 48, 64])
def test_no_sum_gets_longer_for_a_table_per_lane(hl, rows, cols, most, batch):
    """Records of 15 rows (N(0, 0.02^2), chunks of 2048): 24 decoders beside sixteen copies, 16 beside one per lane, whose sums
    would be up to three times as long.  In any workspace that the size call gives, the same."""
    d = planned(hl, rows, cols, 2048, 15)
    free = hl.gemm_launch_plan([d], batch)
    assert free["chunks_per_sum"][0] <= most
    for sized_for in {batch, 64}:
        assert hl.gemm_launch_plan([d], batch, hl.workspace_bytes(d, sized_for)) == free


@pytest.mark.parametrize("chunk,words,batch,warps", [(4096, 28, 1, 26), (4096, 28, 4, 26), (4096, 28, 8, 24), (8192, 54, 1, 12),
                                                      (2048, 14, 1, 25), (1024, 8, 8, 31)])
def test_few_vectors_keep_the_warps_that_keep_sums_short(hl, chunk, words, batch, warps):
    """11008 x 4096: long chunks keep the warps they have beside sixteen copies (one per lane would leave 24, 22 and 10); chunks of
    2048 are six a warp with 27 warps and with the 25 beside a table per lane."""
    assert hl.decode_launch_plan(planned(hl, 11008, 4096, chunk, words), batch)["decoder_warps"] == warps


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,chunk", [(11008, 4096, 4096), (2400, 1056, 2048), (1250, 2080, 1024), (144, 8192, 8192)])
def test_both_layouts_of_the_table(hl, rows, cols, chunk):
    """Whole and ragged tiles, launches that choose either layout; decode bit by bit, products on sampled rows, bound: the rounding
    of fp32 sums of cols terms."""
    import torch
    w, blob, d = flat_blob(hl, rows, cols, chunk)
    dev, err = torch.from_numpy(blob).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.zeros(rows * cols, dtype=torch.int16, device="cuda")
    hl.decode(d, dev, out, err)
    assert np.array_equal(out.cpu().numpy().view(np.uint16).reshape(rows, cols), w)
    pick = np.unique(np.concatenate([np.arange(0, rows, max(1, rows // 64)), np.arange(max(0, rows - 17), rows)]))
    for batch in (1, 2, 8, 12, 32, 50):
        x = wl.activations(batch, cols, 7, "fp16")
        xd, y = torch.from_numpy(x.view(np.int16)).cuda(), torch.zeros((batch, rows), dtype=torch.float32, device="cuda")
        n = hl.workspace_bytes(d, batch)
        ws = torch.zeros(n, dtype=torch.uint8, device="cuda")
        hl.decode_gemm(d, dev, xd, batch, y, ws, n, err) if batch > 1 else hl.decode_gemv(d, dev, xd, y, ws, n, err)
        want, size = orc.matmul(w[pick], x, orc.FP16)
        assert np.all(np.abs(y.cpu().numpy()[:, pick].astype(np.float64) - want) <= cols * 2.0**-23 * size)
    assert int(err.item()) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("batch", [2, 32])
def test_several_matrices_share_a_layout(hl, batch):
    import torch
    mats = [flat_blob(hl, rows, 2048, 2048) for rows in (2048, 512, 528)]
    x = wl.activations(batch, 2048, 7, "fp16")
    xd, err = torch.from_numpy(x.view(np.int16)).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    ys = [torch.zeros((batch, m[2].rows), dtype=torch.float32, device="cuda") for m in mats]
    n = max(hl.workspace_bytes(m[2], batch) for m in mats)
    ws = [torch.zeros(n, dtype=torch.uint8, device="cuda") for _ in mats]
    hl.decode_gemm_multi([m[2] for m in mats], [torch.from_numpy(m[1]).cuda() for m in mats], [xd] * 3, batch, ys, ws, n, err)
    assert int(err.item()) == 0
    for (w, _, _), y in zip(mats, ys):
        want, size = orc.matmul(w, x, orc.FP16)
        assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - want) <= 2048 * 2.0**-23 * size)
