"""Compression of weights that sit in device memory: counts on the device, codebook from the counts, encoder on the
device.  The blob must be the host encoder's byte for byte, and the oracle's slow reader must get the tensor back."""
import numpy as np
import pytest

import workloads as wl
from oracle import oracle as orc


@pytest.fixture(scope="module")
def hl():
    import paper_2502_00922_b200 as m
    m.lib()
    return m


def gen(kind, rows, cols, seed):
    return {"gauss": lambda: wl.gaussian_weights(rows, cols, 0.02, seed),
            "fp16": lambda: wl.gaussian_weights(rows, cols, 0.02, seed, "fp16"),
            "fp16_from_bf16": lambda: wl.gaussian_weights(rows, cols, 0.02, seed, "fp16_from_bf16"),
            "student": lambda: wl.student_t_weights(rows, cols, seed),
            "patterns": lambda: wl.all_patterns_weights(rows, cols, seed),
            "constant": lambda: np.full((rows, cols), 0xBD33, dtype=np.uint16)}[kind]()


def counts_for_codebook(w, dtype):
    """The counters huffllm_build_codebook_from_counts wants, taken from the oracle's field histograms."""
    if dtype == 1:
        return np.concatenate(orc.split_histograms(w, [1, 5, 5, 5])[1:])
    return orc.split_histograms(w, [1, 8, 7])[1]


# ------------------------------------------------------------------ host part: codebook from counts

@pytest.mark.parametrize("kind,dtype,split,budget", [("gauss", 0, 0, 0), ("gauss", 0, 1, 0), ("student", 0, 0, 9), ("fp16", 1, 0, 0),
                                                     ("fp16_from_bf16", 1, 0, 0), ("constant", 0, 0, 0), ("patterns", 0, 1, 9)])
def test_codebook_from_counts_is_the_codebook_of_the_tensor(hl, kind, dtype, split, budget):
    w = gen(kind, 48, 640, 4)
    cb_a = hl.build_codebook(w, dtype, budget, split)
    cb_b = hl.build_codebook_from_counts(counts_for_codebook(w, dtype), dtype, budget, split)
    blob_a, desc_a = hl.encode(cb_a, w, 1024)
    blob_b, desc_b = hl.encode(cb_b, w, 1024)
    assert np.array_equal(blob_a, blob_b) and bytes(desc_a) == bytes(desc_b)
    cb_a.free()
    cb_b.free()


def test_codebook_from_counts_refuses_nonsense(hl):
    with pytest.raises(hl.HuffllmError):
        hl.build_codebook_from_counts(np.zeros(256, dtype=np.uint64), 0)           # nothing counted
    with pytest.raises(hl.HuffllmError):
        hl.build_codebook_from_counts(np.ones(96, dtype=np.uint64), 1, 0, 1)       # whole-exponent split is for bf16
    with pytest.raises(ValueError):
        hl.build_codebook_from_counts(np.ones(96, dtype=np.uint64), 0)


# ------------------------------------------------------------------ device part

CASES = [  # rows, cols, chunk_elems, kind, dtype, split, budget
    (64, 1024, 4096, "gauss", 0, 0, 0),
    (100, 1000, 2048, "gauss", 0, 0, 0),            # ragged rows, columns a multiple of 8 but not of 32
    (37, 333, 512, "student", 0, 0, 9),             # nothing aligned: scalar loads, pad words
    (16, 32, 512, "constant", 0, 0, 0),             # a single block, a single symbol
    (48, 2080, 1024, "patterns", 0, 1, 9),          # whole-exponent code, every exponent in use
    (64, 1024, 1024, "fp16", 1, 0, 0),
    (50, 1096, 2048, "fp16_from_bf16", 1, 0, 0),    # FP16, odd block count in the last chunk (sign plane padding)
    (33, 100, 512, "fp16", 1, 0, 0),
    (512, 4096, 4096, "gauss", 0, 0, 0),
]


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,ce,kind,dtype,split,budget", CASES)
def test_device_encoder_writes_the_host_encoders_blob(hl, rows, cols, ce, kind, dtype, split, budget):
    import torch
    w = gen(kind, rows, cols, 12)
    w_dev = torch.from_numpy(w.view(np.int16)).cuda()
    # counts on the device -> codebook
    widths = [1, 5, 5, 5] if dtype == 1 else [1, 8, 7]
    counts = torch.zeros(hl.split_counts_size(widths), dtype=torch.int64, device="cuda")
    hl.split_histogram(w_dev, rows * cols, widths, counts)
    c = counts.cpu().numpy().view(np.uint64)
    cb = hl.build_codebook_from_counts(c[2:98] if dtype == 1 else c[2:258], dtype, budget, split)
    # encode on the device
    cap = hl.encode_bound(rows, cols, dtype, ce)
    blob_dev = torch.full((cap + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    n_scr = hl.encode_device_scratch_bytes(rows, cols, ce)
    scratch = torch.full((n_scr,), 0x5A, dtype=torch.uint8, device="cuda")
    desc = hl.encode_device(cb, w_dev, rows, cols, ce, blob_dev, cap, scratch, n_scr)
    got = blob_dev.cpu().numpy()
    assert np.all(got[desc.blob_bytes:] == 0xA5), "wrote behind the blob"
    got = got[:desc.blob_bytes]
    # the host encoder's blob, byte for byte
    cb_host = hl.build_codebook(w, dtype, budget, split)
    want, desc_host = hl.encode(cb_host, w, ce)
    assert bytes(desc) == bytes(desc_host)
    assert np.array_equal(got, want)
    hl.validate_blob(got)
    # and, independently of the host encoder, the oracle's reader gets the tensor back
    if rows * cols <= 1 << 17:
        back, _ = orc.decode_blob(got)
        assert np.array_equal(back, w)
    cb.free()
    cb_host.free()


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,ce,kind,dtype,budget,offset", [
    (40, 1023, 1024, "gauss", 0, 0, 1),              # rows on every 2-byte boundary, the tensor itself off 4 bytes
    (17, 4094, 4096, "gauss", 0, 0, 2),              # rows on 4-byte boundaries
    (16, 4104, 512, "student", 0, 12, 8),            # 16-byte loads, codewords of up to 12 bits (pairs of 24 bits)
    (33, 1030, 16384, "fp16", 1, 12, 3),             # the longest records: several stretches per checksum
    (2, 7, 512, "gauss", 0, 0, 0),                   # one chunk, rows shorter than a thread's eight weights
    (16, 32 * 1023, 512, "constant", 0, 0, 0),       # 1023 / 1024 / 1025 chunks of one block, records of the least size:
    (16, 32 * 1024, 512, "constant", 0, 0, 0),       # around the end of a scan CTA
    (16, 32 * 1025, 512, "constant", 0, 0, 0),
    (1040, 1024, 512, "fp16", 1, 7, 0),              # 2080 chunks, records of an odd number of 128-byte units
    (33, 32 * 20011 - 5, 512, "gauss", 0, 0, 0),     # 60033 chunks: a scan CTA has 58 sums in front of it
    (16, 32 * 20483, 512, "fp16", 1, 12, 2),         # 20483 chunks: a thread per record in the checksum pass
    (48, 32 * 16384 - 9, 512, "gauss", 0, 0, 0),     # 49152 chunks: offsets from sums of 1024 chunks each; the last CTA has none
    (16, 32 * 49151, 512, "constant", 0, 0, 0),      # one fewer: from the chunks themselves
    (16, 32 * 49152, 512, "fp16", 1, 0, 0),
    *[(16, 32 * n, 512, "fp16" if dtype else "gauss", dtype, 0, 0) for n in range(49153, 49159) for dtype in (0, 1)],     # a few behind whole groups
    (16, 32 * 50175, 512, "gauss", 0, 0, 0),         # a group less one
    (2320, 10848, 512, "gauss", 0, 0, 0),            # 49155 chunks in 145 row groups
    (1, 8, 512, "gauss", 0, 0, 0), (5, 4104, 512, "gauss", 0, 0, 0), (15, 1000, 16384, "fp16", 1, 0, 0),     # rows off the tensor beside rows read whole
    (23, 2072, 4096, "student", 0, 12, 0), (24, 8200, 8192, "fp16", 1, 12, 0),
])
def test_device_encoder_at_the_edges_of_its_passes(hl, rows, cols, ce, kind, dtype, budget, offset):
    """Loads that are not aligned, sequences that fill their rows, the scan's and the checksum's borders: host blob, byte for byte."""
    import torch
    w = gen(kind, rows, cols, 5)
    buf = torch.zeros(rows * cols + 16, dtype=torch.int16, device="cuda")
    w_dev = buf[offset:offset + rows * cols]
    w_dev.copy_(torch.from_numpy(w.view(np.int16).reshape(-1)))
    cb = hl.build_codebook(w, dtype, budget)
    cap = hl.encode_bound(rows, cols, dtype, ce)
    blob_dev = torch.full((cap + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    n_scr = hl.encode_device_scratch_bytes(rows, cols, ce)
    scratch = torch.full((n_scr,), 0x5A, dtype=torch.uint8, device="cuda")
    desc = hl.encode_device(cb, w_dev, rows, cols, ce, blob_dev, cap, scratch, n_scr)
    want, desc_host = hl.encode(cb, w, ce)
    got = blob_dev.cpu().numpy()
    assert np.all(got[desc.blob_bytes:] == 0xA5)
    assert bytes(desc) == bytes(desc_host) and np.array_equal(got[:desc.blob_bytes], want)
    # a buffer one byte short is refused and nothing is written behind what it holds
    blob_dev.fill_(0xA5)
    with pytest.raises(hl.HuffllmError) as e:
        hl.encode_device(cb, w_dev, rows, cols, ce, blob_dev, int(desc.blob_bytes) - 1, scratch, n_scr)
    assert e.value.status_name == "BUFFER_TOO_SMALL"
    assert np.all(blob_dev.cpu().numpy()[desc.off_payload:] == 0xA5)
    cb.free()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,budget,ce", [(0, 0, 4096), (0, 12, 16384), (1, 0, 2048), (1, 12, 8192)])
@pytest.mark.parametrize("offset", range(8))
def test_device_encoder_takes_rows_on_any_boundary(hl, dtype, budget, ce, offset):
    """Rows that start on every 2-byte boundary, one to nine whole blocks and a ragged one per chunk, a ragged last row group;
    long codes in long chunks: records of more rows than are collected in shared memory.  Host blob, byte for byte."""
    import torch
    kind = "fp16" if dtype else "student"
    for rows, cols in ((37, 2 * ce // 16 + 32 * (1 + offset) + 8 * (offset % 4) + offset % 2), (16, 40 + 32 * offset)):
        w = gen(kind, rows, cols, 20 + offset)
        buf = torch.zeros(rows * cols + 16, dtype=torch.int16, device="cuda")
        w_dev = buf[offset:offset + rows * cols]
        w_dev.copy_(torch.from_numpy(w.view(np.int16).reshape(-1)))
        cb = hl.build_codebook(w, dtype, budget)
        cap = hl.encode_bound(rows, cols, dtype, ce)
        blob_dev = torch.full((cap + 256,), 0xA5, dtype=torch.uint8, device="cuda")
        n_scr = hl.encode_device_scratch_bytes(rows, cols, ce)
        scratch = torch.full((n_scr,), 0x5A, dtype=torch.uint8, device="cuda")
        desc = hl.encode_device(cb, w_dev, rows, cols, ce, blob_dev, cap, scratch, n_scr)
        want, desc_host = hl.encode(cb, w, ce)
        got = blob_dev.cpu().numpy()
        assert bytes(desc) == bytes(desc_host) and np.array_equal(got[:desc.blob_bytes], want)
        assert np.all(got[desc.blob_bytes:] == 0xA5)
        cb.free()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,kind,rows,cols,ce", [
    (0, "constant", 16, 512, 512), (0, "gauss", 32, 1000, 512), (0, "gauss", 100, 2048, 1024), (1, "fp16", 48, 1024, 1024),
    (0, "gauss", 48, 1040, 2048), (1, "fp16", 48, 1040, 2048), (0, "student", 64, 2100, 4096), (1, "fp16_from_bf16", 64, 2100, 4096),
    (0, "gauss", 33, 4100, 8192), (1, "fp16", 33, 4100, 8192),
    (0, "gauss", 16, 32 * 15047, 512), (0, "gauss", 16, 32 * 15048 - 3, 512),     # 15047 records: a warp each; 15048: a thread each
])
def test_checksums_of_records_of_every_size(hl, dtype, kind, rows, cols, ce):
    """Records that take one to four steps of every size, ends inside a step, more records than warps; the host encoder's checksum."""
    import torch
    w = gen(kind, rows, cols, 31)
    w_dev = torch.from_numpy(w.view(np.int16)).cuda()
    cb = hl.build_codebook(w, dtype)
    cap, n_scr = hl.encode_bound(rows, cols, dtype, ce), hl.encode_device_scratch_bytes(rows, cols, ce)
    blob_dev = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    desc = hl.encode_device(cb, w_dev, rows, cols, ce, blob_dev, cap, torch.zeros(n_scr, dtype=torch.uint8, device="cuda"), n_scr)
    want, desc_host = hl.encode(cb, w, ce)
    assert desc.payload_checksum == desc_host.payload_checksum
    assert np.array_equal(blob_dev[:desc.blob_bytes].cpu().numpy(), want)
    cb.free()


@pytest.mark.gpu
def test_full_size_matrix_on_the_device_equals_the_host_blob(hl):
    """A full-size FFN matrix of the benchmark's layer (45 M weights, 11008 chunks)."""
    import torch
    rows, cols, ce = 11008, 4096, 4096
    w = wl.gaussian_weights(rows, cols, 0.02, 1003)
    w_dev = torch.from_numpy(w.view(np.int16)).cuda()
    counts = torch.zeros(hl.split_counts_size([1, 8, 7]), dtype=torch.int64, device="cuda")
    hl.split_histogram(w_dev, rows * cols, [1, 8, 7], counts)
    cb = hl.build_codebook_from_counts(counts.cpu().numpy().view(np.uint64)[2:258], 0)
    cap = hl.encode_bound(rows, cols, 0, ce)
    blob_dev = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    n_scr = hl.encode_device_scratch_bytes(rows, cols, ce)
    desc = hl.encode_device(cb, w_dev, rows, cols, ce, blob_dev, cap, torch.zeros(n_scr, dtype=torch.uint8, device="cuda"), n_scr)
    cb_host = hl.build_codebook(w, 0)
    want, desc_host = hl.encode(cb_host, w, ce)
    assert bytes(desc) == bytes(desc_host)
    assert np.array_equal(blob_dev[:desc.blob_bytes].cpu().numpy(), want)
    cb.free()
    cb_host.free()


@pytest.mark.gpu
def test_device_encoded_blob_feeds_the_product_kernel(hl):
    import torch
    rows, cols = 256, 2048
    w = wl.gaussian_weights(rows, cols, 0.02, 33)
    w_dev = torch.from_numpy(w.view(np.int16)).cuda()
    counts = torch.zeros(hl.split_counts_size([1, 8, 7]), dtype=torch.int64, device="cuda")
    hl.split_histogram(w_dev, rows * cols, [1, 8, 7], counts)
    cb = hl.build_codebook_from_counts(counts.cpu().numpy().view(np.uint64)[2:258], 0)
    cap = hl.encode_bound(rows, cols, 0, 4096)
    blob_dev = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    n_scr = hl.encode_device_scratch_bytes(rows, cols, 4096)
    desc = hl.encode_device(cb, w_dev, rows, cols, 4096, blob_dev, cap, torch.zeros(n_scr, dtype=torch.uint8, device="cuda"), n_scr)
    x = wl.activations(1, cols, 5)
    x_dev = torch.from_numpy(x.view(np.int16).reshape(-1)).cuda()
    y = torch.zeros(rows, dtype=torch.float32, device="cuda")
    ws_bytes = hl.workspace_bytes(desc, 1)
    ws = torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    hl.decode_gemv(desc, blob_dev, x_dev, y, ws, ws_bytes, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    y_ref, y_abs = orc.matmul(w, x)
    assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - y_ref[0]) <= 2e-3 * y_abs[0] + 1e-30)
    cb.free()


@pytest.mark.gpu
def test_device_encoder_errors(hl):
    import torch
    w = wl.gaussian_weights(32, 256, 0.02, 1)
    w_dev = torch.from_numpy(w.view(np.int16)).cuda()
    cb = hl.build_codebook(w, 0)
    cap = hl.encode_bound(32, 256, 0, 512)
    blob = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    n_scr = hl.encode_device_scratch_bytes(32, 256, 512)
    scr = torch.zeros(n_scr, dtype=torch.uint8, device="cuda")
    with pytest.raises(hl.HuffllmError) as e:
        hl.encode_device(cb, w_dev, 32, 256, 512, blob, 1024, scr, n_scr)            # capacity below the payload
    assert e.value.status_name == "BUFFER_TOO_SMALL"
    with pytest.raises(hl.HuffllmError) as e:
        hl.encode_device(cb, w_dev, 32, 256, 512, blob, cap, scr, 16)                # scratch too small
    assert e.value.status_name == "BUFFER_TOO_SMALL"
    # a weight whose exponent the codebook has never seen
    other = torch.from_numpy(np.full((32, 256), 0x7F00, dtype=np.uint16).view(np.int16)).cuda()
    with pytest.raises(hl.HuffllmError) as e:
        hl.encode_device(cb, other, 32, 256, 512, blob, cap, scr, n_scr)
    assert e.value.status_name == "INVALID_ARG"
    # the same in one weight among so many chunks that their sums take a launch of their own
    many = torch.from_numpy(np.tile(w, (6, 1)).reshape(-1)[:48 * 1024].view(np.int16)).cuda().repeat(512).reshape(48, 32 * 16384)
    many[20, 77777] = 0x7F00
    cap2, scr2 = hl.encode_bound(48, 32 * 16384, 0, 512), hl.encode_device_scratch_bytes(48, 32 * 16384, 512)
    blob2 = torch.full((cap2,), 0xA5, dtype=torch.uint8, device="cuda")
    with pytest.raises(hl.HuffllmError) as e:
        hl.encode_device(cb, many, 48, 32 * 16384, 512, blob2, cap2, torch.zeros(scr2, dtype=torch.uint8, device="cuda"), scr2)
    assert e.value.status_name == "INVALID_ARG"
    assert bool((blob2[512 + 1024 + 4 * 49408:] == 0xA5).all())                       # (behind header, lengths, table and index)
    hl.encode_device(cb, w_dev, 32, 256, 512, blob, cap, scr, n_scr)                 # and the context is still fine
    cb.free()
