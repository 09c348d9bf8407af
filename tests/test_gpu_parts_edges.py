"""Edges of the kernels that split a matrix into its two parts and join them again: every truncation, few and many chunks (four
warps or one on each), windows that begin and end anywhere, gaps longer than 32 bitmap words, codes longer than a window, odd widths and unaligned rows."""
import numpy as np
import pytest
import torch

import synth
from oracle import codec, layout

pytestmark = pytest.mark.gpu


def _bits(t):
    return t.detach().cpu().contiguous().view(torch.int16).numpy().astype(np.uint16)


@pytest.fixture(scope="module")
def cass():
    import paper_2605_26558_b200 as m
    return m


@pytest.mark.parametrize("rows,cols,p,t,seg,chunk", [
    (33, 1, 0, 4, 0, 0), (1, 31, 400, 4, 0, 0), (40, 257, 400, 1, 0, 0), (65, 2049, 300, 2, 0, 0), (31, 4097, 500, 3, 0, 0),
    (35, 1000, 400, 5, 0, 0), (34, 999, 400, 6, 256, 32), (33, 801, 200, 7, 0, 0), (37, 2048, 0, 4, 2048, 2048),
    (32, 4096, 990, 4, 2048, 2048), (70, 3001, 999, 4, 0, 0), (64, 1024, 100, 0, 1024, 512),
    (1201, 1024, 400, 4, 1024, 32), (1470, 1031, 300, 2, 1024, 64), (1185, 1058, 600, 5, 1024, 32), (1480, 1040, 0, 4, 1024, 64),
    (1500, 1055, 400, 4, 1024, 32), (401, 2049, 500, 3, 1024, 32), (400, 2050, 400, 0, 1024, 32), (390, 2049, 350, 6, 1024, 32),
    (401, 2050, 450, 1, 1024, 32), (1181, 1025, 400, 4, 1024, 32),
    (8288, 512, 400, 4, 1024, 128), (8289, 511, 400, 3, 1024, 128)])                                     # the last chunks with a place at once, and one row block more
def test_split_and_join(cass, rows, cols, p, t, seg, chunk):
    w = synth.student_t_weight(rows, cols, 6, f"parts/{rows}x{cols}").float()
    if rows > 20 and cols > 900:
        w[3, 100:900] = 0.0                                  # a long gap
        w[7, ::5] *= 2.0 ** 40                               # rare exponents: long codes
        w[11] = 0.0
    w = w.to(torch.bfloat16)
    wb, act = _bits(w), np.ones(cols, dtype=np.float32)
    fmt = cass.default_format(w_p=p, w_t=t, seg_cols=seg, chunk_cols=chunk)
    bound, ws_bytes = cass.cass_encoded_weight_bytes(fmt, rows, cols)
    blob = torch.zeros(bound, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    wd = w.cuda()
    cass.cass_encode_weights(fmt, wd, None, blob, torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda"), status)
    info = cass.cass_weight_blob_info(blob)
    assert int(status.item()) == 0
    want = layout.encode_verification_data(wb, codec.keep_mask_weights(wb, act, p), p, t)
    vdata = torch.full((cass.cass_verification_data_bytes(info) // 4,), -1, dtype=torch.int32, device="cuda")
    cass.cass_encode_verification_data(blob, info, wd, vdata)
    assert np.array_equal(vdata.cpu().numpy().view(np.uint32), want)
    _join_at_every_phase(cass, blob, info, vdata, wb)


def _join_at_every_phase(cass, blob, info, vdata, wb):
    """The joined matrix against its bits, the output on 16-byte boundaries and off them, and nothing written around it."""
    rows, cols = wb.shape
    full = torch.empty(rows * cols + 16, dtype=torch.bfloat16, device="cuda")
    for shift in (0, 1, 6):
        full.fill_(float("nan"))
        cass.cass_decode_full(blob, info, vdata, full[shift: shift + rows * cols].view(rows, cols))
        assert np.array_equal(_bits(full[shift: shift + rows * cols].view(rows, cols)), wb), shift
        assert torch.isnan(full[:shift]).all() and torch.isnan(full[shift + rows * cols:]).all()


@pytest.mark.parametrize("t", range(8))
@pytest.mark.parametrize("cols", [1000, 1002, 1001])
@pytest.mark.parametrize("rows", [992, 1190])
def test_join_of_every_truncation(cass, rows, cols, t):
    """Teams on 992 chunks and a warp each on 1216, for every truncation and for rows on 16-byte, 4-byte and 2-byte boundaries."""
    w = synth.student_t_weight(rows, cols, 8, f"join/{cols}").float()
    w[7, ::5] *= 2.0 ** 40                                   # long codes
    w[20, 50:700] = 0.0                                      # long runs of pruned values
    w = w.to(torch.bfloat16)
    fmt = cass.default_format(w_p=400, w_t=t, seg_cols=1024, chunk_cols=32)
    bound, ws_bytes = cass.cass_encoded_weight_bytes(fmt, rows, cols)
    blob = torch.zeros(bound, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    wd = w.cuda()
    cass.cass_encode_weights(fmt, wd, None, blob, torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda"), status)
    info = cass.cass_weight_blob_info(blob)
    assert int(status.item()) == 0
    assert info.n_rowblocks * info.n_seg * (info.seg_cols // info.chunk_cols) == (992 if rows == 992 else 1216)      # teams up to 1036
    vdata = torch.zeros(cass.cass_verification_data_bytes(info) // 4, dtype=torch.int32, device="cuda")
    cass.cass_encode_verification_data(blob, info, wd, vdata)
    _join_at_every_phase(cass, blob, info, vdata, _bits(w))


def test_join_of_more_verification_data_than_32_bits_count_words(cass):
    """8.6 G values, 999 of 1000 pruned: the last 64 rows' words lie beyond 2^32."""
    rows, cols, p, t = 524736, 16384, 999, 4
    if torch.cuda.mem_get_info()[0] < 80e9:
        pytest.skip("70 GB of the GPU's memory are not free")
    w = torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda")
    w.view(torch.int16).random_(-2 ** 15, 2 ** 15, generator=torch.Generator(device="cuda").manual_seed(7))
    fmt = cass.default_format(w_p=p, w_t=t)
    bound, ws_bytes = cass.cass_encoded_weight_bytes(fmt, rows, cols)
    blob = torch.empty(bound, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    cass.cass_encode_weights(fmt, w, None, blob, torch.empty(ws_bytes, dtype=torch.uint8, device="cuda"), status)
    info = cass.cass_weight_blob_info(blob)
    assert int(status.item()) == 0
    n_bytes = cass.cass_verification_data_bytes(info)
    assert n_bytes // 4 // rows * (rows - 64) > 2 ** 32
    vdata = torch.empty(n_bytes // 4, dtype=torch.int32, device="cuda")
    cass.cass_encode_verification_data(blob, info, w, vdata)
    out = torch.full_like(w, float("nan"))
    cass.cass_decode_full(blob, info, vdata, out)
    for r in range(0, rows, 65536):
        assert torch.equal(w[r: r + 65536].view(torch.int16), out[r: r + 65536].view(torch.int16)), r
