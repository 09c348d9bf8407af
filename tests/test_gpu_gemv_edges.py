"""Edges of the draft GEMV's walk and of where its results are added: segments alone, in a cluster and in a kernel of their
own, pruning on both sides of the second column window, rows whose gaps and codes leave every window."""
import numpy as np
import pytest
import torch

import synth
from oracle import codec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cass():
    import paper_2605_26558_b200 as m
    return m


def _bits(t):
    return t.detach().cpu().contiguous().view(torch.int16).numpy().astype(np.uint16)


@pytest.mark.parametrize("mode,t", [(1, 4), (1, 0), (1, 3), (2, 4)])
@pytest.mark.parametrize("rows,cols,p,seg", [
    (1, 1, 0, 0), (33, 31, 520, 0), (40, 2048, 530, 0), (65, 2049, 400, 0), (70, 700, 700, 256), (37, 2304, 600, 256),
    (64, 2300, 900, 256), (31, 16400, 400, 0), (2000, 513, 800, 256), (9000, 2100, 400, 0)])
def test_walk_and_results(cass, mode, t, rows, cols, p, seg):
    w = synth.student_t_weight(rows, cols, 8, f"gemv/{rows}x{cols}").float()
    if rows > 30 and cols > 600:
        w[2, 50:500] = 0.0                                   # a gap longer than two windows
        w[5, ::7] *= 2.0 ** 30                               # rare exponents: long codes
        w[6, 40:] = 0.0
    w = w.to(torch.bfloat16).cuda()
    fmt = cass.default_format(w_p=p, w_t=t, seg_cols=seg, mode=mode)
    bound, ws_bytes = cass.cass_encoded_weight_bytes(fmt, rows, cols)
    blob = torch.zeros(bound, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    cass.cass_encode_weights(fmt, w, None, blob, torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda"), status)
    info = cass.cass_weight_blob_info(blob)
    dec = torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda")
    cass.cass_decode_weights(blob, info, dec)
    d = codec.bf16_bits_to_f64(_bits(dec))
    x = synth.activation_vector(cols, 4, "gemv/x", rows=8).cuda().contiguous()
    xd = codec.bf16_bits_to_f64(_bits(x))
    ref, scale = xd @ d.T, np.abs(xd) @ np.abs(d).T
    n_pad = info.n_rowblocks * 32
    first = None
    for nb in (1, 2, 4, 8):
        partial = torch.full((nb * info.n_seg * n_pad,), float("nan"), device="cuda")
        y32 = torch.full((nb, rows), float("nan"), device="cuda")
        y16 = torch.zeros(nb, rows, dtype=torch.bfloat16, device="cuda")
        if nb == 1:
            cass.cass_draft_gemv(blob, info, x[0], partial, y16, y32, status)
            first = y32[0].clone()
        else:
            cass.cass_draft_gemv_batch(blob, info, x[:nb].contiguous(), nb, partial, y16, y32, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got = y32.cpu().numpy().astype(np.float64)
        assert (np.abs(got - ref[:nb]) <= 1e-5 * scale[:nb] + 1e-30).all(), nb
        assert torch.equal(y32[0], first)                    # a vector's result does not depend on the others
        assert np.array_equal(_bits(y16), codec.f64_to_bf16_bits(got))
        # the segments' sums are there too, and add up to the result in their order
        s = partial.view(nb, info.n_seg, n_pad)[:, :, :rows]
        acc = torch.zeros(nb, rows, device="cuda")
        for i in range(info.n_seg):
            acc += s[:, i]
        assert torch.equal(acc, y32)
