"""Edges of the two encoders' kernels: row lengths around the register and warp splits of the weight selection, rows with
many equal scores, and spans of tokens against the same tokens appended a few at a time."""
import numpy as np
import pytest
import torch

import synth
from oracle import layout, mx

pytestmark = pytest.mark.gpu


def _bits(t):
    return t.detach().cpu().contiguous().view(torch.int16).numpy().astype(np.uint16)


@pytest.fixture(scope="module")
def cass():
    import paper_2605_26558_b200 as m
    from paper_2605_26558_b200 import engine
    m.engine = engine
    return m


def _blob(cass, w, act, fmt):
    bound, ws_bytes = cass.cass_encoded_weight_bytes(fmt, *w.shape)
    blob = torch.zeros(bound // 4, dtype=torch.int32, device="cuda")
    ws = torch.full((ws_bytes,), 0xA5, dtype=torch.uint8, device="cuda")       # the scratch holds whatever was there
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    cass.cass_encode_weights(fmt, w.cuda(), torch.from_numpy(act).cuda(), blob, ws, status)
    info = cass.cass_weight_blob_info(blob)
    assert int(status.item()) == 0
    return blob[: info.total_bytes // 4].cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("cols", [1, 31, 511, 513, 1024, 1027, 2047, 2056, 4095, 4096, 4104, 8193, 16384, 16391, 32769])
@pytest.mark.parametrize("mode", [1, 2])
def test_rows_around_the_splits(cass, cols, mode):
    rows = 3 if cols > 4096 else 37
    w = synth.student_t_weight(rows, cols, 1, f"edge/w{cols}")
    if cols > 64:
        w[1] = 0.25                                  # every score of the row equal under equal norms
        w[2, : cols // 2] = 0.0                      # half of the row zero: the threshold lies at a tie
        w[0, 5:40] = w[0, 5]
    act = (np.abs(np.random.default_rng(cols).standard_normal(cols)) + 0.05).astype(np.float32)
    act[::2] = 1.0
    fmt = cass.default_format(mode=mode)
    got = _blob(cass, w, act, fmt)
    enc = layout.encode_weight_blob if mode == 1 else mx.encode_weight_blob
    assert np.array_equal(got, enc(_bits(w), act, 400, 4)[0])


@pytest.mark.parametrize("rows,cols", [(4736, 40), (4737, 40), (4800, 520), (4500, 2056), (1200, 9000), (1100, 29000)])
def test_rows_in_turn(cass, rows, cols):
    """More rows than CTAs at once, so that a search starts from another row's threshold: rows like it, rows of another scale,
    rows of one value."""
    g = torch.Generator(device="cuda").manual_seed(cols)
    w = torch.randn(rows, cols, generator=g, device="cuda") + 0.0
    scale = torch.randint(-3, 4, (rows, 1), generator=g, device="cuda") * (torch.rand(rows, 1, generator=g, device="cuda") < 0.3)
    w = (w.abs() + 1e-3) * w.sign() * torch.exp2(scale.float())
    w[::7] = 0.5
    w = torch.where(w == 0, 1e-3, w).to(torch.bfloat16)
    act = torch.rand(cols, generator=g, device="cuda") + 0.05
    fmt = cass.default_format()
    bound, ws_bytes = cass.cass_encoded_weight_bytes(fmt, rows, cols)
    blob = torch.zeros(bound, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    cass.cass_encode_weights(fmt, w, act, blob, torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda"), status)
    dec = torch.empty_like(w)
    cass.cass_decode_weights(blob, cass.cass_weight_blob_info(blob), dec)
    order = torch.sort(w.float().abs() * act, dim=1, stable=True).indices
    keep = torch.ones_like(w, dtype=torch.bool).scatter_(1, order[:, : cols * 400 // 1000], False)
    trunc = (w.view(torch.int16) & -16).view(torch.bfloat16)
    assert int(status.item()) == 0
    assert torch.equal(dec, torch.where(keep, trunc, torch.zeros_like(w)))


@pytest.mark.parametrize("rows,cols,p,seg,chunk", [(9000, 520, 400, 0, 0), (41601, 200, 400, 0, 0), (21000, 470, 300, 0, 0), (2410, 2569, 400, 0, 0),
                                                    (2410, 2570, 600, 0, 0), (1600, 5300, 0, 0, 0), (3000, 2056, 400, 1024, 32), (1600, 4100, 990, 0, 0),
                                                    (4801, 512, 400, 0, 0), (4737, 641, 600, 0, 0), (4801, 1300, 400, 0, 0),
                                                    (83201, 64, 400, 0, 0), (30000, 301, 999, 0, 0), (12000, 513, 400, 0, 0), (16640, 632, 400, 256, 256),
                                                    (4737, 256, 400, 0, 0), (4737, 501, 400, 0, 0), (4736, 1025, 300, 0, 0), (4737, 1025, 300, 0, 0), (4736, 1026, 300, 0, 0),
                                                    (6000, 512, 299, 0, 0), (9473, 65, 300, 0, 0), (40, 3000, 300, 0, 0), (9, 1032, 400, 1024, 1024)])
def test_blobs_by_lanes(cass, rows, cols, p, seg, chunk):
    """Sizes and packing by lanes: 2 to 16 warps a superblock, rows on 16-, 4- and 2-byte boundaries, chunks of few values, a last row
    block that is not full; rows of one value, of none, and with codes longer than a word; fewer blocks of 128 columns than warps,
    blocks that do not share out evenly, a last segment of one.  By warps: of one and two superblocks an SM (4736 rows and more), short
    segments, odd columns and rows that keep more than 70 %."""
    w = synth.student_t_weight(rows, cols, 2, f"lanes/{rows}x{cols}").float()
    w[1] = 0.25
    w[2] = 0.0
    w[3, ::7] *= torch.exp2(torch.arange(len(w[3, ::7]), dtype=torch.float32) % 120 - 60)
    w[5, : cols // 2] = 0.0
    w[-1] *= 2.0 ** 20
    w = w.to(torch.bfloat16)
    act = (np.abs(np.random.default_rng(cols).standard_normal(cols)) + 0.05).astype(np.float32)
    got = _blob(cass, w, act, cass.default_format(w_p=p, seg_cols=seg, chunk_cols=chunk))
    assert np.array_equal(got, layout.encode_weight_blob(_bits(w), act, p, 4, *((seg, chunk) if seg else ()))[0])


@pytest.mark.parametrize("rows,cols", [(9473, 1), (9473, 2), (9473, 8), (9473, 33)])
def test_blobs_of_next_to_no_columns_by_lanes(cass, rows, cols):
    w = synth.student_t_weight(rows, cols, 4, f"narrow/{cols}")
    w[1] = 0.0
    act = (np.abs(np.random.default_rng(cols).standard_normal(cols)) + 0.05).astype(np.float32)
    assert np.array_equal(_blob(cass, w, act, cass.default_format()), layout.encode_weight_blob(_bits(w), act, 400, 4)[0])


@pytest.mark.parametrize("rows,cols", [(70, 2056), (4801, 512)])
@pytest.mark.parametrize("shift", [1, 2, 4])
def test_matrix_off_16_byte_boundaries_by_lanes(cass, rows, cols, shift):
    w = synth.student_t_weight(rows, cols, 5, f"shift/{cols}").cuda()
    act = (np.abs(np.random.default_rng(shift).standard_normal(cols)) + 0.05).astype(np.float32)
    off = torch.empty(rows * cols + 8, dtype=torch.bfloat16, device="cuda")[shift: shift + rows * cols].view(rows, cols)
    off.copy_(w)
    fmt = cass.default_format()
    assert np.array_equal(_blob(cass, off, act, fmt), _blob(cass, w, act, fmt))


def test_constant_rows_and_no_pruning(cass):
    w = torch.full((40, 3000), 0.5, dtype=torch.bfloat16)
    w[7] = 0.0
    act = np.ones(3000, dtype=np.float32)
    for p, t in ((400, 4), (0, 0), (999, 3)):
        got = _blob(cass, w, act, cass.default_format(w_p=p, w_t=t))
        assert np.array_equal(got, layout.encode_weight_blob(_bits(w), act, p, t)[0]), (p, t)


@pytest.mark.parametrize("rows,cols", [(8, 40), (37, 700), (37, 2048), (9, 2056), (8, 14336)])
def test_scores_that_are_no_numbers_rank_highest(cass, rows, cols):
    """NaN and infinite weights and norms: every row keeps its count, and the matrix comes back from its two parts."""
    p = 400
    rng = np.random.default_rng(cols)
    w = _bits(synth.student_t_weight(rows, cols, 9, f"nan/{cols}"))
    w[1, ::3] = 0x7FC1                                   # a third NaN
    w[2, ::2], w[2, 1] = 0xFFC0, 0x7F80                  # half of the row -NaN, an infinity
    w[3] = 0x7FFF
    w[4, : cols - 5] = 0x7F80                            # more infinities than are kept
    w[5, 3] = 0xFF80
    w[6, cols // 3:] = 0x7F81                            # two thirds: among equals the lower columns go
    act = (np.abs(rng.standard_normal(cols)) + 0.05).astype(np.float32)
    act[7::11], act[8::13] = 0.0, np.inf                 # inf x 0 either way round
    w[7, ::2] = 0
    with np.errstate(invalid="ignore", over="ignore"):
        score = (((w & 0x7FFF).astype(np.uint32) << 16).view(np.float32) * act).astype(np.float32)
    key = np.where(np.isnan(score), np.uint32(0x7FFFFFFF), score.view(np.uint32))
    keep = np.ones((rows, cols), dtype=bool)
    np.put_along_axis(keep, np.argsort(key, axis=1, kind="stable")[:, : cols * p // 1000], False, axis=1)
    wd = torch.from_numpy(w.view(np.int16)).cuda().view(torch.bfloat16)
    fmt = cass.default_format(w_p=p)
    bound, ws_bytes = cass.cass_encoded_weight_bytes(fmt, rows, cols)
    blob = torch.zeros(bound, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    cass.cass_encode_weights(fmt, wd, torch.from_numpy(act).cuda(), blob, torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda"), status)
    info = cass.cass_weight_blob_info(blob)
    assert int(status.item()) == 0
    dec = torch.empty_like(wd)
    cass.cass_decode_weights(blob, info, dec)
    assert np.array_equal(_bits(dec), np.where(keep, w & 0xFFF0, 0))
    vdata = torch.zeros(cass.cass_verification_data_bytes(info), dtype=torch.uint8, device="cuda")
    cass.cass_encode_verification_data(blob, info, wd, vdata)
    full = torch.empty_like(wd)
    cass.cass_decode_full(blob, info, vdata, full)
    assert np.array_equal(_bits(full), w)


def _records(cass, eng, layer, seq):
    base, mem, out = eng.mem.data_ptr(), eng.mem.view(torch.int32), []
    for kind in (0, 1):
        v = cass.cass_kv_query(eng.session, layer, kind, 0, seq=seq)
        h, n = eng.shape.n_kv_heads, eng.desc.max_seq
        for ptr, words in ((v.fixed, h * ((n + 31) // 32) * v.fixed_words_per_token * 32), (v.arena, h * v.arena_words),
                           (v.offsets, h * (n + 1)), (v.codebook, 64)):
            o = (ptr - base) // 4
            out.append(mem[o: o + words].clone())
    return out


@pytest.mark.parametrize("d,kv_p,kv_t,kv_mode", [(32, 400, 4, 1), (64, 400, 4, 1), (128, 400, 4, 1), (128, 0, 0, 1), (256, 300, 4, 1),
                                                 (96, 400, 0, 2), (128, 400, 4, 2), (256, 0, 0, 2)])
@pytest.mark.parametrize("n_new", [17, 40, 301])
def test_span_of_tokens_equals_tokens_in_turn(cass, d, kv_p, kv_t, kv_mode, n_new):
    """Two layers, two sequences: the codebook's prompt and a later span give the records, offsets and codebooks that
    appending up to 16 tokens a call gives, rows with ties, zeros and exponents that the codebook knows badly included."""
    shape = synth.ModelShape(n_layers=2, hidden=256, n_q_heads=4, n_kv_heads=2, head_dim=d, ffn=256, vocab=256)
    wt = synth.model_weights(shape, 0, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    fmt = cass.default_format(kv_p=kv_p, kv_t=kv_t, kv_mode=kv_mode)
    n0 = 21
    engs = [cass.engine.Engine(shape, gw, fmt=fmt, max_seq=384, gamma_max=4, batch=2) for _ in range(2)]
    for layer in range(2):
        for seq in range(2):
            k, v = (x.cuda() for x in synth.kv_fill(n0 + n_new, 2, d, 10 * layer + seq, "edge/kv"))
            k[3], v[n0 + 1] = 0.0, 1.5
            k[n0 + 2] *= torch.exp2(torch.arange(d, device="cuda") % 37).to(torch.bfloat16)
            k[n0 + 4, :, ::3] = 0.75
            for e in engs:
                cass.cass_kv_append(e.session, layer, k[:n0].contiguous(), v[:n0].contiguous(), 0, n0, cass.KV_BF16, seq=seq)
    for e in engs:
        e.n_prompt = n0
        e.build_kv_codebook()
        for layer in range(2):
            for seq in range(2):
                k, v = (x.cuda() for x in synth.kv_fill(n0 + n_new, 2, d, 10 * layer + seq, "edge/kv"))
                v[n0 + 1] = 1.5
                k[n0 + 2] *= torch.exp2(torch.arange(d, device="cuda") % 37).to(torch.bfloat16)
                k[n0 + 4, :, ::3] = 0.75
                step = n_new if e is engs[0] else 16
                for i in range(0, n_new, step):
                    m = min(step, n_new - i)
                    cass.cass_kv_append(e.session, layer, k[n0 + i: n0 + i + m].contiguous(), v[n0 + i: n0 + i + m].contiguous(),
                                        n0 + i, m, cass.KV_BF16 | cass.KV_COMPRESSED, seq=seq)
    torch.cuda.synchronize()
    for layer in range(2):
        for seq in range(2):
            for i, (a, b) in enumerate(zip(_records(cass, engs[0], layer, seq), _records(cass, engs[1], layer, seq))):
                assert torch.equal(a, b), (layer, seq, i)
    for e in engs:
        assert e.status()[0] == 0
        e.close()


def test_append_right_behind_a_codebook_of_no_tokens(cass):
    """The last kernel of such a codebook writes the tables that the append reads."""
    d, n0 = 128, 24
    shape = synth.ModelShape(n_layers=1, hidden=256, n_q_heads=4, n_kv_heads=2, head_dim=d, ffn=256, vocab=256)
    wt = synth.model_weights(shape, 0, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    k, v = (x.cuda() for x in synth.kv_fill(n0 + 4, 2, d, 3, "edge/kv"))
    engs = [cass.engine.Engine(shape, gw, max_seq=384, gamma_max=4) for _ in range(2)]
    for e in engs:
        cass.cass_kv_append(e.session, 0, k[:n0].contiguous(), v[:n0].contiguous(), 0, n0, cass.KV_BF16)
    a, b = k[n0:].contiguous(), v[n0:].contiguous()
    for tokens in [n0, 0] * 20:                          # another codebook each time
        for e in engs:
            cass.cass_kv_build_codebook(e.session, tokens)
            if e is engs[1]:
                torch.cuda.synchronize()
            cass.cass_kv_append(e.session, 0, a, b, n0, 4, cass.KV_COMPRESSED)
        torch.cuda.synchronize()
        for i, (x, y) in enumerate(zip(_records(cass, engs[0], 0, 0), _records(cass, engs[1], 0, 0))):
            assert torch.equal(x, y), (tokens, i)
    for e in engs:
        assert e.status()[0] == 0
        e.close()
