"""Compressed KV records of many positions at once (a lane a record) against those of few (a warp a record): the same bytes."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cass():
    import paper_2605_26558_b200 as m
    from paper_2605_26558_b200 import engine
    m.engine = engine
    return m


def _engine(cass, d, layers, batch, max_seq, **fmt):
    shape = synth.ModelShape(n_layers=layers, hidden=64, n_q_heads=8, n_kv_heads=8, head_dim=d, ffn=64, vocab=64)
    wt = synth.model_weights(shape, 1, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    return cass.engine.Engine(shape, gw, fmt=cass.default_format(**fmt), max_seq=max_seq, gamma_max=2, batch=batch)


def _rows(n, d, seed):
    """Ordinary rows, and one each of what a search can trip over: equal magnitudes, zeros, exponents far apart, infinities and
    NaNs, values below the normal numbers, a few distinct values only."""
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(n, 8, d, generator=g)
    x[:, :, : max(1, d // 50)] *= 10.0
    x[1 % n] = 1.5
    x[2 % n] = 0.0
    x[3 % n] *= torch.exp2(torch.randint(-100, 100, (8, d), generator=g).float())
    x[5 % n, :, ::3] = float("inf")
    x[6 % n, :, ::2] = float("nan")
    x[7 % n] *= 1e-39
    x[8 % n] = torch.randint(-2, 3, (8, d), generator=g).float()
    return x.to(torch.bfloat16).cuda()


def _records(cass, eng, layer, seq, n):
    """Everything a reader of positions 0 .. n - 1 sees: whole blocks of the fixed part, arena words in use, offsets, codebook."""
    out, base, m = [], eng.mem.data_ptr(), eng.desc.max_seq
    words = eng.mem.view(torch.int32)
    for kind in (0, 1):
        for head in range(8):
            v = cass.cass_kv_query(eng.session, layer, kind, head, seq=seq)
            o, f, a = ((p - base) // 4 for p in (v.offsets, v.fixed, v.arena))
            off = words[o: o + n + 1]
            out += [off, words[f: f + (n + 31) // 32 * 32 * v.fixed_words_per_token], words[a: a + int(off[-1])]]
        out.append(eng.mem[v.codebook - base: v.codebook - base + 256])
    assert m >= n
    return [t.clone() for t in out]


@pytest.mark.parametrize("d", [32, 64, 96, 128, 224, 256])
@pytest.mark.parametrize("mode,t,p", [(1, 4, 400), (1, 0, 300), (1, 4, 0), (2, 4, 400), (2, 0, 500)])
def test_prompt_records(cass, d, mode, t, p):
    """2 layers x 4 sequences x 16 streams x 5 blocks (the last one not full) at once, against a sequence of a layer by itself."""
    n = 150
    fmt = dict(kv_mode=mode, kv_t=t, kv_p=p)
    many = _engine(cass, d, 2, 4, 192, **fmt)
    kv = {(l, b, k): _rows(n, d, 100 * l + 10 * b + k) for l in range(2) for b in range(4) for k in range(2)}
    for l in range(2):
        for b in range(4):
            cass.cass_kv_append(many.session, l, kv[l, b, 0], kv[l, b, 1], 0, n, cass.KV_BF16, seq=b)
    cass.cass_kv_build_codebook(many.session, n)
    for l, b in ((0, 0), (1, 3)):
        one = _engine(cass, d, 1, 1, 192, **fmt)
        cass.cass_kv_append(one.session, 0, kv[l, b, 0], kv[l, b, 1], 0, n, cass.KV_BF16)
        cass.cass_kv_build_codebook(one.session, n)
        for i, (x, y) in enumerate(zip(_records(cass, many, l, b, n), _records(cass, one, 0, 0, n))):
            assert torch.equal(x, y), (l, b, i)
        one.close()
    assert many.status()[0] == 0
    many.close()


@pytest.mark.parametrize("d", [64, 128, 256])
@pytest.mark.parametrize("mode,t", [(1, 4), (1, 0), (2, 4)])
@pytest.mark.parametrize("start,n,aligned", [(41, 1250, True), (64, 1216, True), (41, 1250, False)])
def test_appended_records(cass, d, mode, t, start, n, aligned):
    """One append of 39 or 40 blocks of 16 streams (from a block's middle; rows on 2-byte boundaries take the other path) against
    appends of up to 100 positions, behind the same codebook of few positions."""
    fmt = dict(kv_mode=mode, kv_t=t, kv_p=400)
    k, v = _rows(start + n, d, 7), _rows(start + n, d, 8)
    engines = [_engine(cass, d, 1, 1, 1408, **fmt) for _ in range(2)]
    for e in engines:
        cass.cass_kv_append(e.session, 0, k[:start].contiguous(), v[:start].contiguous(), 0, start, cass.KV_BF16)
        cass.cass_kv_build_codebook(e.session, start)
    both = cass.KV_BF16 | cass.KV_COMPRESSED

    def part(x, lo, hi):
        x = x[lo:hi].contiguous()
        return x if aligned else torch.cat([x.new_zeros(1), x.flatten()])[1:].view(x.shape)
    a, b = engines
    cass.cass_kv_append(a.session, 0, part(k, start, start + n), part(v, start, start + n), start, n, both)
    for lo in range(start, start + n, 100):
        hi = min(lo + 100, start + n)
        cass.cass_kv_append(b.session, 0, k[lo:hi].contiguous(), v[lo:hi].contiguous(), lo, hi - lo, both)
    for i, (x, y) in enumerate(zip(_records(cass, a, 0, 0, start + n), _records(cass, b, 0, 0, start + n))):
        assert torch.equal(x, y), i
    for kind, src in ((0, k), (1, v)):
        o = (cass.cass_kv_query(a.session, 0, kind, 0).k_or_v_bf16 - a.mem.data_ptr()) // 2
        got = a.mem.view(torch.int16)[o: o + (start + n) * 8 * d].view(-1, 8, d)
        assert torch.equal(got, src.view(torch.int16)), kind
    assert a.status()[0] == b.status()[0] == 0
    for e in engines:
        e.close()
