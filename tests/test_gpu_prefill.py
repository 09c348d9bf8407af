"""The wide prefill passes against the same prompt fed to cass_verify 16 rows (or fewer) a call: caches, activations left
behind, first tokens and calibration statistics."""
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


def _chunked(cass, eng, prompt):
    """First tokens by cass_verify, as many rows a call as it takes."""
    prompt = prompt.cuda().reshape(eng.batch, -1)
    n, chunk = prompt.shape[1], min(16, eng.max_rows // eng.batch)
    for pos in range(0, n, chunk):
        rows = min(chunk, n - pos)
        cass.cass_set_len(eng.session, pos)
        cass.cass_verify(eng.session, prompt[:, pos: pos + rows].contiguous(), rows - 1, eng.targ)
    cass.cass_set_len(eng.session, n)
    return eng.targ[: eng.batch * rows].view(eng.batch, rows)[:, -1].tolist(), rows


def _cache(cass, eng, n):
    out, row, base = [], eng.shape.n_kv_heads * eng.shape.head_dim, eng.mem.data_ptr()
    for layer in range(eng.shape.n_layers):
        for b in range(eng.batch):
            for kind in (0, 1):
                o = (cass.cass_kv_query(eng.session, layer, kind, 0, seq=b).k_or_v_bf16 - base) // 2
                out.append(eng.mem.view(torch.bfloat16)[o: o + n * row])
    return out


def _activation(cass, eng, which, rows):
    p, _, cols = cass.cass_debug_activation(eng.session, which)
    o = (p - eng.mem.data_ptr()) // 2
    return eng.mem.view(torch.bfloat16)[o: o + rows * cols]


@pytest.mark.parametrize("heads,kv,d", [(4, 2, 64), (8, 2, 128), (10, 2, 32), (5, 1, 128)])
@pytest.mark.parametrize("batch,n", [(1, 1), (1, 16), (1, 17), (1, 129), (1, 300), (2, 75), (8, 5), (8, 40)])
def test_wide_passes_equal_verification_calls(cass, heads, kv, d, batch, n):
    shape = synth.ModelShape(n_layers=2, hidden=256, n_q_heads=heads, n_kv_heads=kv, head_dim=d, ffn=344, vocab=512)
    wt = synth.model_weights(shape, 1, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = torch.stack([synth.random_prompt(n, shape.vocab, 40 + b) for b in range(batch)])
    a, b = (cass.engine.Engine(shape, gw, max_seq=384, gamma_max=4, batch=batch) for _ in range(2))
    first = a.prefill(prompt, calibrate=True)
    cass.cass_calib_enable(b.session, True)
    want, rows = _chunked(cass, b, prompt)
    cass.cass_calib_enable(b.session, False)
    assert ([first] if batch == 1 else first) == want
    assert a.lens() == b.lens() == [n] * batch and a.status()[0] == b.status()[0] == 0
    # five query heads a KV head: verification takes 16 rows to the fp32 pipes, the wide pass stays on the tensor cores
    exact = not (heads == 5)
    pairs = list(zip(_cache(cass, a, n), _cache(cass, b, n)))
    pairs += [(_activation(cass, a, w, batch * rows), _activation(cass, b, w, batch * rows)) for w in (0, 1, 2)]
    for i, (x, y) in enumerate(pairs):
        if exact:
            assert torch.equal(x, y), i
        else:
            err = (x.float() - y.float()).norm() / y.float().norm()
            assert err <= 5e-3, (i, float(err))
    na, nb = a.calib_norms(), b.calib_norms()
    for la, lb in zip(na["layers"], nb["layers"]):
        for k in la:
            assert float((la[k] - lb[k]).norm() / lb[k].norm()) <= (1e-5 if exact else 5e-3), k
    # the same prompt again, now that the codebooks are there: compressed records too
    a.build_kv_codebook()
    before = [t.clone() for t in _cache(cass, a, n)]
    assert a.prefill(prompt) == first
    assert all(torch.equal(x, y) for x, y in zip(before, _cache(cass, a, n)))
    a.close()
    b.close()


@pytest.mark.parametrize("heads,kv,d", [(4, 2, 64), (8, 2, 128)])
def test_long_prompts_equal_verification_calls(cass, heads, kv, d):
    """Beyond eight chunks of positions the wide passes' partial results are merged by other kernels than those of verification
    calls (64 positions a chunk at head size 64: up to 8, 16, 32 and more; 128 at head size 128: up to 8, 16 and 32), and the
    scratch takes several launches a layer."""
    n, max_seq = 2300, 2432
    shape = synth.ModelShape(n_layers=1, hidden=256, n_q_heads=heads, n_kv_heads=kv, head_dim=d, ffn=256, vocab=512)
    wt = synth.model_weights(shape, 2, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = synth.random_prompt(n, shape.vocab, 41)
    a, b = (cass.engine.Engine(shape, gw, max_seq=max_seq, gamma_max=4) for _ in range(2))
    # with one layer attention does not reach the caches: its rows are compared at the ends of prompts of several lengths
    for m in (600, 1100, 2100, n):
        first = a.prefill(prompt[:m])
        want, rows = _chunked(cass, b, prompt[:m])
        assert [first] == want, m
        for w in (0, 1, 2):
            assert torch.equal(_activation(cass, a, w, rows), _activation(cass, b, w, rows)), (m, w)
    assert all(torch.equal(x, y) for x, y in zip(_cache(cass, a, n), _cache(cass, b, n)))
    assert a.status()[0] == b.status()[0] == 0
    a.close()
    b.close()


@pytest.mark.parametrize("batch,n", [(1, 33), (1, 127), (1, 128), (1, 192), (1, 193), (1, 257), (1, 385), (1, 1024), (1, 1030), (2, 520), (4, 259)])
def test_wide_projections_equal_verification_calls(cass, batch, n):
    """Edges of the wide projection's tiles (128, 192 and 256 rows, 256 features), several K ranges a tile with a block left over,
    K and features off the tiles' multiples, one pass more than its rows hold."""
    shape = synth.ModelShape(n_layers=1, hidden=1288, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=1032, vocab=512)
    wt = synth.model_weights(shape, 4, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = torch.stack([synth.random_prompt(n, shape.vocab, 50 + b) for b in range(batch)])
    a, b = (cass.engine.Engine(shape, gw, max_seq=1056, gamma_max=4, batch=batch) for _ in range(2))
    first = a.prefill(prompt)
    want, rows = _chunked(cass, b, prompt)
    assert ([first] if batch == 1 else first) == want
    assert a.status()[0] == b.status()[0] == 0
    assert all(torch.equal(x, y) for x, y in zip(_cache(cass, a, n), _cache(cass, b, n)))
    for w in (0, 1, 2):
        assert torch.equal(_activation(cass, a, w, batch * rows), _activation(cass, b, w, batch * rows)), w
    a.close()
    b.close()


@pytest.mark.parametrize("n", [33, 64, 65, 128, 129, 192, 193, 256])
def test_wide_projection_of_few_rows_between_split_ones(cass, n):
    """A projection of so many features that few rows pay in the wide form (tiles of 128 and 192 rows, K and features off the tiles'
    multiples) among others that are split: bf16 results and parts in one layer."""
    shape = synth.ModelShape(n_layers=1, hidden=1288, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=10328, vocab=512)
    wt = synth.model_weights(shape, 8, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = synth.random_prompt(n, shape.vocab, 80)
    a, b = (cass.engine.Engine(shape, gw, max_seq=288, gamma_max=4) for _ in range(2))
    first = a.prefill(prompt)
    want, rows = _chunked(cass, b, prompt)
    assert [first] == want and a.status()[0] == b.status()[0] == 0
    assert all(torch.equal(x, y) for x, y in zip(_cache(cass, a, n), _cache(cass, b, n)))
    for w in (0, 1, 2):
        assert torch.equal(_activation(cass, a, w, rows), _activation(cass, b, w, rows)), w
    a.close()
    b.close()


@pytest.mark.parametrize("heads,kv,batch,n", [(2, 2, 1, 127), (2, 2, 1, 257), (2, 1, 1, 1025), (3, 1, 2, 129), (3, 1, 1, 1190), (4, 1, 4, 300), (8, 1, 1, 300), (7, 1, 1, 1100)])
def test_prefill_attention_of_every_group(cass, heads, kv, batch, n):
    """Head size 128: groups that leave lanes of a CTA without a pair, ends of chunks and of CTAs, more than eight chunks (chains of
    the merge's order).  With more than four query heads a KV head verification takes 16 rows to the fp32 pipes; both round the
    output to bf16 (2^-9 of it each), and a flipped bit of an activation travels on: 5e-3, as above."""
    shape = synth.ModelShape(n_layers=1, hidden=256, n_q_heads=heads, n_kv_heads=kv, head_dim=128, ffn=256, vocab=512)
    wt = synth.model_weights(shape, 5, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = torch.stack([synth.random_prompt(n, shape.vocab, 60 + b) for b in range(batch)])
    a, b = (cass.engine.Engine(shape, gw, max_seq=1216, gamma_max=4, batch=batch) for _ in range(2))
    a.prefill(prompt)
    _, rows = _chunked(cass, b, prompt)
    assert a.status()[0] == b.status()[0] == 0
    x, y = (_activation(cass, e, 1, batch * rows) for e in (a, b))
    if heads // kv <= 4:
        assert torch.equal(x, y)
    else:
        assert (x.float() - y.float()).norm() / y.float().norm() <= 5e-3
    a.close()
    b.close()


@pytest.mark.parametrize("n,max_seq", [(4097, 4224), (4240, 8448), (8300, 8448), (300, 32896)])
def test_prefill_attention_of_many_chunks(cass, n, max_seq):
    """Head size 128: more than 32 and 64 chunks of 128 positions, whose sums are added 32 at a time, and a cache of 257, which the
    one-CTA attention does not take."""
    shape = synth.ModelShape(n_layers=1, hidden=256, n_q_heads=2, n_kv_heads=1, head_dim=128, ffn=256, vocab=512)
    wt = synth.model_weights(shape, 9, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = synth.random_prompt(n, shape.vocab, 90)
    a, b = (cass.engine.Engine(shape, gw, max_seq=max_seq, gamma_max=4) for _ in range(2))
    first = a.prefill(prompt)
    want, rows = _chunked(cass, b, prompt)
    assert [first] == want and a.status()[0] == b.status()[0] == 0
    for w in (0, 1, 2):
        assert torch.equal(_activation(cass, a, w, rows), _activation(cass, b, w, rows)), w
    a.close()
    b.close()


@pytest.mark.parametrize("hidden", [4232, 5120, 8192])
@pytest.mark.parametrize("n", [296, 300])
def test_norms_of_wide_rows(cass, hidden, n):
    """Rows of more than 4096 values take two turns of the norm's threads; from 297 rows on a quarter as many."""
    shape = synth.ModelShape(n_layers=1, hidden=hidden, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=264, vocab=512)
    wt = synth.model_weights(shape, 10, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = synth.random_prompt(n, shape.vocab, 91)
    a, b = (cass.engine.Engine(shape, gw, max_seq=384, gamma_max=4) for _ in range(2))
    first = a.prefill(prompt)
    want, rows = _chunked(cass, b, prompt)
    assert [first] == want and a.status()[0] == b.status()[0] == 0
    for w in (0, 1, 2):
        assert torch.equal(_activation(cass, a, w, rows), _activation(cass, b, w, rows)), w
    a.close()
    b.close()


@pytest.mark.parametrize("heads,kv", [(8, 2), (2, 2)])
@pytest.mark.parametrize("first,last", [(256, 300), (0, 128), (290, 300)])
def test_scores_that_are_no_numbers(cass, heads, kv, first, last):
    """K of some tokens overflows to infinities of both signs, and all scores there are NaN.  Both paths pass over a chunk that such
    tokens begin and the causal limit ends, and lose a row to one that they fill."""
    n, d, hidden = 300, 128, 256
    shape = synth.ModelShape(n_layers=1, hidden=hidden, n_q_heads=heads, n_kv_heads=kv, head_dim=d, ffn=256, vocab=512)
    wt = synth.model_weights(shape, 6, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"].clone(), "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    layer, wide = gw["layers"][0], 7                                       # input channel `wide`: 1e36 of it, for K alone
    gw["embed"][:, wide] = 0.0
    gw["embed"][0, wide] = gw["embed"][0].abs().max()
    layer["norm_attn"] = layer["norm_attn"].clone()
    layer["norm_attn"][wide] = 1e36
    layer["wqkv"] = layer["wqkv"].clone()
    layer["wqkv"][:, wide] = 0.0
    layer["wqkv"][heads * d: (heads + kv) * d, wide] = 1e4 * (1 - 2 * (torch.arange(kv * d, device="cuda") % 2)).to(torch.bfloat16)
    prompt = synth.random_prompt(n, shape.vocab - 1, 70) + 1
    prompt[first: last] = 0
    a, b = (cass.engine.Engine(shape, gw, max_seq=384, gamma_max=4) for _ in range(2))
    a.prefill(prompt)
    _, rows = _chunked(cass, b, prompt)
    assert a.status()[0] == b.status()[0] == 0
    k, v = _cache(cass, a, n)
    k = k.view(n, -1)
    assert not torch.isfinite(k[first: last]).any() and torch.isfinite(k[:first]).all() and torch.isfinite(k[last:]).all() and torch.isfinite(v).all()
    x, y = (_activation(cass, e, 1, rows) for e in (a, b))
    assert torch.isfinite(y).all() == (first == 256) and torch.equal(x.view(torch.int16), y.view(torch.int16))
    a.close()
    b.close()


def test_two_bf16_terms_are_as_accurate_as_the_fp32_pipes(cass):
    """Five query heads a KV head at head size 128: verification takes 16 rows to the fp32 pipes, the wide pass to the tensor
    cores with P in two bf16 terms.  On the same queries and caches both differ from 64 bits by the rounding of the output alone
    (two terms leave 2^-17 of a weight, 2^-8 of that rounding).  P in one term, restated here, comes out 1.11 times as far off."""
    n, heads, d = 304, 5, 128
    shape = synth.ModelShape(n_layers=1, hidden=256, n_q_heads=heads, n_kv_heads=1, head_dim=d, ffn=256, vocab=512)
    wt = synth.model_weights(shape, 3, device="cuda")
    gw = {"layers": [cass.engine.fuse_layer_weights(lw) for lw in wt["layers"]], "embed": wt["embed"], "lm_head": wt["lm_head"],
          "norm_final": wt["norm_final"]}
    prompt = synth.random_prompt(n, shape.vocab, 42)
    a, b = (cass.engine.Engine(shape, gw, max_seq=384, gamma_max=4) for _ in range(2))
    a.prefill(prompt)
    _, rows = _chunked(cass, b, prompt)
    assert rows == 16
    k, v = (t.view(n, d).double() for t in _cache(cass, a, n))
    assert all(torch.equal(x, y) for x, y in zip(_cache(cass, a, n), _cache(cass, b, n)))
    q = _activation(cass, a, 2, rows)
    assert torch.equal(q, _activation(cass, b, 2, rows))
    q = q.view(rows, -1)[:, : heads * d].view(rows, heads, d).double()
    s = torch.einsum("rhd,td->rht", q, k) / d ** 0.5
    seen = torch.arange(n, device="cuda")[None, None, :] <= (n - rows + torch.arange(rows, device="cuda"))[:, None, None]
    want = torch.einsum("rht,td->rhd", torch.softmax(s.masked_fill(~seen, -float("inf")), dim=-1), v)
    p = torch.exp(s.masked_fill(~seen, -float("inf")) - s.masked_fill(~seen, -float("inf")).amax(-1, keepdim=True)).to(torch.bfloat16).double()
    one = (torch.einsum("rht,td->rhd", p, v) / p.sum(-1, keepdim=True)).to(torch.bfloat16).double()
    wide, pipes = ((_activation(cass, e, 1, rows).view(rows, heads, d).double() - want).norm() / want.norm() for e in (a, b))
    assert (one - want).norm() / want.norm() > 1.05 * pipes                # what the bound below tells apart
    assert wide <= 1.02 * pipes and pipes <= 2.0 ** -9
    a.close()
    b.close()
