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
