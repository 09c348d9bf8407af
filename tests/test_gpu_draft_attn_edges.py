"""Draft attention where a warp's 32 records do not all fit its staging: long codes, raw exponents, a ragged last block."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cass():
    import paper_2605_26558_b200 as m
    return m


@pytest.mark.parametrize("n,every", [(1, 1), (31, 2), (33, 1), (64, 3), (97, 1)])
def test_draft_attention_records_of_any_length(cass, n, every):
    from paper_2605_26558_b200 import engine
    sh = synth.ModelShape(n_layers=1, hidden=256, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=256, vocab=64)
    wt = synth.model_weights(sh, 0)
    gw = {"layers": [engine.fuse_layer_weights({k: v.cuda() for k, v in lw.items()}) for lw in wt["layers"]],
          "embed": wt["embed"].cuda(), "lm_head": wt["lm_head"].cuda(), "norm_final": wt["norm_final"].cuda()}
    eng = engine.Engine(sh, gw, fmt=cass.default_format(kv_p=0, kv_t=0), max_seq=160, gamma_max=4)
    g = torch.Generator().manual_seed(n)
    k, v = (torch.randn(n, 2, 64, generator=g) for _ in range(2))
    # every `every`-th token spreads its values over many exponents: codes of a dozen bits, or raw exponents
    spread = 2.0 ** torch.randint(-9, 10, (n, 2, 64), generator=g).float()
    pick = (torch.arange(n) % every == 0).view(n, 1, 1)
    k, v = (torch.where(pick, t * spread, t).to(torch.bfloat16) for t in (k, v))
    k = (k.float() / 64).to(torch.bfloat16)
    cass.cass_kv_append(eng.session, 0, k.cuda().contiguous(), v.cuda().contiguous(), 0, n, cass.KV_BF16)
    cass.cass_kv_build_codebook(eng.session, n)
    cass.cass_set_len(eng.session, n - 1)
    q = torch.randn(1, 4, 64, generator=g).to(torch.bfloat16)
    out = torch.zeros(1, 4, 64, dtype=torch.bfloat16, device="cuda")
    cass.cass_draft_attention(eng.session, 0, q.cuda().contiguous(), out)
    torch.cuda.synchronize()
    assert eng.status()[0] == 0
    kd, vd, qd = k.double(), v.double(), q.double()[0].view(2, 2, 64)
    s = torch.einsum("hgd,nhd->hgn", qd, kd) / 8.0                 # nothing pruned or truncated: the records are exact
    ref = torch.einsum("hgn,nhd->hgd", torch.softmax(s, -1), vd).reshape(4, 64).numpy()
    err = np.abs(out[0].cpu().double().numpy() - ref)
    assert (err <= 1e-2 * np.abs(ref).max() + 1e-3).all(), err.max()
    eng.close()
