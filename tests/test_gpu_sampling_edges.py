"""Edges of the clustered softmax and inverse-CDF kernels: vocabularies around the splits over CTAs and registers and beyond
both, one-hot and empty residual weights, thresholds at both ends."""
import numpy as np
import pytest
import torch

from oracle import model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cass():
    import paper_2605_26558_b200 as m
    return m


@pytest.mark.parametrize("vocab", [1, 5, 255, 257, 2048, 2049, 4097, 16385, 32769, 131073, 163841, 460001])
def test_softmax_and_draws_around_the_splits(cass, vocab):
    rows = 3
    g = torch.Generator().manual_seed(vocab)
    logits = (torch.randn(rows, vocab, generator=g) * 4).cuda()
    logits[1] = -3.0                                        # a flat row
    probs = torch.full((rows, vocab), -1.0, device="cuda")
    cass.cass_softmax(logits, rows, vocab, 0.8, probs)
    want = np.stack([model.softmax(logits[r].cpu().numpy(), 0.8) for r in range(rows)])
    got = probs.cpu().numpy().astype(np.float64)
    assert np.allclose(got, want, rtol=2e-5, atol=1e-9)
    probs[2] = 0.0
    probs[2, vocab // 2] = 1.0                              # one-hot: found for every u
    c = np.cumsum(probs.cpu().numpy().astype(np.float64), axis=1)
    for u in (0.0, 0.25, 0.999999):
        toks = torch.full((rows,), -1, dtype=torch.int32, device="cuda")
        cass.cass_sample(probs, rows, vocab, torch.full((rows,), u, device="cuda"), toks)
        t = toks.tolist()
        assert t[2] == vocab // 2
        for r in range(2):
            lo = c[r, t[r] - 1] if t[r] else 0.0
            assert lo <= u * c[r, -1] + 2e-5 and c[r, t[r]] >= u * c[r, -1] - 2e-5, (r, u, t[r])


@pytest.mark.parametrize("vocab", [257, 5000, 128256])
def test_acceptance_draws_from_the_residual_or_the_target(cass, vocab):
    """Sequence 0 rejects its first draft and draws from the only positive residual; 1 accepts all and draws from the last
    target row; 2 rejects where p and q agree everywhere else, so that no residual is left and the target itself is drawn."""
    g = 2
    p = torch.zeros(3, g + 1, vocab)
    q = torch.zeros(3, g, vocab)
    p[0, 0, 7], q[0, 0, 3] = 1.0, 1.0
    p[0, 1:, 1] = 1.0
    q[0, 1, 1] = 1.0
    p[1, :, 5], q[1, :, 5] = 1.0, 1.0
    p[1, 2] = 0.0
    p[1, 2, vocab - 1] = 1.0
    p[2, :, 9], q[2, :, 9] = 0.5, 1.0                       # r q > p: rejected, and p - q is nowhere positive
    draft = torch.tensor([[3, 1], [5, 5], [9, 9]], dtype=torch.int32)
    n_acc, out, nxt = (torch.full((n,), -9, dtype=torch.int32, device="cuda") for n in (3, 9, 3))
    cass.cass_accept_sampling(None, 3, draft.cuda(), p.cuda(), q.cuda(), vocab, torch.full((3, g), 0.9, device="cuda"),
                              torch.full((3,), 0.5, device="cuda"), g, n_acc, out, nxt)
    assert n_acc.tolist() == [0, 2, 0]
    assert out.view(3, 3).tolist() == [[7, -1, -1], [5, 5, vocab - 1], [9, -1, -1]] and nxt.tolist() == [7, vocab - 1, 9]


def test_threads_with_different_vocabularies(cass):
    """Calls of two threads, each on its own stream, whose draws need different amounts of shared memory."""
    import threading
    sizes, errors = (1000, 200000), []
    probs = [torch.full((1, n), 1.0 / n, device="cuda") for n in sizes]
    u = torch.full((1,), 0.5, device="cuda")
    start = threading.Barrier(len(sizes))

    def calls(i):
        stream, tok = torch.cuda.Stream(), torch.zeros(1, dtype=torch.int32, device="cuda")
        start.wait()
        try:
            for _ in range(3000):
                cass.cass_sample(probs[i], 1, sizes[i], u, tok, stream=stream)
            stream.synchronize()
            assert abs(int(tok.item()) - sizes[i] // 2) <= 1 + sizes[i] // 10000
        except Exception as e:                              # noqa: BLE001
            errors.append((sizes[i], repr(e)))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=calls, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
