"""The policy's own kernels at the edges of their tiles: one training step's
gradients against PyTorch autograd for row counts around a product's 16, a
tile's 64 and a stage's 256 rows and for groups smaller and larger than a warp;
scores around the 16 rows of a product and the 32 of a warp; features in
buffers of every alignment."""
import numpy as np
import pytest

import paper_2207_12116_gb300 as pccp
from synthetic import config_instance
from tests.test_gpu_policy import bf, ref_scores

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[2], [16], [17], [40, 1, 23], [31, 32], [33, 32], [100, 3], [64] * 4,
                                   [64] * 4 + [2], [5] * 203, [1000, 24]])
def test_training_step(sizes):
    g = np.random.default_rng(sum(sizes))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    x = g.uniform(0, 1, (int(off[-1]), 12)).astype(np.float32)
    t = g.uniform(0, 1, int(off[-1])).astype(np.float32)
    for a, b in zip(off[:-1], off[1:]):
        t[a:b] /= t[a:b].sum()
    pol = pccp.Policy.random(7)
    w0 = pol.weights()
    loss = pol.train_step(*(torch.from_numpy(v).cuda() for v in (x, off, t)), lr=1e-3)
    got, w1 = pol.gradients(), pol.weights()
    P = {k: torch.tensor(w0[k], requires_grad=True) for k in ("w1", "b1", "w2", "b2", "w3")}
    ste = lambda a: a + (bf(a.detach()) - a).detach()  # BF16 value, identity gradient
    h1 = torch.relu(ste(torch.from_numpy(x)) @ ste(P["w1"]).T + P["b1"])
    h2 = torch.relu(ste(h1) @ ste(P["w2"]).T + P["b2"])
    s = h2 @ P["w3"] + w0["b3"]
    L = sum(-(torch.from_numpy(t[a:b]) * torch.log_softmax(s[a:b], 0)).sum()
            for a, b in zip(off[:-1], off[1:])) / len(sizes)
    L.backward()
    assert abs(loss - L.item()) < 1e-2 * max(1.0, abs(L.item()))
    for k, v in P.items():
        gr = v.grad.numpy()
        assert np.abs(got[k] - gr).max() <= 2e-2 * np.abs(gr).max() + 1e-6, k
        # Adam's first step: lr against the gradient's sign
        big = np.abs(gr) > 0.1 * np.abs(gr).max()
        assert np.allclose((w1[k] - w0[k])[big], -1e-3 * np.sign(gr[big]), rtol=0.05), k
    # the images of the new weights serve the next scores
    assert np.allclose(pol.score(torch.from_numpy(x).cuda()).cpu(), ref_scores(w1, x), rtol=1e-2, atol=1e-2)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 255, 256, 257, 77824, 77825])
def test_scores(n):
    pol = pccp.Policy.random(n)
    w, x = pol.weights(), np.random.default_rng(n).uniform(-1, 2, (n, 12)).astype(np.float32)
    flat = torch.empty(12 * n + 1, device="cuda")
    for k in (0, 1):  # rows need no alignment beyond a float's
        f = flat[k:k + 12 * n].view(n, 12)
        f.copy_(torch.from_numpy(x))
        s, r = pol.score(f).cpu(), ref_scores(w, x)
        assert s.shape == (n,)
        tol = 1e-2 * float(r.abs().max()) + 1e-3
        assert torch.allclose(s, r, atol=tol, rtol=1e-2)


def test_features_in_unaligned_buffers():
    m = pccp.Model.from_rcpsp(config_instance("tiny8", 3))
    lb = torch.from_numpy(np.tile(m.lb0, (5, 1)).astype(np.int32)).cuda()
    ub = torch.from_numpy(np.tile(m.ub0, (5, 1)).astype(np.int32)).cuda()
    lb[:, 0] += torch.arange(5, dtype=torch.int32, device="cuda")
    want = pccp.policy_features(m, lb, ub)
    import ctypes
    n = want.numel()
    for k in range(1, 4):
        flat = torch.zeros(n + 8, device="cuda")
        out = flat[k:k + n]
        rc = pccp.pccp_policy_features(m.handle, 5, *(ctypes.c_void_p(v.data_ptr()) for v in (lb, ub)),
                                            ctypes.c_void_p(0), ctypes.c_void_p(out.data_ptr()),
                                            ctypes.c_void_p(0))
        torch.cuda.synchronize()
        assert rc == 0 and torch.equal(out.view_as(want), want) and not flat[k + n:].any()
