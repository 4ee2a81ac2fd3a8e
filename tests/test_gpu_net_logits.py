"""Logits of rms_propose at the edges of the 16-column blocks and 32-row warps that store them: every value in place,
nothing beyond the rows and bins of the call, and the same bin and confidence as without them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbins", [2, 15, 17, 104, 401, 512])
@pytest.mark.parametrize("n", [1, 16, 17, 129])
def test_logits_in_place(n, nbins):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    rng = np.random.default_rng(nbins)
    nchan, hidden, guard = 20, 16, 64
    Q, U = (rng.normal(size=(n, nchan)).astype(np.float32) for _ in range(2))
    q, u = torch.from_numpy(Q).cuda(), torch.from_numpy(U).cuda()
    with rms.Plan(np.linspace(120e6, 168e6, nchan), np.linspace(-60, 60, nbins), "bf16x3") as plan:
        net = L.Net(plan, hidden=hidden, max_batch=16, seed=3)
        W1, b1 = rng.normal(0, 0.2, (hidden, 2 * nchan)), np.full(hidden, 2.0)
        W2, b2 = rng.normal(0, 1, (nbins, hidden)), 8.0 * np.arange(nbins)
        net.set_params(np.concatenate([W1.ravel(), b1, W2.ravel(), b2]).astype(np.float32))
        buf = torch.full((guard + n * nbins + guard,), 7.0, device="cuda")
        z = buf[guard:guard + n * nbins].view(n, nbins)
        out = [[torch.full((n,), -7, dtype=torch.int32, device="cuda"), torch.zeros(n, device="cuda")] for _ in range(2)]
        rms.rms_propose(net.handle, q, u, n, "los", 3, z, *out[0])
        rms.rms_propose(net.handle, q, u, n, "los", 3, None, *out[1])
        plan.sync()
        net.close()
    assert bool((buf[:guard] == 7.0).all()) and bool((buf[guard + n * nbins:] == 7.0).all())
    for a, b in zip(*out):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    # the bias tells every bin apart from its neighbours, the spectra every row: BF16 rounding of weights, inputs and h
    # moves a logit by at most |W2| |h| 2^-7
    bf = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(torch.bfloat16).double().numpy()
    s = np.sqrt(np.mean(Q.astype(np.float64) ** 2 + U.astype(np.float64) ** 2, axis=1, keepdims=True))
    x = np.stack([Q, U], axis=2).reshape(n, 2 * nchan)
    h = np.maximum(bf(x) @ bf(W1).T / s + b1, 0.0)
    zr = bf(h) @ bf(W2).T + b2
    assert np.all(np.abs(z.double().cpu().numpy() - zr) <= 2.0 ** -7 * (h @ np.abs(W2).T) + 1e-3)
