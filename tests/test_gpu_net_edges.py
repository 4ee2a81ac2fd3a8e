"""Network epilogues at their edges: column quarters that are partial or empty, one row, ragged batches, one and two
tiles of bins, the smallest and largest hidden layer -- gradients and proposals against the FP64 network oracle at the
operands the kernels multiply (BF16 weights and data), with the tolerances of the full-size test."""
import numpy as np
import pytest

from oracle import net as onet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bf16(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.bfloat16).double().numpy()


@pytest.mark.parametrize("hidden,nbins,n,layout", [(16, 2, 1, "los"), (16, 33, 127, "chan"), (64, 64, 128, "los"),
                                                   (48, 257, 129, "chan"), (256, 401, 257, "los"), (256, 512, 300, "chan")])
def test_net_edges(hidden, nbins, n, layout):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    rng = np.random.default_rng(hidden + nbins)
    nchan = 45
    freq = np.linspace(120e6, 168e6, nchan)
    w = np.ones(nchan)
    w[[3, 17]] = 0.0
    act = np.flatnonzero(w)
    nin = 2 * len(act)
    p = {"W1": rng.normal(0, 1 / np.sqrt(nin), (hidden, nin)), "b1": rng.normal(0, 0.1, hidden),
         "W2": rng.normal(0, 2.0 / np.sqrt(hidden), (nbins, hidden)), "b2": rng.normal(0, 0.2, nbins)}
    p = {k: v.astype(np.float32).astype(np.float64) for k, v in p.items()}
    Q = rng.normal(size=(n, nchan)).astype(np.float32)
    U = rng.normal(size=(n, nchan)).astype(np.float32)
    Q[:, w == 0] = np.nan
    lab = rng.integers(0, nbins, n).astype(np.int32)
    q, u = (torch.from_numpy(np.ascontiguousarray(a.T if layout == "chan" else a)).cuda() for a in (Q, U))
    with rms.Plan(freq, np.linspace(-60, 60, nbins), "bf16x3", weights=w) as plan:
        net = L.Net(plan, hidden=hidden, max_batch=n, seed=3)
        net.set_params(np.concatenate([p[k].ravel() for k in ("W1", "b1", "W2", "b2")]))
        loss = torch.zeros(1, device="cuda")
        rms.rms_net_grad(net.handle, q, u, n, layout, torch.from_numpy(lab).cuda(), loss)
        g = L.unpack(net.grads(), nin, hidden, nbins)
        z = torch.full((n, nbins), 9.0, device="cuda")
        b = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        c = torch.zeros(n, device="cuda")
        rms.rms_propose(net.handle, q, u, n, layout, 3, z, b, c)
        plan.sync()
        net.close()
    s = np.sqrt(np.mean(Q[:, act].astype(np.float64) ** 2 + U[:, act].astype(np.float64) ** 2, axis=1))
    x = np.stack([Q[:, act], U[:, act]], axis=2).reshape(n, nin)
    pq = dict(p, W1=bf16(p["W1"]), W2=bf16(p["W2"]))
    lr, gr = onet.loss_and_grads(pq, bf16(x) / s[:, None], lab)
    assert abs(float(loss.item()) - lr) <= 1e-2 * abs(lr)
    for k in ("W1", "b1", "W2", "b2"):
        rel = np.linalg.norm(g[k] - gr[k]) / np.linalg.norm(gr[k])
        assert rel <= 2e-2, (k, rel)
    # the proposal from the kernel's own logits: first maximum and the softmax mass within 3 bins of it
    zh = z.cpu().numpy().astype(np.float64)
    np.testing.assert_array_equal(b.cpu().numpy(), np.argmax(zh, axis=1))
    e = np.exp(zh - zh.max(axis=1, keepdims=True))
    near = np.abs(np.arange(nbins)[None, :] - np.argmax(zh, axis=1)[:, None]) <= 3
    np.testing.assert_allclose(c.cpu().numpy(), (e * near).sum(1) / e.sum(1), atol=2e-5)
