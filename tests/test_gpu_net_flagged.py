"""LOS-major gradients of plans with flagged channels: the image columns of those channels belong to no weight, so in the
split-K epilogue some lanes of a warp add nothing while the others go on.  Against the FP64 network oracle at the
operands the kernels multiply, with the tolerance of the full-size test."""
import numpy as np
import pytest

from oracle import net as onet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bf16(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.bfloat16).double().numpy()


# a load's eight columns are four channels, one to a lane column: each of them flagged, all but one, whole groups, and
# every channel of a K block but the first and last
@pytest.mark.parametrize("flagged", [range(0, 45, 4), range(3, 45, 4), [c for c in range(45) if c % 4 != 1],
                                     list(range(4, 12)) + [30], range(17, 31)])
@pytest.mark.parametrize("hidden,n", [(16, 5), (144, 300)])
def test_flagged_los_major_gradient(flagged, hidden, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    rng = np.random.default_rng(hidden + len(flagged))
    nchan, nbins = 45, 33
    w = np.ones(nchan)
    w[list(flagged)] = 0.0
    act = np.flatnonzero(w)
    nin = 2 * len(act)
    p = {"W1": rng.normal(0, 1 / np.sqrt(nin), (hidden, nin)), "b1": rng.normal(0, 0.1, hidden),
         "W2": rng.normal(0, 2.0 / np.sqrt(hidden), (nbins, hidden)), "b2": rng.normal(0, 0.2, nbins)}
    p = {k: v.astype(np.float32).astype(np.float64) for k, v in p.items()}
    Q = rng.normal(size=(n, nchan)).astype(np.float32)
    U = rng.normal(size=(n, nchan)).astype(np.float32)
    Q[:, w == 0] = np.nan
    lab = rng.integers(0, nbins, n).astype(np.int32)
    with rms.Plan(np.linspace(120e6, 168e6, nchan), np.linspace(-60, 60, nbins), "bf16x3", weights=w) as plan:
        net = L.Net(plan, hidden=hidden, max_batch=n, seed=3)
        net.set_params(np.concatenate([p[k].ravel() for k in ("W1", "b1", "W2", "b2")]))
        rms.rms_net_grad(net.handle, torch.from_numpy(Q).cuda(), torch.from_numpy(U).cuda(), n, "los",
                         torch.from_numpy(lab).cuda())
        g = L.unpack(net.grads(), nin, hidden, nbins)
        plan.sync()
        net.close()
    s = np.sqrt(np.mean(Q[:, act].astype(np.float64) ** 2 + U[:, act].astype(np.float64) ** 2, axis=1))
    x = np.stack([Q[:, act], U[:, act]], axis=2).reshape(n, nin)
    pq = dict(p, W1=bf16(p["W1"]), W2=bf16(p["W2"]))
    _, gr = onet.loss_and_grads(pq, bf16(x) / s[:, None], lab)
    for k in ("W1", "b1", "W2", "b2"):
        rel = np.linalg.norm(g[k] - gr[k]) / np.linalg.norm(gr[k])
        assert rel <= 2e-2, (k, rel)
