"""FP16X3 on folded grids: every active channel of every line of sight reaches the scale's maximum.

Each line of sight holds one value 10^6 times the others; were it left out of the maximum, the scaled value would
overflow FP16.  The gate is the precision's (gpu_helpers.TOL).
"""
import numpy as np
import pytest

import gpu_helpers as gh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    rms.build()
    rms.load()
    return rms


# channels either side of 16 warps and of 32 per lane x 16 warps; LOS either side of 128 per block; rows on and off
# 16 bytes (an odd number of LOS, data off 16 bytes)
@pytest.mark.parametrize("nchan,nlos,shift", [(2, 4, 0), (15, 129, 0), (17, 132, 0), (129, 260, 1), (515, 640, 0),
                                              (700, 701, 0)])
@pytest.mark.parametrize("layout", ["chan", "los"])
def test_scale_sees_every_channel(rms, oracle_mod, layout, nchan, nlos, shift):
    rng = np.random.default_rng(nchan)
    freq = np.linspace(120e6, 168e6, nchan)
    w = rng.uniform(0.5, 1.5, nchan)
    w[rng.choice(nchan, nchan // 10, replace=False)] = 0.0
    act = np.flatnonzero(w)
    phi = np.linspace(-60.0, 60.0, 41)
    Q = rng.normal(size=(nlos, nchan)).astype(np.float32)
    U = rng.normal(size=(nlos, nchan)).astype(np.float32)
    i = np.arange(nlos)
    big = act[i % len(act)]
    Q[i[::2], big[::2]] = 1e6
    U[i[1::2], big[1::2]] = -1e6
    Q[:, w == 0] = 1e30                                  # flagged channels stay out of it
    buf = torch.zeros(2, nlos * nchan + 4, device="cuda")
    q, u = (buf[k, shift:shift + nlos * nchan] for k in range(2))
    for t, X in ((q, Q), (u, U)):
        t.copy_(torch.from_numpy(np.ascontiguousarray(X.T if layout == "chan" else X)).reshape(-1))
    F = torch.empty(nlos, len(phi), 2, device="cuda")
    with rms.Plan(freq, phi, "fp16x3", weights=w) as plan:
        for kind in (rms.RMS_CONTRACT_AUTO, rms.RMS_CONTRACT_SINGLE):
            rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_CONTRACTION, kind)
            plan.synth(q, u, nlos, layout, F)
            plan.sync()
            Fh = F.cpu().numpy()
            Qa, Ua = np.where(w == 0, 0, Q), np.where(w == 0, 0, U)
            per, _ = gh.errors(Fh[..., 0] + 1j * Fh[..., 1], oracle_mod.synth(Qa, Ua, oracle_mod.plan(freq, "freq", w), phi))
            assert per.max() <= gh.TOL["fp16x3"], (kind, per.max())
