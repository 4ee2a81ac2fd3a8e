"""Window synthesis at its edges (widths, ragged LOS counts, partial K blocks, rows too long to stage, data off
16 bytes, centres at both clamps) against the FP64 sum over each LOS's own window."""
import numpy as np
import pytest

import gpu_helpers as gh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,nlos,nchan,layout,shift", [(8, 1, 33, "los", 0), (64, 63, 75, "chan", 0),
                                                           (64, 129, 75, "los", 1), (128, 200, 75, "los", 0),
                                                           (64, 300, 75, "chan", 1), (24, 130, 600, "los", 0),
                                                           (64, 20011, 40, "los", 0), (64, 100, 560, "chan", 0)])
@pytest.mark.parametrize("path", ["bf16x3", "bf16"])
def test_window_edges(oracle_mod, path, width, nlos, nchan, layout, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    rng = np.random.default_rng(width + nlos + nchan)
    freq = np.linspace(120e6, 168e6, nchan)
    w = rng.uniform(0.5, 1.5, nchan)
    w[rng.choice(nchan, 3, replace=False)] = 0.0
    phi = np.linspace(-60.0, 60.0, 121)
    n_fine = 2 * (len(phi) - 1) + 1
    op = oracle_mod.plan(freq, "freq", w)
    Q = rng.normal(size=(nlos, nchan)).astype(np.float32)
    U = rng.normal(size=(nlos, nchan)).astype(np.float32)
    Q[:, w == 0] = np.nan
    centre = rng.integers(0, n_fine, nlos).astype(np.int32)
    centre[0] = -5                                   # below and above the clamps
    centre[-1] = n_fine + 9
    lo, hi = width // 2, n_fine - 1 - (width // 2 - 1)
    c = np.clip(centre, lo, hi)
    arr = [torch.zeros(nlos * nchan + 4, device="cuda")[shift:shift + nlos * nchan] for _ in range(2)]
    for t, a in zip(arr, (Q, U)):
        t.copy_(torch.from_numpy(np.ascontiguousarray(a.T if layout == "chan" else a)).reshape(-1))
    with rms.Plan(freq, phi, path, weights=w) as plan:
        win = L.Window(plan, width)
        F = torch.full((nlos, width, 2), 7.0, device="cuda")
        wi = torch.full((nlos,), -7, dtype=torch.int32, device="cuda")
        wa, wp = torch.zeros(nlos, device="cuda"), torch.zeros(nlos, device="cuda")
        rms.rms_synth_window(win.handle, arr[0], arr[1], nlos, layout, torch.from_numpy(centre).cuda(), F, wi, wa, wp)
        plan.sync()
        Fg = F.cpu().numpy()
        win.close()
    idx, best = gh.argmax_fp32(Fg)
    np.testing.assert_array_equal(wi.cpu().numpy(), idx)
    np.testing.assert_array_equal(wa.cpu().numpy(), np.sqrt(best).astype(np.float32))
    step = (phi[1] - phi[0]) / 2
    fine = phi[0] + step * (c[:, None] + np.arange(-width // 2, width // 2)[None, :])
    np.testing.assert_allclose(wp.cpu().numpy(), fine[np.arange(nlos), idx], rtol=2e-7, atol=1e-6)
    rows = np.unique(np.r_[0, nlos - 1, rng.choice(nlos, min(nlos, 300))])
    live = np.flatnonzero(w)
    x = op.lambda2[live] - op.lambda0sq
    P = (Q[rows][:, live].astype(np.float64) + 1j * U[rows][:, live]) * w[live]
    Fo = op.K * np.einsum("lc,lmc->lm", P, np.exp(-2j * fine[rows][:, :, None] * x))
    got = Fg[rows, :, 0] + 1j * Fg[rows, :, 1].astype(np.float64)
    # a window is a slice of its LOS's F, so the error is relative to what F can reach: noise spectra have
    # rms(F) = K sqrt(sum w^2 |P|^2), a row maximum on the full grid of about 2.5 times that
    scale = 2.5 * op.K * np.sqrt((np.abs(P) ** 2).sum(axis=1))
    err = (np.abs(got - Fo).max(axis=1) / scale).max()
    print(path, width, nlos, nchan, layout, err)
    assert err <= (1e-2 if path == "bf16" else gh.TOL[path])
