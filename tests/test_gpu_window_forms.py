"""Window synthesis either side of the lines between its one-kernel form and the split with the rotating contraction: one
item per CTA pair and one line of sight more, few and more channels, a half-empty second round, many rounds -- against
the FP64 sum over each line of sight's own window, relative to what a noise spectrum's |F| can reach."""
import numpy as np
import pytest

import gpu_helpers as gh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# rounds: items of 128 LOS in units of one per CTA pair (76 on 152 SMs)
@pytest.mark.parametrize("rounds,nchan,layout,width", [(1.0, 40, "los", 64), (1.01, 40, "los", 64), (1.01, 64, "los", 64),
                                                      (1.01, 65, "los", 64), (1.01, 48, "los", 128), (1.01, 49, "los", 128),
                                                      (1.49, 151, "chan", 64), (1.51, 151, "chan", 64),
                                                      (1.01, 150, "chan", 8), (1.01, 151, "los", 8),
                                                      (8.0, 48, "chan", 64), (8.1, 48, "chan", 64), (8.1, 49, "chan", 64)])
@pytest.mark.parametrize("path", ["bf16x3", "bf16"])
def test_window_forms(path, rounds, nchan, layout, width):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    rng = np.random.default_rng(nchan)
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    n = int(rounds * pairs * 128) - (0 if rounds == int(rounds) else 3)
    freq = np.linspace(120e6, 168e6, nchan + 2)
    w = np.ones(nchan + 2)
    w[[0, nchan // 2]] = 0.0                              # nchan active channels
    phi = np.linspace(-60.0, 60.0, 201)
    X = torch.randn(2, n, nchan + 2, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    q, u = (x.t().contiguous() if layout == "chan" else x for x in X)
    centre = rng.integers(width // 2, 401 - width // 2, n).astype(np.int32)
    with rms.Plan(freq, phi, path, weights=w) as plan:
        win = L.Window(plan, width)
        F = torch.full((n, width, 2), 7.0, device="cuda")
        wi = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        wa = torch.zeros(n, device="cuda")
        rms.rms_synth_window(win.handle, q, u, n, layout, torch.from_numpy(centre).cuda(), F, wi, wa, None)
        plan.sync()
        win.close()
    idx, best = gh.argmax_fp32(F.cpu().numpy())
    np.testing.assert_array_equal(wi.cpu().numpy(), idx)
    np.testing.assert_array_equal(wa.cpu().numpy(), np.sqrt(best).astype(np.float32))
    rows = np.unique(np.r_[0, n - 1, rng.choice(n, 300)])
    live = np.flatnonzero(w)
    lam2 = (299792458.0 / freq[live]) ** 2
    x = lam2 - lam2.mean()
    Xr = X[:, torch.from_numpy(rows).cuda()][:, :, torch.from_numpy(live).cuda()].double().cpu().numpy()
    P = Xr[0] + 1j * Xr[1]
    fine = phi[0] + (phi[1] - phi[0]) / 2 * (centre[rows][:, None] + np.arange(-width // 2, width // 2)[None, :])
    Fo = np.einsum("lc,lmc->lm", P, np.exp(-2j * fine[:, :, None] * x)) / nchan
    Fg = F[torch.from_numpy(rows).cuda()].double().cpu().numpy()
    scale = 2.5 * np.sqrt((np.abs(P) ** 2).sum(axis=1)) / nchan
    err = (np.abs(Fg[..., 0] + 1j * Fg[..., 1] - Fo).max(axis=1) / scale).max()
    print(path, rounds, nchan, layout, width, err)
    assert err <= (1e-2 if path == "bf16" else gh.TOL[path])
