"""The learned peak map either side of the line where its window and its fallback rows come from the network's image: one
item per CTA pair of the one-kernel form and one line of sight more, both layouts, symmetric and general grids, flagged
channels and half-filled K blocks.  Fallback peaks are the full-grid call's bits; window peaks are rms_synth_window's
up to both forms' errors, whose gate is the precision's (gpu_helpers.TOL) relative to what a noise spectrum's |F| can
reach, 2.5 K sqrt(sum |P|^2)."""
import numpy as np
import pytest

import gpu_helpers as gh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nchan,bad", [(16, 0), (45, 4), (70, 3)])      # 16 channels; 41 of 3 blocks of 16; 67 of 5
@pytest.mark.parametrize("top", [60.0, 63.0])                           # symmetric, general
@pytest.mark.parametrize("layout", ["chan", "los"])
@pytest.mark.parametrize("path", ["bf16x3", "bf16"])
def test_learned_from_image(path, layout, top, nchan, bad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    rng = np.random.default_rng(nchan)
    nphi, W = 101, 64
    w = np.ones(nchan)
    w[rng.choice(nchan, bad, replace=False)] = 0.0
    phi = np.linspace(-60.0, top, nphi)
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    tol = 1e-2 if path == "bf16" else gh.TOL[path]
    with rms.Plan(np.linspace(120e6, 168e6, nchan), phi, path, weights=w) as plan:
        net, win = L.Net(plan, hidden=32, max_batch=64, seed=8), L.Window(plan, W)
        net.set_params(rng.normal(0, 0.4, net.nparams).astype(np.float32))
        for n in (128 * pairs, 128 * pairs + 1):
            X = torch.randn(2, n, nchan, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
            X[:, :, torch.from_numpy(w == 0).cuda()] = float("nan")
            X[0, 7, 0 if w[0] else 1] = float("nan")
            q, u = (x.t().contiguous() if layout == "chan" else x.contiguous() for x in X)
            b, wk, fb, centre = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(4))
            c, wa, wp, fa, fp, php, pka = (torch.empty(n, device="cuda") for _ in range(7))
            nfb = torch.zeros(1, dtype=torch.int64, device="cuda")
            rms.rms_propose(net.handle, q, u, n, layout, W // 4 - 2, None, b, c)
            rms.rms_window_centres(win.handle, b, n, centre)
            rms.rms_synth_window(win.handle, q, u, n, layout, centre, None, wk, wa, wp)
            plan.synth(q, u, n, layout, None, None, fa, fp)
            tau = float(np.nanmedian(c.cpu().numpy()))
            rms.rms_peakmap_learned(win.handle, net.handle, q, u, n, layout, tau, php, pka, fb, nfb)
            plan.sync()
            c, wk, wa, wp, fa, fp, php, pka = (t.cpu().numpy() for t in (c, wk, wa, wp, fa, fp, php, pka))
            fell = fb.cpu().numpy().astype(bool)
            assert int(nfb.item()) == fell.sum() and 0.3 < fell.mean() < 0.99
            np.testing.assert_array_equal(php[fell], fp[fell])
            np.testing.assert_array_equal(pka[fell], fa[fell])
            # a window whose maximum ties with its edge may fall either way: at most a handful
            expect = ~(c >= tau) | (wk <= 0) | (wk >= W - 1)
            assert np.count_nonzero(expect != fell) <= 3
            stay = ~fell & ~expect
            P2 = torch.nansum(X.double() ** 2, dim=(0, 2)).cpu().numpy()
            scale = 2.5 * np.sqrt(P2) / w.sum()
            err = np.abs(pka[stay] - wa[stay]) / scale[stay]
            print(path, layout, top, nchan, n, err.max(), np.mean(php[stay] != wp[stay]))
            assert err.max() <= 2 * tol
            assert np.mean(php[stay] != wp[stay]) <= 2 * tol * 100      # (a tie's chance is of the order of the error)
        net.close()
        win.close()
