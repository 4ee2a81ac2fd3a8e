"""Phi grids that are not symmetric about zero (the general form of the layout stage and the contraction) at their edges:
every precision, both layouts, single CTAs and CTA pairs under both schedules, with F and without, against the FP64
oracle; and the learned peak map's fallback on such a grid against the calls it is made of.

The spectra are noise, whose |F| has rms K sqrt(sum w^2 |P|^2) and a maximum of about 2.5 times that on a full grid, so
an error is relative to that: a grid of a few samples can miss its LOS's maximum.  The gates are the precisions'
(gpu_helpers.TOL; plain BF16's per line of sight 1e-2)."""
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


def cube(rng, nlos, nchan, layout, shift, w):
    Q = rng.normal(size=(nlos, nchan)).astype(np.float32)
    U = rng.normal(size=(nlos, nchan)).astype(np.float32)
    Q[:, w == 0] = np.nan
    if nlos > 3:
        U[2, np.flatnonzero(w)[0]] = np.nan
        Q[3] = 0.0
        U[3] = 0.0
    arr = [torch.zeros(nlos * nchan + 4, device="cuda")[shift:shift + nlos * nchan] for _ in range(2)]
    for t, a in zip(arr, (Q, U)):
        t.copy_(torch.from_numpy(np.ascontiguousarray(a.T if layout == "chan" else a)).reshape(-1))
    return Q, U, arr


# one sample; 208 phase rows and two more; one 256-row pair tile and more; five tiles; one K block, an odd number of them,
# and 40 and 41 (plain BF16 with F changes its issuer there); ragged M tiles; rows off 16 bytes
@pytest.mark.parametrize("nlos,nchan,nphi,layout,shift", [(1, 75, 1, "los", 0), (127, 75, 2, "chan", 0), (129, 75, 104, "los", 1),
                                                         (257, 75, 105, "chan", 1), (300, 656, 129, "los", 0),
                                                         (1000, 640, 257, "chan", 0), (513, 16, 515, "chan", 0)])
@pytest.mark.parametrize("path", ["bf16", "bf16x3", "fp16x3", "fp32_table", "fp32_fly"])
def test_general_edges(rms, oracle_mod, path, nlos, nchan, nphi, layout, shift):
    rng = np.random.default_rng(nlos + nphi)
    freq = np.linspace(120e6, 168e6, nchan)
    w = rng.uniform(0.5, 1.5, nchan)
    if nchan == 75:
        w[rng.choice(nchan, 7, replace=False)] = 0.0
    phi = np.linspace(-60.0, 63.0, nphi) if nphi > 1 else np.array([7.0])
    Q, U, (q, u) = cube(rng, nlos, nchan, layout, shift, w)
    op = oracle_mod.plan(freq, "freq", w)
    Fo = oracle_mod.synth(Q, U, op, phi)
    good = np.all(np.isfinite(Fo), axis=1)
    live = np.flatnonzero(w)
    P2 = (Q[:, live].astype(np.float64) ** 2 + U[:, live].astype(np.float64) ** 2) * w[live] ** 2
    scale = 2.5 * op.K * np.sqrt(P2.sum(axis=1))
    scale[scale == 0] = 1.0
    tensor = not path.startswith("fp32")
    with rms.Plan(freq, phi, path, weights=w) as plan:
        for kind in (rms.RMS_CONTRACT_AUTO, rms.RMS_CONTRACT_SINGLE, rms.RMS_CONTRACT_PAIR) if tensor else (None,):
            got = []
            for sched in (rms.RMS_SCHEDULE_AUTO, rms.RMS_SCHEDULE_WHOLE) if tensor else (None,):
                if tensor:
                    rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_CONTRACTION, kind)
                    rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_SCHEDULE, sched)
                for with_f in (True, False):
                    F = torch.full((nlos, nphi, 2), 3.0, device="cuda") if with_f else None
                    pi = torch.full((nlos,), -7, dtype=torch.int32, device="cuda")
                    pa, pp = torch.zeros(nlos, device="cuda"), torch.zeros(nlos, device="cuda")
                    plan.synth(q, u, nlos, layout, F, pi, pa, pp)
                    plan.sync()
                    if tensor and kind != rms.RMS_CONTRACT_AUTO:
                        assert rms.rms_plan_info(plan.handle, rms.RMS_INFO_LAST_PAIR) == (kind == rms.RMS_CONTRACT_PAIR)
                    got.append(([F] if with_f else []) + [pi, pa, pp])
            Fh = got[0][0].cpu().numpy()
            err = np.abs(Fh[good, :, 0] + 1j * Fh[good, :, 1].astype(np.float64) - Fo[good]).max(axis=1) / scale[good]
            print(path, kind, nlos, nchan, nphi, layout, err.max())
            assert err.max() <= (1e-2 if path == "bf16" else gh.TOL[path])
            assert np.all(np.isnan(Fh[~good]))
            gh.check_peaks_self(Fh, *(t.cpu().numpy() for t in got[0][1:]), phi)
            if nlos > 3:
                assert got[0][1][2] == -1 and got[0][1][3] == 0
            for other in got[1:]:                    # the other schedule, and calls without F: the same bits
                for x, y in zip(got[0][-len(other):], other):
                    assert torch.equal(x.view(torch.int32), y.view(torch.int32))


@pytest.mark.parametrize("layout", ["chan", "los"])
@pytest.mark.parametrize("path", ["bf16x3", "bf16"])
def test_learned_fallback_on_a_general_grid(rms, path, layout):
    from paper_1810_06250_gb300 import learned as L
    rng = np.random.default_rng(5)
    n, nchan, nphi, W = 1000, 75, 201, 64
    freq = np.linspace(120e6, 168e6, nchan)
    w = np.ones(nchan)
    w[rng.choice(nchan, 7, replace=False)] = 0.0
    _, _, (q, u) = cube(rng, n, nchan, layout, 0, w)
    with rms.Plan(freq, np.linspace(-60.0, 63.0, nphi), path, weights=w) as plan:
        net, win = L.Net(plan, hidden=64, max_batch=64, seed=8), L.Window(plan, W)
        p = rng.normal(0, 0.3, net.nparams).astype(np.float32)
        net.set_params(p)
        b = torch.empty(n, dtype=torch.int32, device="cuda")
        c, wa, wp, fa, fp, php, pka = (torch.empty(n, device="cuda") for _ in range(7))
        wk, fb, centre = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(3))
        rms.rms_propose(net.handle, q, u, n, layout, W // 4 - 2, None, b, c)
        rms.rms_window_centres(win.handle, b, n, centre)
        rms.rms_synth_window(win.handle, q, u, n, layout, centre, None, wk, wa, wp)
        plan.synth(q, u, n, layout, None, None, fa, fp)
        tau = float(np.nanmedian(c.cpu().numpy()))
        rms.rms_peakmap_learned(win.handle, net.handle, q, u, n, layout, tau, php, pka, fb, None)
        plan.sync()
        c, wk, wa, wp, fa, fp, php, pka, fb = (t.cpu().numpy() for t in (c, wk, wa, wp, fa, fp, php, pka, fb))
        net.close()
        win.close()
    expect = ~(c >= tau) | (wk <= 0) | (wk >= W - 1)
    np.testing.assert_array_equal(fb.astype(bool), expect)
    assert 0.3 < expect.mean() < 0.99
    np.testing.assert_array_equal(php, np.where(expect, fp, wp))
    np.testing.assert_array_equal(pka, np.where(expect, fa, wa))
