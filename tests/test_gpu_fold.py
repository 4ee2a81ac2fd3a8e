"""Folded contraction (phi grids symmetric about zero) at its edges, against the FP64 oracle and the general path.

The gates are those of the precisions (gpu_helpers.TOL): folding forms the same
products from the same split operands and adds them in another order.
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


def grid(kind, n):
    """Symmetric grids: uniform, uneven steps, descending."""
    if kind == "uneven":
        h = np.cumsum(np.linspace(0.3, 0.9, n // 2))
        return np.concatenate([-h[::-1], [0.0] * (n % 2), h])
    phi = np.linspace(-60.0, 60.0, n) if n > 1 else np.zeros(1)
    return phi[::-1].copy() if kind == "down" else phi


# one column pair; even and odd grids; one pair either side of the 208- and 256-row tiles; three tiles
@pytest.mark.parametrize("kind,nphi", [("up", 1), ("up", 2), ("up", 3), ("up", 103), ("down", 104), ("up", 207),
                                       ("uneven", 209), ("up", 256), ("up", 257), ("uneven", 515), ("down", 630)])
@pytest.mark.parametrize("path", ["bf16x3", "fp16x3", "bf16", "fp32_table", "fp32_fly"])
def test_fold_edges(rms, oracle_mod, path, kind, nphi):
    rng = np.random.default_rng(nphi)
    nchan = 75                                   # 68 active: two full K blocks of 32 and a partial one
    freq = np.linspace(120e6, 168e6, nchan)
    w = rng.uniform(0.5, 1.5, nchan)
    w[rng.choice(nchan, 7, replace=False)] = 0.0
    phi = grid(kind, nphi)
    op = oracle_mod.plan(freq, "freq", w)
    guard = 16
    with rms.Plan(freq, phi, path, weights=w) as plan, \
            rms.Plan(freq, np.append(phi, 77.0), path, weights=w) as general:     # one more sample: no symmetry
        for nlos, shift, layout in ((1, 0, "chan"), (63, 1, "los"), (65, 2, "chan"), (130, 3, "los"), (257, 1, "chan")):
            Q = rng.normal(size=(nlos, nchan)).astype(np.float32)
            U = rng.normal(size=(nlos, nchan)).astype(np.float32)
            Q[:, w == 0] = np.nan
            if nlos > 3:
                U[2, np.flatnonzero(w)[0]] = np.nan
                Q[3] = 0.0
                U[3] = 0.0
            q = torch.from_numpy(np.ascontiguousarray(Q.T if layout == "chan" else Q)).cuda()
            u = torch.from_numpy(np.ascontiguousarray(U.T if layout == "chan" else U)).cuda()
            # F at every 8-byte offset within a sector, between guard values that must survive
            buf = torch.full((guard + nlos * nphi + guard, 2), 7.0, device="cuda")
            F = buf[guard + shift:guard + shift + nlos * nphi].view(nlos, nphi, 2)
            pi = torch.full((nlos,), -7, dtype=torch.int32, device="cuda")
            pa, pp = torch.zeros(nlos, device="cuda"), torch.zeros(nlos, device="cuda")
            plan.synth(q, u, nlos, layout, F, pi, pa, pp)
            G = torch.empty(nlos, nphi + 1, 2, device="cuda")
            general.synth(q, u, nlos, layout, G)
            plan.sync()
            general.sync()
            outside = torch.cat([buf[:guard + shift], buf[guard + shift + nlos * nphi:]])
            assert bool((outside == 7.0).all())
            Fh, Gh = F.cpu().numpy(), G.cpu().numpy()[:, :nphi]
            Fo = oracle_mod.synth(Q, U, op, phi)
            good = np.all(np.isfinite(Fo), axis=1)
            assert np.all(np.isnan(Fh[~good]))
            # a grid of a few samples can miss its LOS's maximum, so that the error relative to the row exceeds
            # the precision's gate on either path: there the folded error is held to the general path's
            per, _ = gh.errors(Fh[good, :, 0] + 1j * Fh[good, :, 1], Fo[good])
            gen, _ = gh.errors(Gh[good, :, 0] + 1j * Gh[good, :, 1], Fo[good])
            print(path, nphi, nlos, layout, per.max(), gen.max())
            tol = 1e-2 if path == "bf16" else gh.TOL[path]
            assert np.all((per <= tol) | (per <= 1.5 * gen)), (nlos, layout, per.max(), gen.max())
            gh.check_peaks_self(Fh, pi.cpu().numpy(), pa.cpu().numpy(), pp.cpu().numpy(), phi)
            if nlos > 3:
                assert pi[2] == -1 and pi[3] == 0


# several items per CTA pair with a ragged last one; three phase tiles; LOS-major rows too long for the staging
# slots (75 channels otherwise); an odd number of LOS (channel-major rows off 16 bytes); data off 16 bytes
@pytest.mark.parametrize("nlos,nchan,nphi,layout,shift", [(20011, 75, 103, "los", 0), (20011, 75, 401, "chan", 0),
                                                         (29500, 75, 515, "los", 0), (20000, 75, 257, "chan", 1),
                                                         (20011, 75, 64, "los", 1), (19999, 600, 33, "los", 0)])
@pytest.mark.parametrize("path", ["bf16x3", "fp16x3", "bf16"])
def test_one_kernel_matches_two(rms, path, nlos, nchan, nphi, layout, shift):
    """The layout stage inside the contraction: the same bits as the split kernel and the contraction in turn."""
    rng = np.random.default_rng(nlos + nphi)
    freq = np.linspace(120e6, 168e6, nchan)
    w = rng.uniform(0.5, 1.5, nchan)
    w[rng.choice(nchan, 7, replace=False)] = 0.0
    phi = grid("up", nphi)
    data = torch.randn(2, nlos * nchan + 4, device="cuda", generator=torch.Generator("cuda").manual_seed(nphi))
    data[0, 5 * nchan:6 * nchan] = float("nan")
    data[:, 7 * nchan:9 * nchan] = 0.0
    q, u = (data[i, shift:shift + nlos * nchan] for i in range(2))
    got = []
    with rms.Plan(freq, phi, path, weights=w) as plan:
        for kind in (rms.RMS_CONTRACT_AUTO, rms.RMS_CONTRACT_PAIR):
            rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_CONTRACTION, kind)
            for with_f in (True, False):
                F = torch.full((nlos, nphi, 2), 3.0, device="cuda") if with_f else None
                out = [torch.full((nlos,), -7, dtype=torch.int32, device="cuda")]
                out += [torch.full((nlos,), -7.0, device="cuda") for _ in range(5)]
                rms.rms_synth_peaks(plan.handle, q, u, nlos, layout, F, *out)
                plan.sync()
                got.append(([F] if with_f else []) + out)
    for a, b in ((0, 2), (1, 3)):
        for x, y in zip(got[a], got[b]):
            assert torch.equal(x.view(torch.int32), y.view(torch.int32))
    for x, y in zip(got[0][1:], got[1]):
        assert torch.equal(x.view(torch.int32), y.view(torch.int32))
