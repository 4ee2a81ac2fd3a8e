"""RM-CLEAN's register kernel where its argmax search changes path: grid lengths around 32-sample rows and the
kernel's limit, exact ties, values outside the FP32 stand-in's range, NaN -- bit for bit against the FP64 oracle."""
import numpy as np
import pytest

from oracle import clean as oc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 31, 32, 33, 224, 401, 512, 513, 800, 1024, 1025])
def test_clean_edges(N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    rms.build()
    rng = np.random.default_rng(N)
    phi = np.linspace(-60.0, 60.0, N)
    dphi = phi[1] - phi[0]
    m = (np.arange(2 * N - 1) - (N - 1)) * dphi
    R2 = np.exp(-(m / (4 * dphi)) ** 2) * np.exp(0.3j * m / dphi)
    n = 12
    F = (rng.normal(size=(n, N)) + 1j * rng.normal(size=(n, N))).astype(np.complex64)
    F[1] = F[1, 0]                                  # every sample ties
    F[2, N // 2] = F[2, 0] = 9.0                    # two samples tie
    F[3, -1] = 9.0j
    F[3, 0] = -9.0                                  # equal modulus, other components
    F[4] *= np.float32(1e-22)                       # below the stand-in's range
    F[5] *= np.float32(1e19)                        # above it
    F[6] = 0.0
    F[7, N // 3] = np.nan
    F[8] = np.nan
    F[9, 0] = 3e38
    F[10] *= (1 + 3e-6 * rng.random(N)).astype(np.float32)
    F[10] /= np.abs(F[10]).astype(np.float32)       # moduli equal to a few units in the last place
    gain, thr, iters, fwhm = np.float32(0.2), np.float32(0.0), 15, 4.0 * dphi
    with rms.Plan(np.linspace(120e6, 168e6, 16), phi, "fp32_table") as plan:
        c = rms.rms_clean_create(plan.handle, fwhm, R2)
        Fd = torch.from_numpy(F.view(np.float32).reshape(n, N, 2)).cuda()
        out = [torch.full((n, N, 2), 5.0, device="cuda") for _ in range(3)]
        it = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        rms.rms_clean(c, Fd, n, float(gain), iters, float(thr), *out, it)
        torch.cuda.synchronize()
        rms.rms_clean_destroy(c)
    cl, res, comp = [o.cpu().numpy().view(np.complex64)[..., 0] for o in out]
    with np.errstate(all="ignore"):
        ocl, ores, ocomp, oit = oc.clean(F.astype(np.complex128), R2, float(gain), iters, float(thr), fwhm, dphi)
        ores, ocomp, ocl = (a.astype(np.complex64) for a in (ores, ocomp, ocl))
    np.testing.assert_array_equal(it.cpu().numpy(), oit)
    np.testing.assert_array_equal(res, ores)
    np.testing.assert_array_equal(comp, ocomp)
    # the restore adds in another order than the oracle's sum: FP64 rounding, seen after rounding to FP32
    ok = np.isfinite(ocl)
    np.testing.assert_array_equal(np.isfinite(cl), ok)
    scale = np.abs(np.where(ok, ocl, 0)).max(axis=1, keepdims=True)
    assert np.all(np.abs(np.where(ok, cl - np.where(ok, ocl, 0), 0)) <= 2e-7 * scale)
