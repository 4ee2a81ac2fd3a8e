"""A plan keeps what its calls read: on a grid symmetric about zero the folded phase matrix, a quarter of the general one,
takes that one's place (FP16X3 keeps both: its no-allocation call evaluates every depth by itself), and rms_plan_get still
gives the general matrix."""
import numpy as np
import pytest

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


def test_folded_plan_is_smaller(rms):
    nchan, nphi = 1024, 6001
    freq = np.linspace(120e6, 168e6, nchan)
    torch.zeros(1, device="cuda")

    def device_bytes(top):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        with rms.Plan(freq, np.linspace(-60.0, top, nphi), "bf16x3"):
            return free - torch.cuda.mem_get_info()[0]

    device_bytes(60.0)                              # (kernels loaded on first use)
    general = 2 * (2 * nphi) * (2 * nchan) * 2      # hi and lo parts, 2 bytes an element
    sym, asym = device_bytes(60.0), device_bytes(63.0)
    assert sym <= asym - general // 2, (sym, asym, general)


@pytest.mark.parametrize("flagged", [0, 9])
def test_general_matrix_of_a_folded_plan(rms, oracle_mod, flagged):
    nchan, nphi = 75, 41
    freq = np.linspace(120e6, 168e6, nchan)
    w = np.random.default_rng(2).uniform(0.5, 1.5, nchan)
    w[:flagged] = 0.0
    phi = np.linspace(-60.0, 60.0, nphi)
    op = oracle_mod.plan(freq, "freq", w)
    act = op.active
    with rms.Plan(freq, phi, "bf16x3", weights=w) as plan:
        hi, lo = ((plan.get(k).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
                  for k in (rms.RMS_GET_B_HI, rms.RMS_GET_B_LO))
    th = 2.0 * phi[:, None] * (op.lambda2[act] - op.lambda0sq)[None, :]
    wn = w[act] / w.max()
    B, n, k = hi + lo, 2 * nphi, 2 * len(act)
    for r, c, want in ((0, 0, np.cos(th)), (0, 1, np.sin(th)), (1, 0, -np.sin(th)), (1, 1, np.cos(th))):
        np.testing.assert_allclose(B[r:n:2, c:k:2], wn * want, rtol=0, atol=2.0 ** -16)
    assert not B[n:, :].any() and not B[:, k:].any()
