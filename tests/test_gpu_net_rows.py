"""Proposals do not depend on how many rows a call has: the 32-row tiles and narrow output tiles of small calls give the
same bits as the thread-per-row split and whole output tiles of a large one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# rows of whole and partial 16-byte pieces, one K block and several, data off 16 bytes; hidden layers of one and two
# narrow tiles, whole and ragged
@pytest.mark.parametrize("nchan,hidden,shift", [(16, 256, 0), (45, 144, 0), (60, 256, 1), (128, 64, 0)])
@pytest.mark.parametrize("layout", ["los", "chan"])
def test_rows_of_a_small_call(layout, nchan, hidden, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    rng = np.random.default_rng(nchan)
    freq = np.linspace(120e6, 168e6, nchan)
    w = np.ones(nchan)
    w[[3, 7]] = 0.0
    n_all = 200 * torch.cuda.get_device_properties(0).multi_processor_count + 1      # beyond the small calls' rule
    X = torch.randn(2, n_all, nchan, device="cuda", generator=torch.Generator("cuda").manual_seed(nchan))
    X[:, :, 3] = float("nan")                            # a flagged channel
    X[0, 5] = 0.0
    X[1, 5] = 0.0                                        # an empty row
    X[0, 6, 9] = float("nan")

    def propose(net, n):
        buf = torch.empty(2, n * nchan + 4, device="cuda")
        q, u = (buf[k, shift:shift + n * nchan] for k in range(2))
        for k, t in enumerate((q, u)):
            t.copy_((X[k, :n].t().contiguous() if layout == "chan" else X[k, :n]).reshape(-1))
        z = torch.empty(n, 101, device="cuda")
        b = torch.empty(n, dtype=torch.int32, device="cuda")
        c = torch.empty(n, device="cuda")
        rms.rms_propose(net.handle, q, u, n, layout, 3, z, b, c)
        return z, b, c

    with rms.Plan(freq, np.linspace(-60, 60, 101), "bf16x3", weights=w) as plan:
        net = L.Net(plan, hidden=hidden, max_batch=64, seed=3)
        want = propose(net, n_all)
        for n in (1, 31, 33, 127, 129, 1000):
            got = propose(net, n)
            plan.sync()
            for a, b in zip(got, want):
                assert torch.equal(a.view(torch.int32), b[:n].view(torch.int32)), n
        net.close()
