"""FP32 CUDA-core contraction: its copying warps' pipeline at the edges, against the FP64 oracle.

The gates are those of the precisions (gpu_helpers.TOL).
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


# fewer and more 16-channel chunks than the four stages, whole and partial; a block of 256 LOS whole, short by one,
# one over; rows on and off 16 bytes; folded and general grids of one and several phi tiles
@pytest.mark.parametrize("nchan,flagged", [(1, 0), (16, 0), (65, 3), (150, 9)])
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("path", ["fp32_table", "fp32_fly"])
def test_simt_pipeline_edges(rms, oracle_mod, path, sym, nchan, flagged):
    rng = np.random.default_rng(nchan)
    freq = np.linspace(120e6, 168e6, nchan) if nchan > 1 else np.array([150e6])
    w = rng.uniform(0.5, 1.5, nchan)
    w[rng.choice(nchan, flagged, replace=False)] = 0.0
    op = oracle_mod.plan(freq, "freq", w)
    for nphi, nlos, layout, shift in ((141, 255, "chan", 0), (141, 256, "los", 0), (20, 513, "chan", 1),
                                      (141, 260, "chan", 0), (70, 259, "los", 1), (141, 512, "chan", 1)):
        phi = np.linspace(-60.0, 60.0 if sym else 63.0, nphi)
        data = torch.randn(2, nlos * nchan + 4, device="cuda", generator=torch.Generator("cuda").manual_seed(nlos))
        q, u = (data[i, shift:shift + nlos * nchan] for i in range(2))
        shape = (nchan, nlos) if layout == "chan" else (nlos, nchan)
        Q, U = (x.cpu().numpy().reshape(shape) for x in (q, u))
        if layout == "chan":
            Q, U = Q.T, U.T
        with rms.Plan(freq, phi, path, weights=w) as plan:
            F = torch.empty(nlos, nphi, 2, device="cuda")
            pi = torch.full((nlos,), -7, dtype=torch.int32, device="cuda")
            pa, pp = torch.zeros(nlos, device="cuda"), torch.zeros(nlos, device="cuda")
            plan.synth(q, u, nlos, layout, F, pi, pa, pp)
            plan.sync()
        Fh = F.cpu().numpy()
        per, _ = gh.errors(Fh[..., 0] + 1j * Fh[..., 1], oracle_mod.synth(Q, U, op, phi))
        assert per.max() <= gh.TOL[path], (nphi, nlos, layout, per.max())
        gh.check_peaks_self(Fh, pi.cpu().numpy(), pa.cpu().numpy(), pp.cpu().numpy(), phi)


# a few LOS more than one block per SM, and 1.5 to 3.1 blocks per SM with a ragged last one; one, two and several phi
# tiles, with a whole and a partial last one
@pytest.mark.parametrize("per_sm,extra,layout", [(1.0, 1, "chan"), (1.5, 77, "los"), (3.1, 130, "chan")])
@pytest.mark.parametrize("nphi", [20, 64, 128, 141, 211])
@pytest.mark.parametrize("path,sym", [("fp32_table", True), ("fp32_table", False), ("fp32_fly", True)])
def test_simt_balanced_runs(rms, path, sym, nphi, per_sm, extra, layout):
    """The same bits as calls of at most one block per SM, whose blocks are each one CTA's or one cluster's."""
    nchan = 20
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    nlos = int(256 * nsm * per_sm) + extra
    freq = np.linspace(120e6, 168e6, nchan)
    phi = np.linspace(-60.0, 60.0 if sym else 63.0, nphi)
    X = torch.randn(2, nlos, nchan, device="cuda", generator=torch.Generator("cuda").manual_seed(nphi))
    X[:, 7] = 0.0
    X[0, 300, 2] = float("nan")

    def synth(plan, a, b):
        n = b - a
        q, u = ((X[i, a:b].t() if layout == "chan" else X[i, a:b]).contiguous() for i in range(2))
        F = torch.empty(n, nphi, 2, device="cuda")
        out = [torch.full((n,), -7, dtype=torch.int32, device="cuda")] + [torch.zeros(n, device="cuda") for _ in range(2)]
        plan.synth(q, u, n, layout, F, *out)
        return [F] + out

    with rms.Plan(freq, phi, path) as plan:
        got = [synth(plan, 0, nlos) for _ in range(2)]
        step = 256 * nsm
        parts = [synth(plan, a, min(a + step, nlos)) for a in range(0, nlos, step)]
        plan.sync()
    for k in range(4):
        want = torch.cat([p[k] for p in parts]).view(torch.int32)
        for g in got:
            assert torch.equal(g[k].view(torch.int32), want), k


def test_simt_two_threads_one_plan(rms):
    """Calls that share blocks between CTAs, on one plan from two host threads and streams: the plan orders them."""
    import threading
    nchan, nphi = 12, 64
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    nlos = 256 * nsm + 256 * 40
    X = torch.randn(2, 2, nchan, nlos, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    out = [[[torch.empty(nlos, dtype=torch.int32, device="cuda"), torch.empty(nlos, device="cuda")] for _ in range(20)] for _ in range(2)]
    with rms.Plan(np.linspace(120e6, 168e6, nchan), np.linspace(-60.0, 60.0, nphi), "fp32_table") as plan:
        want = []
        for t in range(2):
            want.append([torch.empty(nlos, dtype=torch.int32, device="cuda"), torch.empty(nlos, device="cuda")])
            plan.synth(X[t, 0], X[t, 1], nlos, "chan", None, *want[t])
        torch.cuda.synchronize()

        def work(t):
            s = torch.cuda.Stream()
            for i, a in out[t]:
                plan.synth(X[t, 0], X[t, 1], nlos, "chan", None, i, a, stream=s)
            s.synchronize()

        threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        plan.sync()
    for t in range(2):
        for i, a in out[t]:
            assert torch.equal(i, want[t][0]) and torch.equal(a, want[t][1])
