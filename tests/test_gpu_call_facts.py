"""rms_plan_info's facts of the last synthesis call are those of rms_synth, whatever the learned entry points launch on
the same plan in between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["bf16x3", "bf16"])
def test_learned_calls_leave_the_facts(path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    from paper_1810_06250_gb300 import learned as L
    rms.build()
    n, nchan = 500, 60
    q, u = torch.randn(2, n * nchan, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    i, c = (torch.full((n,), 70, dtype=torch.int32, device="cuda") for _ in range(2))
    a, p = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    with rms.Plan(np.linspace(120e6, 168e6, nchan), np.linspace(-60.0, 60.0, 101), path) as plan:
        net, win = L.Net(plan, hidden=32, max_batch=16, seed=1), L.Window(plan, 64)

        def facts():
            return [rms.rms_plan_info(plan.handle, k) for k in (rms.RMS_INFO_LAST_CTAS, rms.RMS_INFO_LAST_PAIR,
                                                                rms.RMS_INFO_LAST_PANELS, rms.RMS_INFO_LAST_KERNELS)]

        plan.synth(q, u, n, "los", None, i, a, p)
        want = facts()
        assert want[3] == 1                     # the one-kernel form
        rms.rms_synth_window(win.handle, q, u, n, "los", c, None, i, a, p)
        assert facts() == want
        rms.rms_peakmap_learned(win.handle, net.handle, q, u, n, "los", 2.0, p, a, i, None)
        assert facts() == want
        plan.sync()
        net.close()
        win.close()
