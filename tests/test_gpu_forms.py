"""Which form a synthesis call took, as rms_plan_info reports it: on symmetric grids one kernel (behind FP16X3's exponents)
wherever the plan and the call allow it, else layout stage, contraction and, after single-tile jobs, the peak merge.
The shapes are those whose two forms other tests compare bit by bit, so that those comparisons have two sides."""
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


def facts(rms, plan):
    return tuple(rms.rms_plan_info(plan.handle, k) for k in (rms.RMS_INFO_LAST_KERNELS, rms.RMS_INFO_LAST_PAIR,
                                                             rms.RMS_INFO_LAST_PANELS))


# (channels, flagged, lines of sight, depths); the split precisions' one-kernel form takes up to 512 active channels
@pytest.mark.parametrize("nchan,flagged,nlos,nphi", [(75, 7, 20011, 103), (75, 7, 29500, 515), (128, 0, 1, 101),
                                                     (310, 5, 4001, 101), (512, 0, 4096, 101), (540, 8, 4096, 101),
                                                     (600, 7, 19999, 33)])
@pytest.mark.parametrize("layout", ["chan", "los"])
@pytest.mark.parametrize("path", ["bf16x3", "fp16x3", "bf16"])
def test_form_of_a_call(rms, path, layout, nchan, flagged, nlos, nphi):
    w = np.ones(nchan)
    w[:flagged] = 0.0
    q, u = torch.randn(2, nlos * nchan, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    pi = torch.empty(nlos, dtype=torch.int32, device="cuda")
    F = torch.empty(nlos, nphi, 2, device="cuda")
    fp16 = path == "fp16x3"
    one = path == "bf16" or nchan - flagged <= 512
    with rms.Plan(np.linspace(120e6, 168e6, nchan), np.linspace(-60.0, 60.0, nphi), path, weights=w) as plan:
        plan.synth(q, u, nlos, layout, F, pi)
        k, pair, panels = facts(rms, plan)
        assert (k == 1 + fp16 and pair == 1 and panels == 0) if one else k == 3 + fp16
        rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_CONTRACTION, rms.RMS_CONTRACT_PAIR)
        plan.synth(q, u, nlos, layout, F, pi)
        k, pair, panels = facts(rms, plan)
        assert k == 3 + fp16 and pair == 1 and panels > 0
        rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_SCHEDULE, rms.RMS_SCHEDULE_WHOLE)
        plan.synth(q, u, nlos, layout, F, pi)
        assert facts(rms, plan) == (2 + fp16, 1, 0)
        plan.sync()
    # a grid without symmetry: FP16X3 finds its exponents inside the split
    with rms.Plan(np.linspace(120e6, 168e6, nchan), np.linspace(-60.0, 63.0, nphi), path, weights=w) as plan:
        rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_SCHEDULE, rms.RMS_SCHEDULE_WHOLE)
        plan.synth(q, u, nlos, layout, F, pi)
        assert facts(rms, plan)[0] == 2
        plan.sync()
