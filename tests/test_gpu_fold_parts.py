"""One item per CTA pair: the one-kernel form releases an item's K blocks in parts; the same bits as two kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 4 K blocks (one part), 5 (a part of one), 10 (three parts), 16 (four), 17 (parts of eight); a single ragged item, several;
# rows on and off 16 bytes
@pytest.mark.parametrize("nchan", [128, 150, 310, 512, 540])
@pytest.mark.parametrize("nlos,shift", [(1, 0), (130, 1), (4001, 0), (4096, 0)])
@pytest.mark.parametrize("layout", ["chan", "los"])
@pytest.mark.parametrize("path", ["bf16x3", "fp16x3", "bf16"])
def test_parts_match_two_kernels(path, layout, nlos, shift, nchan):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    rms.build()
    nphi = 101
    freq = np.linspace(120e6, 168e6, nchan)
    w = np.ones(nchan)
    if nchan in (310, 540):
        w[::70] = 0.0
    data = torch.randn(2, nlos * nchan + 4, device="cuda", generator=torch.Generator("cuda").manual_seed(nchan))
    data[0, nchan // 2] = float("nan")
    q, u = (data[i, shift:shift + nlos * nchan] for i in range(2))
    got = []
    with rms.Plan(freq, np.linspace(-60.0, 60.0, nphi), path, weights=w) as plan:
        for kind in (rms.RMS_CONTRACT_AUTO, rms.RMS_CONTRACT_PAIR):
            rms.rms_plan_set_option(plan.handle, rms.RMS_OPT_CONTRACTION, kind)
            F = torch.full((nlos, nphi, 2), 3.0, device="cuda")
            i = torch.full((nlos,), -7, dtype=torch.int32, device="cuda")
            a, p = torch.zeros(nlos, device="cuda"), torch.zeros(nlos, device="cuda")
            plan.synth(q, u, nlos, layout, F, i, a, p)
            plan.sync()
            got.append((F, i, a, p))
    for x, y in zip(*got):
        assert torch.equal(x.view(torch.int32), y.view(torch.int32))
