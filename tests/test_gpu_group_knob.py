"""RMS_GROUP_KBLOCKS: the K blocks of a partial sum are what the environment asks for, whatever the pipeline's stages hold.
Partials of 3 and of 4 of 12 K blocks add the same products up differently, so some of F's last bits differ; both are
within the gate of the FP64 oracle.  The knob is read once per process."""
import os
import subprocess
import sys

import numpy as np
import pytest

import gpu_helpers as gh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCRIPT = """
import sys
import numpy as np, torch
import paper_1810_06250_gb300 as rms
rng = np.random.default_rng(3)
n, nchan, phi = 200, 192, np.linspace(-60.0, 63.0, 40)       # 12 K blocks, tiles of 80 phase rows: two blocks a stage
q, u = (torch.from_numpy(rng.normal(size=(n, nchan)).astype(np.float32)).cuda() for _ in range(2))
F = torch.empty(n, len(phi), 2, device="cuda")
with rms.Plan(np.linspace(120e6, 168e6, nchan), phi, "bf16x3") as plan:
    plan.synth(q, u, n, "los", F)
    plan.sync()
np.save(sys.argv[1], F.cpu().numpy())
"""


def test_groups_are_what_the_knob_says(tmp_path, oracle_mod):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_06250_gb300 as rms
    rms.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    got = {}
    for g in (3, 4, 12):
        out = str(tmp_path / ("%d.npy" % g))
        subprocess.run([sys.executable, "-c", SCRIPT, out], check=True, cwd=root, timeout=300,
                       env=dict(os.environ, RMS_GROUP_KBLOCKS=str(g), PYTHONPATH=root))
        got[g] = np.load(out)
    rng = np.random.default_rng(3)
    Q, U = (rng.normal(size=(200, 192)).astype(np.float32) for _ in range(2))
    op = oracle_mod.plan(np.linspace(120e6, 168e6, 192), "freq", np.ones(192))
    Fo = oracle_mod.synth(Q, U, op, np.linspace(-60.0, 63.0, 40))
    scale = 2.5 * op.K * np.sqrt((Q.astype(np.float64) ** 2 + U.astype(np.float64) ** 2).sum(axis=1))
    for g, F in got.items():
        err = (np.abs(F[..., 0] + 1j * F[..., 1].astype(np.float64) - Fo).max(axis=1) / scale).max()
        assert err <= gh.TOL["bf16x3"], (g, err)
    for a, b in ((3, 4), (3, 12), (4, 12)):
        assert np.any(got[a] != got[b]), (a, b)
