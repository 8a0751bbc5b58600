"""The gathers (field, and derivatives for the forces) where their forms change: rows of a multiple of four
points (wide loads) and not, rows whose stencils wrap in each place of a group of four, and the last size
with five threads per atom and the first with one on a GPU of 152 SMs. The mixed mode against the FP64 mode,
whose gathers have no wide form: fields to 1e-5, forces to 1e-4 RMS-relative (FP32 arithmetic)."""
import numpy as np
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mols,grid", [(64, (20, 18, 18)), (216, (20, 20, 20)), (216, (21, 20, 20)), (216, (22, 20, 20)),
                                       (216, (23, 20, 20)), (20753, (84, 84, 84)), (20753, (86, 84, 84)),
                                       (20754, (84, 84, 84)), (20754, (86, 84, 84))])
def test_against_fp64(mols, grid):
    s = synth.water_box(mols, max(18.0, 3.107 * mols ** (1 / 3)), seed=6)
    mu = 0.08 * np.random.default_rng(2).normal(size=(s.n, 3)) * s.alpha[:, None]
    t = torch.tensor(mu, device="cuda")
    res = []
    for p in (binding.AP_FP64, binding.AP_MIXED):
        c = binding.Context(s, cutoff=7.0, buffer=1.0, beta=0.5446, grid=grid, precision=p)
        c.build()
        c.permanent_field()
        out = torch.empty_like(t)
        c.matvec(t, out)
        _, f = c.energy_forces(t)
        res.append((c.field.clone(), out, f.clone()))
    for a, b, tol in zip(res[1], res[0], (1e-5, 1e-5, 1e-4)):
        assert (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item() < tol
