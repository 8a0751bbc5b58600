"""The FP32 modes' own transforms: grid sizes of every register transform, odd and unequal sides, an odd
number of rows (the last row of a plane has no partner), both sides of the size rule, and sides
with factors it does not take (the library's transforms). Against the FP64 mode on the same grid, whose
transforms are always the library's: fields to 1e-5, forces and virial to 1e-4 (FP32 arithmetic, as in
the parity tests; FP32 transforms add about 1e-6)."""
import numpy as np
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [(24, 24, 24), (25, 27, 30), (32, 21, 28), (27, 45, 20), (36, 49, 35), (50, 42, 54),
         (64, 64, 65), (63, 81, 60), (96, 96, 96), (96, 96, 98), (22, 26, 34), (24, 25, 26)]


def _rel(a, b):
    return (torch.sqrt(torch.mean((a - b) ** 2) / torch.mean(b ** 2))).item()


@pytest.mark.parametrize("prec", [binding.AP_MIXED, binding.AP_FIXED])
@pytest.mark.parametrize("grid", GRIDS)
def test_against_fp64(grid, prec):
    s = synth.water_box(216, 18.643, seed=9)
    mu = 0.08 * np.random.default_rng(3).normal(size=(s.n, 3)) * s.alpha[:, None]
    t = torch.tensor(mu, device="cuda")
    res = []
    for p in (binding.AP_FP64, prec):
        # a broad Gaussian, so that the reciprocal part carries its weight of the field
        c = binding.Context(s, cutoff=7.0, buffer=1.0, beta=0.5446, grid=grid, precision=p)
        c.build()
        c.permanent_field()
        out = torch.empty_like(t)
        c.matvec(t, out)
        _, f0 = c.energy_forces(t)
        f0 = f0.clone()
        _, f, v = c.energy_forces(t, virial=True)
        res.append((c.field.clone(), out, f.clone(), v.clone(), f0))
    ref, got = res
    assert _rel(got[0], ref[0]) < 1e-5
    assert _rel(got[1], ref[1]) < 1e-5
    assert _rel(got[2], ref[2]) < 1e-4
    assert _rel(got[3], ref[3]) < 1e-4
    assert _rel(got[4], got[2]) < 1e-5
