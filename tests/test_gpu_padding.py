"""Small centred molecules of odd size. Positions are held relative to the centre of their block's box, so
the middle atom of such a molecule lies at the block's origin (or, moved by `off`, a rounding step beside
it), and the last atom shares a target pair with a padding slot. The padding half of a pair must stay zero
wherever the atoms lie, or its NaN reaches the solvers' dot products and the virial's sums.

The mixed and fixed modes against the FP64 mode (whose targets are single): fields, products and dipoles to
1e-5 RMS-relative and forces and the virial to 1e-4 (FP32 pair arithmetic; the solves stop at 1e-6 D, of
dipoles of about 0.2 D)."""
import numpy as np
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

T = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]) / np.sqrt(3.0)
AXES = np.concatenate([np.eye(3), -np.eye(3)])
CUBE = np.array([[a, b, c] for a in (-1, 1) for b in (-1, 1) for c in (-1, 1)], float)
# central atom first
MOLECULES = {"CH4": 1.09 * T, "CO2": 1.16 * np.array([[0.0, 0, 1], [0, 0, -1]]), "SF6": 1.56 * AXES, "bcc": 1.7 * CUBE}


def _system(name, off):
    rng = np.random.default_rng(3)
    arms = MOLECULES[name]
    n = len(arms) + 1
    xyz = np.concatenate([np.full((1, 3), off), arms]) + 12.0
    q = rng.normal(0.0, 0.3, n)
    Q = rng.normal(0.0, 0.1, (n, 3, 3))
    Q = Q + Q.transpose(0, 2, 1)
    Q -= np.eye(3) * (np.trace(Q, axis1=1, axis2=2) / 3)[:, None, None]
    # the bonds to the central atom are excluded
    excl = np.stack([np.zeros(n - 1), np.arange(1, n)], 1).astype(np.int32)
    return synth.System(xyz, np.full(3, 24.0), q - q.mean(), rng.normal(0.0, 0.1, (n, 3)),
                        Q.reshape(n, 9)[:, [0, 1, 2, 4, 5, 8]], np.full(n, 0.8),
                        np.tile(np.array([synth.FRAME_NONE, -1, -1], np.int32), (n, 1)), excl, np.zeros(n, np.int32),
                        np.zeros(n, np.int32))


def _outputs(s, precision):
    c = binding.Context(s, cutoff=7.0, buffer=1.0, beta=0.5446, grid=(24, 24, 24), precision=precision)
    pairs = s.excl
    c.set_scaled_pairs(pairs, np.tile([0.0, 0.5], (len(pairs), 1)))
    c.build()
    c.permanent_field()
    out = {"field": c.field.clone()}
    v = torch.tensor(0.1 * np.random.default_rng(5).normal(size=(s.n, 3)), device="cuda")
    t = torch.empty_like(v)
    c.matvec(v, t)
    out["product"] = t
    c.solve(tol=1e-6)
    out["pcg"] = c.mu.clone()
    _, f = c.energy_forces(v)
    out["forces"] = f.clone()
    _, f, w = c.energy_forces(v, virial=True)
    out["forces with virial"], out["virial"] = f.clone(), w.clone()
    c.solve_diis(tol=1e-6)
    out["diis"] = c.mu.clone()
    c.permanent_field_dp()
    c.solve_dp(tol=1e-6)
    out["mu_d"], out["mu_p"] = c.mu_d.clone(), c.mu_p.clone()
    _, f, w = c.energy_forces_dp(v, 1.1 * v, virial=True)
    out["two-set forces"], out["two-set virial"] = f.clone(), w.clone()
    return out


@pytest.mark.parametrize("off", [0.0, 1e-7, 1e-6])
@pytest.mark.parametrize("name", sorted(MOLECULES))
def test_centred_molecule(name, off):
    s = _system(name, off)
    ref = _outputs(s, binding.AP_FP64)
    for precision in (binding.AP_MIXED, binding.AP_FIXED):
        for k, got in _outputs(s, precision).items():
            tol = 1e-4 if "forces" in k or "virial" in k else 1e-5
            assert (torch.linalg.norm(got - ref[k]) / torch.linalg.norm(ref[k])).item() < tol, k
