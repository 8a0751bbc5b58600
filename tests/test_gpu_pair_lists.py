"""Pair lists and the kernels that walk them, where their shapes change: ragged last blocks and
odd atoms, the quarter-block layout's last size and the first of the whole-block one, candidate
sets of more than one shared-memory chunk, and boxes so short along one, two or three dimensions that an
atom is in range of a block in two images. Against the FP64 oracle on the same grid: FP64 to 1e-9
(rounding), the mixed mode to 1e-5 (FP32 pair arithmetic), forces to 1e-8 and 1e-4; the mixed
mode's errors are RMS-relative, as in the parity tests."""
import numpy as np
import pytest

from oracle import Oracle, Params
from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _water(dims, mols, seed, cell=3.107):
    """mols waters on a dims lattice in its (non-cubic) box, random orientations."""
    rng = np.random.default_rng(seed)
    sites = np.stack(np.meshgrid(*[(np.arange(d) + 0.5) * cell for d in dims], indexing="ij"), -1).reshape(-1, 3)
    sites = sites[np.sort(rng.choice(len(sites), mols, replace=False))]
    box = np.array(dims, float) * cell
    xyz = synth._orient_waters(rng, sites, box, 1.7)
    q, dip, quad, alpha, frame, excl = synth._water_arrays(xyz, 0)
    return synth.System(xyz, box, q, dip, quad, alpha, frame, excl, np.repeat(np.arange(mols), 3).astype(np.int32),
                        np.ones(3 * mols, np.int32))


# name: lattice, waters, cutoff, buffer
CASES = {
    "short_in_three": ((6, 6, 6), 211, 7.0, 2.0),        # 633 atoms: ragged, every box edge short
    "short_in_two": ((6, 7, 16), 640, 7.0, 2.0),
    "short_in_one": ((6, 15, 15), 1300, 7.0, 2.0),
    "quarter_blocks_last": ((15, 15, 15), 3242, 7.0, 2.0),   # 9,726 atoms: 304 blocks
    "whole_blocks_first": ((15, 15, 15), 3243, 7.0, 2.0),    # 9,729 atoms: 305 blocks, one atom in the last
    "two_chunks": ((15, 15, 15), 3300, 10.5, 1.0),           # about 1,150 candidates a block
}


def _rel(a, b):
    return np.sqrt(np.mean((a - b) ** 2) / np.mean(b ** 2))


@pytest.mark.parametrize("prec,tol_field,tol_force", [(binding.AP_FP64, 1e-9, 1e-8), (binding.AP_MIXED, 1e-5, 1e-4)])
@pytest.mark.parametrize("name", sorted(CASES))
def test_against_oracle(name, prec, tol_field, tol_force):
    dims, mols, rc, buf = CASES[name]
    s = _water(dims, mols, 11)
    grid = tuple(2 * int(np.ceil(L / 2)) for L in s.box)
    c = binding.Context(s, cutoff=rc, buffer=buf, beta=0.5446, grid=grid, precision=prec)
    c.build()
    c.permanent_field()
    o = Oracle(s, Params(beta=0.5446, grid=grid, cutoff=rc))
    assert _rel(c.field.cpu().numpy(), o.permanent_field()) < tol_field
    mu = 0.08 * np.random.default_rng(5).normal(size=(s.n, 3)) * s.alpha[:, None]
    t = torch.tensor(mu, device="cuda")
    out = torch.empty_like(t)
    c.matvec(t, out)
    assert _rel(out.cpu().numpy(), o.apply_T(mu)) < tol_field
    _, f, v = c.energy_forces(t, virial=True)
    f = f.clone()
    assert _rel(f.cpu().numpy(), o.forces(mu)) < tol_force
    assert _rel(v.cpu().numpy(), o.virial(mu)) < tol_force
    _, f2 = c.energy_forces(t)
    assert _rel(f2.cpu().numpy(), f.cpu().numpy()) < tol_field
