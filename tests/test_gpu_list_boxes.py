"""Large systems' pair lists drop whole blocks by the blocks' present boxes first, from eight blocks an SM on (1,216
on 152 SMs). Atoms that have moved since the lists' build must be found all the same: a context whose lists were
built before the atoms moved (smoothly, by up to half the buffer) against one built after, whose blocks are others.
The pairs are the same, so FP64 to 1e-9 (the order of the sums), the mixed mode to 1e-5 RMS-relative."""
import numpy as np
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _water(dims, mols, seed, cell=3.107):
    rng = np.random.default_rng(seed)
    sites = np.stack(np.meshgrid(*[(np.arange(d) + 0.5) * cell for d in dims], indexing="ij"), -1).reshape(-1, 3)
    sites = sites[np.sort(rng.choice(len(sites), mols, replace=False))]
    box = np.array(dims, float) * cell
    xyz = synth._orient_waters(rng, sites, box, 1.7)
    q, dip, quad, alpha, frame, excl = synth._water_arrays(xyz, 0)
    return synth.System(xyz, box, q, dip, quad, alpha, frame, excl, np.repeat(np.arange(mols), 3).astype(np.int32),
                        np.ones(3 * mols, np.int32))


# 1,215, 1,216 and 1,217 blocks, the last ragged
@pytest.mark.parametrize("mols", [12957, 12970, 12974])
@pytest.mark.parametrize("precision,tol", [(binding.AP_MIXED, 1e-5), (binding.AP_FP64, 1e-9)])
def test_moved_atoms(mols, precision, tol):
    s = _water((19, 24, 31), mols, 3)
    grid = tuple(2 * int(np.ceil(L / 2)) for L in s.box)
    w = 2 * np.pi * s.xyz / s.box
    moved = s.xyz + np.stack([np.sin(w[:, 1] + w[:, 2]), np.cos(w[:, 2] - w[:, 0]), np.sin(w[:, 0])], 1) / np.sqrt(3.0)
    res = []
    for first in (s.xyz, moved):
        c = binding.Context(s, cutoff=7.0, buffer=2.0, beta=0.5446, grid=grid, precision=precision)
        c.set_positions(first)
        c.build()
        c.set_positions(moved)
        c.permanent_field()
        v = torch.tensor(0.1 * np.random.default_rng(5).normal(size=(s.n, 3)), device="cuda")
        t = torch.empty_like(v)
        c.matvec(v, t)
        res.append((c.field.clone(), t))
    for a, b in zip(*res):
        assert (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item() < tol
