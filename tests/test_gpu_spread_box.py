"""The dipole spread through shared-memory boxes at the edges of its rule, on a GPU of 152 SMs: the last block
count below it and the first one on it (ragged and whole last blocks), rows that are no multiple of four points, a
grid too fine for the boxes, unequal sides, and a box with an empty slab, whose blocks that straddle it
do not fit. The mixed mode's product against the FP64 mode's (always the direct spread): 1e-5
RMS-relative (FP32 arithmetic, as in the parity tests)."""
import numpy as np
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _water(dims, mols, seed, slab=0.0, cell=3.107):
    """mols waters (0: all) on a dims lattice, random orientations, none in a slab across the middle of x."""
    rng = np.random.default_rng(seed)
    box = np.array(dims, float) * cell
    sites = np.stack(np.meshgrid(*[(np.arange(d) + 0.5) * cell for d in dims], indexing="ij"), -1).reshape(-1, 3)
    sites = sites[np.abs(sites[:, 0] / box[0] - 0.5) >= 0.5 * slab]
    if mols:
        sites = sites[np.sort(rng.choice(len(sites), mols, replace=False))]
    mols = len(sites)
    xyz = synth._orient_waters(rng, sites, box, 1.7)
    q, dip, quad, alpha, frame, excl = synth._water_arrays(xyz, 0)
    return synth.System(xyz, box, q, dip, quad, alpha, frame, excl, np.repeat(np.arange(mols), 3).astype(np.int32),
                        np.ones(3 * mols, np.int32))


# lattice, waters, grid, share of x left empty
CASES = {
    "direct_last": ((19, 19, 19), 6474, (60, 60, 60), 0.0),     # 607 blocks
    "boxes_first": ((19, 19, 19), 6485, (60, 60, 60), 0.0),     # 608 blocks, the last ragged
    "whole_last": ((19, 19, 19), 6496, (60, 60, 60), 0.0),      # 609 whole blocks
    "row_not_of_four": ((19, 19, 19), 6496, (58, 60, 60), 0.0),
    "fine_grid": ((19, 19, 19), 6496, (92, 92, 92), 0.0),
    "unequal": ((24, 18, 16), 0, (76, 50, 50), 0.0),
    "empty_slab": ((30, 18, 18), 0, (80, 48, 48), 0.3),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_against_fp64(name):
    dims, mols, grid, slab = CASES[name]
    s = _water(dims, mols, 8, slab)
    t = torch.tensor(0.08 * np.random.default_rng(2).normal(size=(s.n, 3)) * s.alpha[:, None], device="cuda")
    out = []
    for p in (binding.AP_FP64, binding.AP_MIXED, binding.AP_FIXED):   # the fixed mode never takes the boxes
        c = binding.Context(s, cutoff=7.0, buffer=1.0, beta=0.5446, grid=grid, precision=p)
        c.build()
        c.permanent_field()
        o = torch.empty_like(t)
        c.matvec(t, o)
        out.append(o)
        if p == binding.AP_FIXED:
            again = torch.empty_like(t)
            c.matvec(t, again)
            assert torch.equal(o, again)
    for o in out[1:]:
        assert (torch.linalg.norm(o - out[0]) / torch.linalg.norm(out[0])).item() < 1e-5
