"""The one-kernel vector work of small solves at the edges of its shapes: part of one block's threads, one CTA
and the first of two, a full cluster at one, two and four slots per thread, and the first size that the
separate kernels take. Against the FP64 mode's solve of the same system (separate kernels): the
dipoles to 1e-5 RMS-relative (FP32 vectors and pair arithmetic), the same iteration count to one (both stop on
the same measure), and the fixed mode twice to the bit."""
import numpy as np
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# waters -> slots (rounded up to 32 atoms)
MOLS = [64, 170, 171, 1365, 1366, 2730, 2731, 5461, 5462]


@pytest.mark.parametrize("mols", MOLS)
def test_against_fp64(mols):
    s = synth.water_box(mols, max(16.2, 3.107 * mols ** (1 / 3)), seed=4)
    grid = tuple(2 * int(np.ceil(L / 2)) for L in s.box)
    res = {}
    for p in (binding.AP_FP64, binding.AP_MIXED, binding.AP_FIXED):
        c = binding.Context(s, cutoff=7.0, buffer=1.0, beta=0.5446, grid=grid, precision=p)
        c.build()
        c.permanent_field()
        info = c.solve(tol=1e-6)
        res[p] = c.mu.clone(), info.iterations
        if p == binding.AP_FIXED:
            c.solve(tol=1e-6)
            assert torch.equal(c.mu, res[p][0])
    ref, it = res[binding.AP_FP64]
    for p in (binding.AP_MIXED, binding.AP_FIXED):
        mu, n = res[p]
        assert (torch.linalg.norm(mu - ref) / torch.linalg.norm(ref)).item() < 1e-5
        assert abs(n - it) <= 1
