"""The FP32 modes add up a target's pair terms over its threads in more than FP32, and contract the sums with the
target's own multipoles in FP64. Clusters of a central atom and seven others, each cluster out of the
others' range, and an Ewald parameter so small that the reciprocal part is exactly zero: then what the central
atom gets from each of the seven alone is one FP32 term (eight entries of a list go to eight threads), and
all seven together must give the sum of those terms to about 2^-45 of their magnitude (compensated FP32 pairs and
FP64; a plain FP32 sum is off by 2^-25 or so of it), or to the fixed mode's units of 2^-34 each. Where a cluster's
atoms lie in several blocks two of them can fall to one thread, whose share is an FP32 sum, so of many
clusters half are asked for. One cluster takes the quarter-block layout, 1,331 the whole-block one."""
import numpy as np
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

M, SPACING = 8, 24.0


def _clusters(m):
    """m^3 clusters: the central atom first, seven atoms around it at 2.5 to 4.5 A."""
    rng = np.random.default_rng(9)
    sites = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * SPACING
    d = rng.normal(size=(len(sites), M - 1, 3))
    d *= (rng.uniform(2.5, 4.5, (len(sites), M - 1)) / np.linalg.norm(d, axis=2))[..., None]
    xyz = np.concatenate([sites[:, None], sites[:, None] + d], 1).reshape(-1, 3)
    n = len(xyz)
    center = np.arange(n) % M == 0
    Q = rng.normal(0.0, 0.3, (n, 3, 3))
    Q = Q + Q.transpose(0, 2, 1)
    Q -= np.eye(3) * (np.trace(Q, axis1=1, axis2=2) / 3)[:, None, None]
    return synth.System(xyz, np.full(3, m * SPACING), np.where(center, rng.normal(size=n), 0.0),
                        rng.normal(0.0, 0.3, (n, 3)) * center[:, None], Q.reshape(n, 9)[:, [0, 1, 2, 4, 5, 8]] * center[:, None],
                        np.full(n, 1.1), np.tile(np.array([synth.FRAME_NONE, -1, -1], np.int32), (n, 1)),
                        np.zeros((0, 2), np.int32), np.arange(n, dtype=np.int32) // M, np.zeros(n, np.int32))


@pytest.mark.parametrize("precision", [binding.AP_MIXED, binding.AP_FIXED])
@pytest.mark.parametrize("m", [1, 11])
def test_sum_of_single_terms(m, precision):
    s = _clusters(m)
    c = binding.Context(s, cutoff=7.0, buffer=1.0, beta=1e-4, grid=(32, 32, 32), precision=precision)
    c.build()
    c.permanent_field()
    rng = np.random.default_rng(1)
    full = rng.normal(size=(s.n, 3))
    charges = rng.normal(size=s.n)
    which = np.arange(s.n) % M

    def run(active):
        """product, forces (dipoles on the active atoms) and field (charges on them) at the central atoms"""
        v = torch.tensor(full * np.isin(which, active)[:, None], device="cuda")
        out = torch.empty_like(v)
        c.matvec(v, out)
        _, f = c.energy_forces(v)
        mp = c.mpole.clone()
        c.mpole.zero_()
        c.mpole[:, 0] = torch.tensor(charges * np.isin(which, active), device="cuda")
        c.permanent_field()
        e = c.field.clone()
        c.mpole.copy_(mp)
        c.permanent_field()
        return [t.cpu().numpy()[::M].copy() for t in (out, f, e)]

    alone = [run([k]) for k in range(1, M)]
    together = run(list(range(1, M)))
    unit = 2.0 ** -34 if precision == binding.AP_FIXED else 0.0
    for q in range(3):
        terms = np.stack([a[q] for a in alone])
        off = np.abs(together[q] - terms.sum(0))
        ok = (off <= 2.0 ** -45 * np.abs(terms).sum(0) + M * unit).all(1)
        assert ok.mean() >= (1.0 if m == 1 else 0.5), (q, ok.mean(), off.max())
