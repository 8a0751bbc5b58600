"""The device memory that a build takes for its pair lists and candidates, per ordered block pair: at most 1,702
bytes of lists and an eighth more, 32 of the block pair itself and a quarter more, and 128 of an exclusion mask for the pairs
that have one and a quarter more (and granularity)."""
import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_bytes_per_block_pair():
    s = synth.water_box(8000, 62.2, 5)
    c = binding.Context(s, cutoff=7.0, buffer=2.0, beta=0.5446, grid=(64, 64, 64))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    c.build()
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    blocks, pairs, excl = c.stats()
    ordered = 2 * pairs - blocks
    bound = ordered * (1702 * 1.125 + 32 * 1.25) + 2 * excl * 128 * 1.25 + 512 * blocks + (16 << 20)
    assert used < bound, (used, bound, used / ordered)
