"""Contexts of several host threads share the kernels. The product's kernel asks for as much shared memory as
its context's tuning says, and one context's launches must not take another's limit away: one thread tunes a
context over and over (which tries every setting), another applies the product of an untuned one meanwhile.
Both contexts have at most 304 blocks, so they launch the same kernel."""
import threading

import pytest

from paper_2011_01207_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tuning_beside_an_untuned_context():
    s = synth.water_box(216, 18.64, 1001)
    cs = []
    for _ in range(2):
        c = binding.Context(s, cutoff=7.0, buffer=2.0, beta=0.5446, grid=(24, 24, 24), stream=torch.cuda.Stream())
        torch.cuda.synchronize()
        c.build()
        c.permanent_field()
        torch.cuda.synchronize()
        cs.append(c)
    failed, done = [], threading.Event()

    def products():
        v = torch.ones((s.n, 3), dtype=torch.float64, device="cuda")
        out = torch.empty_like(v)
        torch.cuda.synchronize()
        try:
            while not done.is_set():
                for _ in range(50):
                    cs[1].matvec(v, out)
                cs[1].stream.synchronize()
        except binding.ApError as e:
            failed.append(e)

    t = threading.Thread(target=products)
    t.start()
    try:
        for _ in range(25):
            binding.ap_autotune(cs[0].ctx, reps=1)
    except binding.ApError as e:
        failed.append(e)
    finally:
        done.set()
        t.join()
    assert not failed, failed[0]
