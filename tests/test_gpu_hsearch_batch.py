"""The h search from a poor h in a batch that mixes instances of 100,000 particles
and more, whose searches go on 32 particles together, with smaller ones, whose
searches go on one warp a particle: each instance gives the bits it gives alone."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FIELDS = ("x", "y", "z", "vx", "vy", "vz", "h", "u", "rho", "p", "c", "ax", "ay", "az", "du", "nnb")


@pytest.mark.parametrize("precision,factor", [(0, 0.7), (0, 1.4), (1, 0.7)])
def test_large_and_small_instances(precision, factor):
    from paper_1809_08013_gb300 import binding as B
    insts = [ics.square_patch(47, seed=1), ics.evrard(3000, seed=2), ics.evrard(100000, seed=3),
             ics.square_patch(20, seed=4), ics.evrard(99999, seed=5)]
    for s, p in insts:
        p.precision = precision
        s["h"] = s["h"] * factor
    counts = [len(s["x"]) for s, _ in insts]
    state = {f: np.concatenate([s[f] for s, _ in insts]) for f in ics.FIELDS}
    ctx = B.Context(sum(counts), max_instances=len(insts))
    arr = B.alloc_arrays(state, ninst=len(insts))
    ctx.batch_set(counts, [p for _, p in insts])
    ctx.batch_step(arr, nsteps=1)
    ctx.sync()
    off = np.concatenate([[0], np.cumsum(counts)])
    for k, (s, p) in enumerate(insts):
        one = B.Context(counts[k])
        a = B.alloc_arrays(s)
        one.step(p, a, nsteps=1)
        one.sync()
        for f in FIELDS:
            got = arr[f][off[k]:off[k + 1]].cpu().numpy()
            assert np.array_equal(got.view(np.uint8), a[f].cpu().numpy().view(np.uint8)), (k, f)
        one.close()
    ctx.close()
