"""The first count of the h search (k_h_count) over its block widths: a group
of 32 particles is served by 8, 4, 2 or 1 warps, fewer the larger the batch.
The rows do not depend on the width, so an instance gives the same bits alone
(8 to 1 warps) and in a batch large enough for one warp per group; and h and
the neighbour sets of every width are the oracle's."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics
from test_gpu_rows import _steep_sphere

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FIELDS = ("x", "y", "z", "vx", "vy", "vz", "h", "u", "rho", "p", "c", "ax", "ay", "az", "du", "nnb")


def _insts():
    out = [ics.evrard(5000, seed=1), _steep_sphere(3.0)]
    for side, seed in ((13, 2), (27, 3), (33, 4), (41, 5)):  # 8, 4, 2 and 1 warps alone
        s, p = ics.square_patch(side, seed=seed)
        out.append((ics.random_velocities(s, seed=seed, scale=0.3), p))
    return out


def test_rows_do_not_depend_on_the_width():
    from paper_1809_08013_gb300 import binding as B
    insts = _insts()
    counts = [len(s["x"]) for s, _ in insts]
    state = {f: np.concatenate([s[f] for s, _ in insts]) for f in ics.FIELDS}
    ctx = B.Context(sum(counts), max_instances=len(insts))
    arr = B.alloc_arrays(state, ninst=len(insts))
    ctx.batch_set(counts, [p for _, p in insts])
    ctx.batch_step(arr, nsteps=2)
    ctx.sync()
    off = np.concatenate([[0], np.cumsum(counts)])
    for k, (s, p) in enumerate(insts):
        one = B.Context(counts[k])
        a = B.alloc_arrays(s)
        one.step(p, a, nsteps=2)
        one.sync()
        for f in FIELDS:
            got = arr[f][off[k]:off[k + 1]].cpu().numpy()
            assert np.array_equal(got.view(np.uint8), a[f].cpu().numpy().view(np.uint8)), (k, f)
        one.close()
    ctx.close()


@pytest.mark.parametrize("k", [2, 3, 4, 5])
def test_sets_at_every_width(orc, k):
    from paper_1809_08013_gb300 import binding as B
    s, p = _insts()[k]
    h, nnb, _, _ = orc.h_iterate(p, s["x"], s["y"], s["z"], s["h"])
    off, idx, ng = orc.csr(p, s["x"], s["y"], s["z"], h)
    ctx = B.Context(len(h))
    arr = B.alloc_arrays({**s, "h": h})  # the first count already converges
    ctx.build_neighbors(p, arr)
    assert ctx.sync() == B.SPH_OK
    assert np.array_equal(arr["h"].cpu().numpy().view(np.int64), h.view(np.int64))
    assert np.array_equal(arr["nnb"].cpu().numpy(), nnb)
    goff, gidx, gng = ctx.neighbors_caller(len(h))
    assert np.array_equal(goff, off) and np.array_equal(gng, ng)
    row = np.repeat(np.arange(len(h)), np.diff(off))
    part = (np.arange(len(idx)) - np.repeat(off[:-1], np.diff(off)) >= np.repeat(ng, np.diff(off)))
    assert np.array_equal(gidx, idx[np.lexsort((idx, part, row))])
    ctx.close()
