"""Rows of S_i as a step leaves them: the outer parts appended by the density
kernel and sorted by k_rowlen_sort, against the oracle's sets, on spheres
whose density profile makes the outer parts from empty to over a hundred
entries, and one whose rows overflow their slabs."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _steep_sphere(power):
    """Evrard directions and masses with radii U^power (0.5 is the Evrard profile)."""
    s, p = ics.evrard(6000, seed=4)
    r = np.sqrt(s["x"] ** 2 + s["y"] ** 2 + s["z"] ** 2)
    for c in "xyz":
        s[c] *= r ** (2 * power) / r
    s["h"][:] = 0.2 * 1.44 * np.cbrt(1.0 / 6000)
    return s, p


# (power, rows of each class of the sort that must occur, does a row overflow its slab)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("power,classes,overflow", [(0.5, (1, 8, 24, 64), False),
                                                    (3.0, (1, 8, 24, 64, 121), False),
                                                    (5.0, (1, 8, 24, 64, 121), True)])
def test_rows_after_a_step(orc, power, classes, overflow, precision):
    from paper_1809_08013_gb300 import binding as B
    s, p = _steep_sphere(power)
    p.precision = precision
    h, _, _, _ = orc.h_iterate(p, s["x"], s["y"], s["z"], s["h"])
    off, idx, ng = orc.csr(p, s["x"], s["y"], s["z"], h)
    no = np.diff(off) - ng
    for a, b in zip((0,) + classes, classes):  # the input holds rows of every class
        assert np.any((no > a) & (no <= b))
    assert (np.max(np.diff(off)) > 224) == overflow
    ctx = B.Context(len(s["x"]), nnz_capacity=400 * len(s["x"]))
    arr = B.alloc_arrays(s)
    ctx.step(p, arr, nsteps=1)
    # h of the steepest sphere's centre lies more than 2^15 below the mean h of the state that
    # enters the step, the unit of the pair kernels: reported; the neighbour sets are exact
    wide = np.mean(s["h"]) / np.min(h) > 2.0 ** 15
    assert ctx.sync() == (B.SPH_E_RANGE if wide else B.SPH_OK)
    goff, gidx, gng = ctx.neighbors_caller(len(s["x"]))
    assert np.array_equal(goff, off) and np.array_equal(gng, ng)
    for i in range(len(s["x"])):
        a, m, e = off[i], off[i] + ng[i], off[i + 1]
        assert np.array_equal(gidx[a:m], np.sort(idx[a:m]))
        assert np.array_equal(gidx[m:e], np.sort(idx[m:e]))
    if not overflow:  # each outer part in ascending internal index
        ioff, iidx, ing, _ = ctx.neighbors_to_host()
        inner = np.ones(len(iidx) - 1, dtype=bool)
        inner[(ioff[1:-1] - 1)] = False                    # across rows
        starts = ioff[:-1] + ing
        pos = np.arange(len(iidx) - 1)
        row = np.searchsorted(ioff, pos, side="right") - 1
        inner &= pos >= starts[row]                        # inside an outer part
        assert np.all(np.diff(iidx.astype(np.int64))[inner] > 0)
    ctx.close()
