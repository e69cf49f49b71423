"""The CSR fallback (a row of S_i that does not fit its slab): its rows against
the oracle's at sizes where its items hold one row a warp, a few, and the most,
and at the ends of an item; and contexts stepping at the same time on streams of
their own, fallback and all, against the same steps alone."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics
from test_gpu_rows import _steep_sphere

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _many(n, seed):
    """Gather sets of about 140 entries, over the 128 of a slab."""
    s, p = ics.evrard(n, seed=seed)
    p.n_target = 140
    s["h"][:] *= (140 / 100) ** (1 / 3)
    return s, p


@pytest.mark.parametrize("n", [141, 2000, 6007, 45001, 90003, 160001])
def test_rows_of_the_fallback(orc, n):
    from paper_1809_08013_gb300 import binding as B
    s, p = _many(n, n)
    h, _, _, _ = orc.h_iterate(p, s["x"], s["y"], s["z"], s["h"])
    off, idx, ng = orc.csr(p, s["x"], s["y"], s["z"], h)
    assert np.max(ng) > 128  # the input needs the fallback
    ctx = B.Context(n, nnz_capacity=int(off[-1]))
    ctx.step(p, B.alloc_arrays(s), nsteps=1)
    assert ctx.sync() == B.SPH_OK
    goff, gidx, gng = ctx.neighbors_caller(n)
    assert np.array_equal(goff, off) and np.array_equal(gng, ng)
    row = np.repeat(np.arange(n), np.diff(off))
    part = np.arange(len(idx)) - np.repeat(off[:-1], np.diff(off)) >= np.repeat(ng, np.diff(off))
    assert np.array_equal(gidx, idx[np.lexsort((idx, part, row))])
    ctx.close()
    small = B.Context(n, nnz_capacity=int(off[-1]) - 1)  # one entry too few: refused as before
    small.step(p, B.alloc_arrays(s), nsteps=1)
    assert small.sync() == B.SPH_E_CAPACITY
    small.close()


def test_contexts_at_the_same_time():
    from paper_1809_08013_gb300 import binding as B
    kinds = [_many(6000, 1), ics.square_patch(16, seed=2), _steep_sphere(5.0), _many(30000, 3),
             ics.square_patch(24, seed=4)]
    alone, ctxs = [], []
    for s, p in kinds:
        ctx, a = B.Context(len(s["x"]), nnz_capacity=600 * len(s["x"])), B.alloc_arrays(s)
        ctx.step(p, a, nsteps=4)
        alone.append((ctx.sync(), {f: a[f].clone() for f in ("x", "vx", "h", "rho", "ax", "du", "nnb")}))
        ctx.close()
        ctxs.append((B.Context(len(s["x"]), nnz_capacity=600 * len(s["x"])), p, B.alloc_arrays(s),
                     torch.cuda.Stream()))
    torch.cuda.synchronize()
    for ctx, p, a, st in ctxs:
        ctx.step(p, a, nsteps=4, stream=st)
    for (ctx, p, a, st), (status, want) in zip(ctxs, alone):
        assert ctx.sync(st) == status
        for f in want:  # NaN == NaN: the same bits
            assert torch.equal(a[f].view(torch.uint8), want[f].view(torch.uint8)), f
    for c in ctxs:
        c[0].close()
