"""The internal order of a batch against a stable sort by cell code on the CPU,
instance by instance (the sort's fourth pass, over the instance), on both sides
of its change of tile size and in contexts with room for more particles than
the batch has, among them one whose capacity needs fewer groups of tiles than
the batch."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics
from test_gpu_sort import expected_order

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("capacity,counts", [
    (262144, [100003, 513, 1, 161627]),             # 262,144 keys: the largest chained sort
    (400000, [100003, 513, 1, 161628]),             # one more: a histogram kernel per pass
    (2097153, [1, 511, 261632] + [262144] * 7),     # 1,024 tiles of a context of 1,025
])
def test_order_within_each_instance(capacity, counts):
    from paper_1809_08013_gb300 import binding as B
    insts = []
    for k, n in enumerate(counts):
        s, p = ics.evrard(n, seed=100 + k)
        s["h"][:] = 0.75 * n ** (-1.0 / 3.0)  # one h: its mean is exact
        p.n_target = p.n_tol = 8
        insts.append((s, p))
    state = {f: np.concatenate([s[f] for s, _ in insts]) for f in ics.FIELDS}
    ctx = B.Context(capacity, nnz_capacity=48 * capacity, max_instances=16)
    arr = B.alloc_arrays(state, ninst=len(insts))
    ctx.batch_set(counts, [p for _, p in insts])
    ctx.batch_step(arr, nsteps=1)
    ctx.sync()
    _, _, _, order = ctx.neighbors_to_host()
    order = order[order >= 0]
    a = 0
    for k, (s, _) in enumerate(insts):
        want = a + expected_order(s, max(2 * counts[k], 4096))
        assert np.array_equal(order[a:a + counts[k]], want), k
        a += counts[k]
    ctx.close()


def test_one_context_for_problems_of_other_sizes():
    from paper_1809_08013_gb300 import binding as B
    ctx = B.Context(300000, nnz_capacity=48 * 300000)
    for n in (300000, 262145, 262144, 5000, 262145):  # with and without a histogram kernel
        s, p = ics.evrard(n, seed=n)
        s["h"][:] = 0.75 * n ** (-1.0 / 3.0)
        p.n_target = p.n_tol = 8
        ctx.build_neighbors(p, B.alloc_arrays(s))
        assert np.array_equal(ctx.neighbors_to_host()[3], expected_order(s, max(2 * n, 4096))), n
    ctx.close()
