"""The autotuner times a value of defer_lanes only where the batch's h search
reads it: runs that do the same work are no choice."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sides,skin,read", [((12, 14), 0.0, False), ((12, 14), 0.2, True),
                                             ((12, 47), 0.0, True)])
def test_defer_lanes_is_tried_where_it_is_read(sides, skin, read):
    from paper_1809_08013_gb300 import binding as B
    insts = [ics.square_patch(side, seed=side) for side in sides]
    for _, p in insts:
        p.list_skin = skin
    counts = [len(s["x"]) for s, _ in insts]
    state = {f: np.concatenate([s[f] for s, _ in insts]) for f in ics.FIELDS}
    ctx = B.Context(sum(counts), max_instances=len(insts))
    ctx.batch_set(counts, [p for _, p in insts])
    arr = B.alloc_arrays(state, ninst=len(insts))
    res = ctx.autotune(arr, nsteps=1, cell_scales=[1.0], pair_threads=[2], defer_lanes=[4, 8])
    tried = {t["defer_lanes"] for t in res["trials"]}
    assert tried == ({16, 8, 4} if read else {16})
    assert res["defer_lanes"] in tried
    ctx.close()
