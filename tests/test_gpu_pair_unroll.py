"""The pair kernels that evaluate several neighbours at a time, where a lane's
share of a row is not a multiple of that number: rows of 0 to ~30 entries, two
coincident particles, every number of lanes, against the oracle."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics
from parity_util import TOL_FP64, check, force_err, normwise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL_MIXED = 1e-5  # the stated accuracy of precision 1


@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("precision,kernel,gradients", [(0, 0, 0), (0, 1, 0), (0, 0, 1), (1, 0, 0)])
@pytest.mark.parametrize("target", [1, 4, 7, 13])
def test_short_rows(orc, target, precision, kernel, gradients, lanes):
    from paper_1809_08013_gb300 import binding as B
    s, p = ics.evrard(700, seed=target)
    s = ics.random_velocities(s, seed=3, scale=0.2)
    for f in ("x", "y", "z"):
        s[f][1] = s[f][0]  # r = 0: density counts the pair, the forces do not
    p.n_target, p.n_tol = target, min(2, target - 1)
    p.precision, p.kernel, p.gradients, p.pair_threads = precision, kernel, gradients, lanes
    o = orc.pipeline(p, s)
    ctx = B.Context(len(s["x"]))
    arr = B.alloc_arrays(s)
    ctx.build_neighbors(p, arr)
    ctx.density(p, arr)
    rho = arr["rho"].cpu().numpy()
    for f in ("rho", "p", "c"):  # the forces from the oracle's thermodynamic state
        arr[f].copy_(torch.as_tensor(o[f]))
    ctx.forces(p, arr)
    ctx.sync()
    tol = TOL_FP64 if precision == 0 else TOL_MIXED
    errs = {"rho": normwise(rho, o["rho"])}
    # (the IAD matrix of a few neighbours is so ill-conditioned that its inverse
    # amplifies the rounding of tau beyond the bar; 13 neighbours are enough)
    if not (gradients and target < 13):
        for k in ("ax", "ay", "az", "du", "mumax"):
            errs[k] = force_err(k, arr[k].cpu().numpy(), o[k], o, p.periodic_z)
    check(errs, tol)
    ctx.close()
