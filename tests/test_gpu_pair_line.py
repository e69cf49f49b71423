"""The pair kernels take their neighbours several at a time in a batch of at
most 50,000 particles (the density with an append of each in flight), one at a
time beyond. An instance on one side of that line alone and on the other side
inside a batch must give the same bits: both add a row's terms in its order."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics
from test_gpu_batch import FIELDS_OUT, B, host, run_alone, run_batch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,kernel,gradients", [(0, 0, 0), (0, 1, 0), (0, 0, 1), (1, 0, 0)])
def test_same_bits_on_both_sides_of_the_line(B, precision, kernel, gradients):  # noqa: F811
    insts = []
    for side, seed in ((13, 31), (37, 32)):  # 2,197 + 50,653 particles
        s, p = ics.square_patch(side, seed=seed)
        p.precision, p.kernel, p.gradients = precision, kernel, gradients
        insts.append((ics.random_velocities(s, seed=seed + 2, scale=1.0), p))
    _, arr, counts, _ = run_batch(B, insts, 2)
    alone = run_alone(B, *insts[0], 2)
    for f in FIELDS_OUT:
        got, want = host(arr[f])[:counts[0]], host(alone[f])
        assert np.array_equal(got, want), f
