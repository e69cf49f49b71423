"""The internal order (order[]) against a stable sort by cell code on the CPU,
at sizes on both sides of the sort's tiles and of its change of tile size."""
import numpy as np
import pytest

from paper_1809_08013_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _trunc32(v):
    """Float32 of v rounded toward zero."""
    f = v.astype(np.float32)
    over = np.abs(f.astype(np.float64)) > np.abs(v)
    return np.where(over, np.nextafter(f, np.float32(0)), f)


def _spread(v):
    out = np.zeros_like(v)
    for b in range(8):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def expected_order(s, cap_cells):
    w = 2.0 * np.mean(s["h"])
    while True:  # the cell grid: width 2 <h>, widened to the cell budget
        cnt, width = [], []
        for d in "xyz":
            ext = s[d].max() - s[d].min()
            c = min(max(np.floor(ext / w) + 1.0, 1.0), 256.0)
            width.append(ext / (c - 0.5) if c * w <= ext else w)
            cnt.append(int(c))
        if cnt[0] * cnt[1] * cnt[2] <= cap_cells:
            break
        w *= 1.25
    code = np.zeros(len(s["x"]), dtype=np.int64)
    for d, (name, c, ww) in enumerate(zip("xyz", cnt, width)):
        f = np.floor((_trunc32(s[name]) - np.float32(s[name].min())) * np.float32(1.0 / ww))
        code |= _spread(np.clip(f, 0, c - 1).astype(np.int64)) << d
    return np.argsort(code, kind="stable")


@pytest.mark.parametrize("n", [1, 2, 511, 512, 513, 8191, 8193, 100003, 262144, 262145, 600001])
def test_order_is_the_stable_sort_by_cell(n):
    from paper_1809_08013_gb300 import binding as B
    s, p = ics.evrard(n, seed=n)
    s["h"][:] = np.float64(0.75) * n ** (-1.0 / 3.0)  # one h: its mean is exact
    ctx = B.Context(n)
    arr = B.alloc_arrays(s)
    ctx.build_neighbors(p, arr)
    _, _, _, order = ctx.neighbors_to_host()
    assert np.array_equal(order, expected_order(s, max(2 * n, 4096)))
    ctx.close()
