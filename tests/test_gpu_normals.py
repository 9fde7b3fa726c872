"""The float64 logarithm, sine and cosine of the Box–Muller transform at the ends of
their table intervals, against the transform in long double arithmetic.

Tolerance: log within an ulp, the angle's functions within 1.2e-16, a square root and a
product: a normal is at most sqrt(106 log 2) = 8.6, each of the four roundings at most
2^-53 of it, the log's half under the root: 4.5 * 2^-53 * 8.6 = 4.3e-15.
"""
import numpy as np
import pytest
import torch

import paper_2605_24882_gb300 as wm
from oracle.philox import philox4x32_10

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 7, 2 ** 63 + 5])
def test_normals_against_long_double(seed):
    n = 400_000
    z = wm.normals(seed, 3, 0, 0, n).cpu().numpy()
    q = np.arange(n // 2, dtype=np.uint64)
    c = np.stack([q, np.full_like(q, 3), np.zeros_like(q), np.zeros_like(q)])
    o = philox4x32_10(c, np.array([seed & 0xFFFFFFFF, seed >> 32], dtype=np.uint64)).astype(np.uint64)
    m = [((a >> np.uint64(5)) * np.uint64(1 << 26) + (b >> np.uint64(6)) + np.uint64(1)) for a, b in
         ((o[0], o[1]), (o[2], o[3]))]
    u = [x.astype(np.longdouble) * np.longdouble(2.0) ** -53 for x in m]
    # the angle from the nearest quarter turn, so that it is small and exact
    k = np.rint(u[1] * 4)
    f = (u[1] - k / 4) * (2 * np.longdouble("3.14159265358979323846264338327950288"))
    k = k.astype(np.int64) & 3
    s, co = np.sin(f), np.cos(f)
    sn = np.where(k == 0, s, np.where(k == 1, co, np.where(k == 2, -s, -co)))
    cs = np.where(k == 0, co, np.where(k == 1, -s, np.where(k == 2, -co, s)))
    rad = np.sqrt(-2 * np.log(u[0]))
    err = np.abs(z.reshape(-1, 2) - np.stack([rad * cs, rad * sn], axis=1).astype(np.longdouble)).max()
    assert float(err) < 4.3e-15
    # table intervals: every one of the logarithm's 128 and the turn's 64 is met
    mant = np.frexp(u[0].astype(np.float64))[0] * 2 - 1
    assert len(np.unique((mant * 128).astype(int))) == 128
    assert len(np.unique(np.rint(u[1] * 64).astype(int) & 63)) == 64


def test_two_elements_per_thread_give_the_same_loads():
    """Enough samples switch the loads to two elements per thread; the values of a sample
    do not depend on it."""
    hier = wm.Hierarchy(wm.Geometry("sphere", 2, 32), 1)
    many = hier.noise_loads(5, 64)  # 6,144 elements x 64 samples
    few = hier.noise_loads(5, 8)
    assert torch.equal(many[:8], few)
