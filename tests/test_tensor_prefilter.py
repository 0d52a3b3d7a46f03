"""The interaction's tensor-core candidate test never rejects a pair that the
FP32 neighbour test accepts.

Operand rows (half precision, K = 16): in cells about the unit's centre, x in
two halves (x = xh + xl), y and z in one, |p|^2 and |q|^2 - thr in two; their
product is (|q|^2 - thr) + |p|^2 - 2 q.p without the term 2 ql pl of x, with
thr = 1 + 2^-9 + 2^-16 R^2, R the largest |x| of the unit's candidates (at
most 17: units span at most 32 cells).  Bound on what is lost, for |q - p| <=
1: y and z are off by at most 2^-11 (candidate, |y| <= 1.5) + 2^-13 (particle,
|y| <= 0.5) each, 1.73e-3 in |q - p|^2 in all; 2 ql pl by 2 (2^-12 R)^2; the
two-half norms by 2^-22 R^2 each; FP32 accumulation of at most 9 terms below 2
R^2 + 4 by 9 * 2^-23 (2 R^2 + 4).  The sum stays below the margin.  This
emulates the rows with numpy and adds the accumulation bound.  CPU only."""
import numpy as np
import pytest


def h(x):
    return np.asarray(x, np.float32).astype(np.float16)


def split(v):
    v = np.asarray(v, np.float32)
    hi = h(v)
    return hi, h(v - hi.astype(np.float32))


def value(q, p, R):
    """The product of the rows in exact arithmetic, and the accumulation bound."""
    thr = np.float32(2.0 ** -16 * R * R + (1.0 + 2.0 ** -9))
    (qxh, qxl), (pxh, pxl) = split(q[:, 0]), split(p[:, 0])
    qy, qz, py, pz = h(q[:, 1]), h(q[:, 2]), h(p[:, 1]), h(p[:, 2])
    f = np.float32
    qx, px = qxh.astype(f) + qxl.astype(f), pxh.astype(f) + pxl.astype(f)
    nh, nl = split(qx * qx + (qy.astype(f) ** 2 + qz.astype(f) ** 2) - thr)
    mh, ml = split(px * px + (py.astype(f) ** 2 + pz.astype(f) ** 2))
    d = np.float64
    terms = [-2 * qxh.astype(d) * pxh.astype(d), -2 * qxh.astype(d) * pxl.astype(d),
             -2 * qxl.astype(d) * pxh.astype(d), -2 * qy.astype(d) * py.astype(d),
             -2 * qz.astype(d) * pz.astype(d), mh.astype(d), ml.astype(d), nh.astype(d),
             nl.astype(d)]
    return sum(terms), 9 * 2.0 ** -23 * (2 * R * R + 4)


@pytest.mark.parametrize("R", [1.5, 4.5, 9.0, 17.0])
def test_no_pair_inside_the_support_is_rejected(R):
    rng = np.random.default_rng(int(R * 2))
    n = 400000
    q = np.empty((n, 3))
    q[:, 0] = rng.uniform(-R + 1, R - 1, n)
    q[:, 1:] = rng.uniform(-0.5, 0.5, (n, 2))
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    # at the support (within the FP32 test's own rounding) and inside
    r = np.where(rng.random(n) < 0.7, 1.0 + rng.uniform(-1e-6, 5e-7, n), rng.uniform(0, 1, n))
    p = q + u * r[:, None]
    inside = (np.abs(p[:, 0]) <= R) & (np.abs(p[:, 1:]) <= 1.5).all(1)
    v, acc = value(q[inside], p[inside], R)
    assert inside.sum() > n // 4
    assert np.all(v + acc < 0)


@pytest.mark.parametrize("R", [1.5, 4.5, 17.0])
def test_the_rounding_bound_stays_below_the_margin(R):
    lost = 2 * np.sqrt(2) * (2.0 ** -11 + 2.0 ** -13) + 2 * (2.0 ** -12 * R) ** 2 + \
        2 * 2.0 ** -22 * R * R + 9 * 2.0 ** -23 * (2 * R * R + 4) + 1e-6
    assert lost < 2.0 ** -9 + 2.0 ** -16 * R * R
