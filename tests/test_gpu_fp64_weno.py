"""The FP64 reconstruction by itself (weights without quotients) against the method's form in extended precision:
smooth and rough windows over forty orders of magnitude, epsilon scaled by weights down to 1e-60, constant
windows, both upwind directions.  A difference t of the window carries up to five roundings of its largest value,
a weight four times their share of t, and the candidates differ by about t / 3: sixteen units of the largest
value with the roundings of the candidates themselves, and as many again allowed."""
import numpy as np
import pytest

from . import device_unit

pytestmark = pytest.mark.gpu

BODY = "y[0] = weno5_one(x[0], x[1], x[2], x[3], x[4], x[5], x[5] > 0 ? 0.1 : 0.3, x[5] > 0 ? 0.3 : 0.1, x[6]);"
L = np.longdouble


def _face(w, sign, e4):
    """The value at the face beyond w2 in the direction of the sign, weights d_k / (eps + beta_k)^2."""
    w = w.astype(L)
    a, b, c, d, e = np.where(sign > 0, w, w[::-1])
    eps = e4.astype(L) / 4
    k13, q = L(13) / 12, L(1) / 4
    be = [eps + k13 * (a - 2 * b + c) ** 2 + q * (a - 4 * b + 3 * c) ** 2, eps + k13 * (b - 2 * c + d) ** 2 + q * (b - d) ** 2,
          eps + k13 * (c - 2 * d + e) ** 2 + q * (3 * c - 4 * d + e) ** 2]
    m = np.minimum(be[0], np.minimum(be[1], be[2]))
    al = [L(1) / 10 * (m / be[0]) ** 2, L(6) / 10 * (m / be[1]) ** 2, L(3) / 10 * (m / be[2]) ** 2]
    r = [(2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6]
    return sum(x * y for x, y in zip(al, r)) / sum(al)


def _compare(tmp_path, w, e4):
    n = w.shape[1]
    for sign in (1.0, -1.0):
        x = np.concatenate([w, np.full((1, n), 3.0 * sign), e4[None]])
        y = device_unit.run(tmp_path, "double", BODY, x, 1)[0]
        err = np.abs(y - _face(w, np.full(n, sign), e4)) / np.max(np.abs(w), axis=0)
        assert np.max(err) <= 32 * np.finfo(np.float64).eps


def test_windows_over_many_scales_match_the_direct_form(tmp_path):
    rng = np.random.default_rng(9)
    n = 20000
    rough = np.exp(rng.uniform(0, 3, (1, n)) * rng.normal(size=(5, n)))
    smooth = 1.0 + 0.01 * np.sin(0.3 * np.arange(5)[:, None] + rng.uniform(0, 6, n))
    for g in (rough, rough * np.sign(rng.normal(size=(5, n))), smooth, np.ones((5, n))):
        wt = 10.0 ** rng.uniform(-60, 0, n)
        f = g * wt * 10.0 ** rng.uniform(-20, 20, n)
        _compare(tmp_path, f, 4e-6 * wt * wt)


def test_indicators_far_apart_match_the_direct_form(tmp_path):
    # one side of the window 2^50 .. 2^480 times the other: indicators up to 2^960 apart, beyond the ratio from
    # which a stencil is given no weight, and (the last, by epsilon alone) beyond what a difference of exponents holds
    rng = np.random.default_rng(10)
    n = 20000
    for k in range(6):
        w = 1.0 + 0.1 * rng.normal(size=(5, n))
        big = 2.0 ** rng.uniform(50, 480, n)
        if k < 4:
            w[k + 1 if k < 2 else 0:5 if k < 2 else k - 1] *= big
            e4 = np.full(n, 4e-6)
        elif k == 4:  # (the rough stencils' values around zero, as in a jump back)
            w[0] *= big
            w[1] = w[2]
            e4 = np.full(n, 4e-6)
        else:  # smooth stencils whose indicator is epsilon alone, 2^-1000
            w[1:] = 1.0
            w[0] = 2.0 ** rng.uniform(1, 60, n)
            e4 = np.full(n, 2.0 ** -1000)
        _compare(tmp_path, w, e4)


def test_windows_that_are_not_finite_stay_so(tmp_path):
    rng = np.random.default_rng(11)
    for bad in (np.inf, -np.inf, np.nan):
        w = 1.0 + 0.1 * rng.normal(size=(5, 500))
        w[np.arange(500) % 5, np.arange(500)] = bad
        for sign in (1.0, -1.0):
            x = np.concatenate([w, np.full((1, 500), 3.0 * sign), np.full((1, 500), 4e-6)])
            assert not np.any(np.isfinite(device_unit.run(tmp_path, "double", BODY, x, 1)))
