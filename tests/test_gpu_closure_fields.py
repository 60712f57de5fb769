"""The closure's fields from the raw sums (n, u, T, q), by themselves: the steps whose rounding is part of the
library's precision."""
import numpy as np
import pytest

from . import device_unit

pytestmark = pytest.mark.gpu

FIELDS = """
    Wide<real> sv[kSums], nw, u[3], Tc;
    real q[3];
    for (int k = 0; k < kSums; ++k) { %s; }
    clo_fields<real>(sv, nw, u, Tc, q);
    for (int a = 0; a < 3; ++a) y[a] = %s, y[3 + a] = q[a];
    y[6] = %s;
"""
FIELDS_FP32 = FIELDS % ("sv[k] = w_from_t((real)x[k]); sv[k].lo = (real)(x[k] - (double)(real)x[k])", "u[a].hi", "Tc.hi")


def _sums(count, seed):
    rng = np.random.default_rng(seed)
    x = np.zeros((13, count))
    x[0] = np.exp(rng.uniform(-8, 3, count))
    x[1:4] = rng.normal(size=(3, count)) * x[0]
    return x


def test_heat_flux_takes_the_rounded_wide_kinetic_energy(tmp_path):
    # with only n and n u given, q_a = n |u|^2 u_a: products of FP32 values with one rounding each, |u|^2 the
    # double-float sum rounded once (wide values within 2^-40 of the exact ones round like them but for one in
    # 2^15)
    x = _sums(20000, 3)
    y = device_unit.run(tmp_path, "float", FIELDS_FP32, x, 7)
    f32 = lambda v: np.float32(v).astype(np.float64)  # noqa: E731
    u = x[1:4] / x[0]
    nuu = f32(f32(x[0]) * f32(np.sum(u * u, axis=0)))
    q = f32(nuu * f32(u))
    assert np.mean(y[:3] != f32(u)) < 1e-3
    assert np.mean(y[3:6] != q) < 1e-3


def test_fp64_velocities_and_temperature_are_rounded_quotients(tmp_path):
    # u = (n u) / n and, at rest, T = tr / (3 n), each the correctly rounded quotient
    x = _sums(20000, 5)
    y = device_unit.run(tmp_path, "double", FIELDS % ("sv[k].v = x[k]", "u[a].v", "Tc.v"), x, 7)
    assert np.array_equal(y[:3], x[1:4] / x[0])
    x[1:4] = 0.0
    x[4:7] = np.exp(np.random.default_rng(6).uniform(-1, 1, (3, x.shape[1]))) * x[0]
    y = device_unit.run(tmp_path, "double", FIELDS % ("sv[k].v = x[k]", "u[a].v", "Tc.v"), x, 7)
    assert np.array_equal(y[6], ((x[4] + x[5]) + x[6]) / (3.0 * x[0]))
