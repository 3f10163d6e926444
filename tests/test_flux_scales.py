"""The FP64 flux over the whole range of densities: it is homogeneous of degree one in the conserved
variables, so scaling both sides by a power of two scales it by the same factor, also where the
product rho rho p that gives both reciprocals would leave the FP64 range. Host instantiation.

The scaled runs take the general reciprocals where the unscaled ones take the joint one: a few
roundings of 2^-53 in the primitives, amplified by the fit of dF/dt as in the other tests of this
flux (1e-11 of the largest F^n, 1e-10 of the largest dF/dt)."""
import ctypes

import numpy as np
import pytest

import paper_2203_09047_gb300 as gks
from paper_2203_09047_gb300 import build

D = ctypes.POINTER(ctypes.c_double)


@pytest.fixture(scope="module")
def lib():
    build.build()
    return gks.load_library()


def _run(lib, P, vl, gl, vr, gr, n, g):
    p = lambda a: np.ascontiguousarray(a, dtype=np.float64).ctypes.data_as(D)
    acc, out = np.zeros(10), [np.zeros(5), np.zeros((5, 3)), np.zeros(5), np.zeros((5, 3))]
    st = lib.gks_gp_face_host(p(P), p(vl), p(gl), p(vr), p(gr), p(n), ctypes.c_double(0.25),
                              ctypes.c_double(2e-3), acc.ctypes.data_as(D), p(g),
                              *[o.ctypes.data_as(D) for o in out])
    return st, acc, out


@pytest.mark.parametrize("mode,tau_model", [(0, 0), (1, 1)])
@pytest.mark.parametrize("power", [-560, -500, -330, -100, 100, 330, 480])
def test_scaled_states(lib, mode, tau_model, power):
    ff = np.tile([1.0, 0, 0, 0, 1 / 1.4], 6)
    P = np.concatenate([[1.4, 0.0, 0.01, 1.0, mode, tau_model, 1.0, 1.0, 0.7], np.zeros(24), ff])
    rng = np.random.default_rng(71)
    state = lambda: np.array([1.1, 0.3, -0.2, 0.4, 2.9]) + 0.05 * rng.normal(size=5)
    vl, vr, gl, gr = state(), state(), rng.normal(size=(5, 3)) * 0.2, rng.normal(size=(5, 3)) * 0.2
    n, g = np.array([0.48, 0.6, 0.64]), rng.normal(size=10)
    st, F, G = _run(lib, P, vl, gl, vr, gr, n, g)
    c = 2.0 ** power
    st_c, F_c, G_c = _run(lib, P, c * vl, c * gl, c * vr, c * gr, n, g)
    assert st == 0 and st_c == 0
    for h, tol in ((slice(0, 5), 1e-11), (slice(5, 10), 1e-10)):
        np.testing.assert_allclose(F_c[h] / c, F[h], rtol=0, atol=tol * np.abs(F[h]).max())
    if abs(power) <= 330:  # the reverse divides by rho once more
        for a, b in zip(G_c, G):  # cotangents of states do not scale
            np.testing.assert_allclose(a, b, rtol=0, atol=1e-9 * np.abs(b).max())


def test_non_physical_sides_are_refused(lib):
    ff = np.tile([1.0, 0, 0, 0, 1 / 1.4], 6)
    P = np.concatenate([[1.4, 0.0, 0.01, 1.0, 0, 0, 1.0, 1.0, 0.7], np.zeros(24), ff])
    ok = np.array([1.0, 0.1, 0.0, 0.0, 2.5])
    z, n, g = np.zeros((5, 3)), np.array([1.0, 0.0, 0.0]), np.ones(10)
    for bad in ([-1.0, 0.1, 0, 0, 2.5], [0.0, 0, 0, 0, 2.5], [1.0, 3.0, 0, 0, 2.5],
                [np.nan, 0, 0, 0, 2.5], [1.0, 0, 0, 0, np.nan], [-1.0, 0, 0, 0, -2.5]):
        assert _run(lib, P, ok, z, np.array(bad), z, n, g)[0] == 1
