"""erfc(z)/2 and its derivative from the FP64 table of the flux kernels, on the host.

Error bound: with u = 2^-53, the coefficients and the last FMA round once each and the lower terms
weigh at most 2 |z| / 128 <= 1/16 of the value, which gives 2.2 u; the Taylor remainder at |z| = 4
is 0.4 u of the derivative. 4 u bounds both."""
import ctypes

import numpy as np
import pytest

import oracle
import paper_2203_09047_gb300 as gks
from paper_2203_09047_gb300 import build

D = ctypes.POINTER(ctypes.c_double)


@pytest.fixture(scope="module")
def lib():
    build.build()
    return gks.load_library()


def _table(lib, z):
    f, d = np.full_like(z, np.nan), np.full_like(z, np.nan)
    p = lambda a: a.ctypes.data_as(D)
    return lib.gks_half_erfc_host(len(z), p(z), p(f), p(d)), f, d


@pytest.mark.parametrize("lo,hi", [(-4, -3), (-1, 1), (3, 4)])
def test_table_against_extended_precision(lib, lo, hi):
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 120
    h = 1.0 / 128.0  # record boundaries lie at odd multiples of h
    z = np.concatenate([np.random.default_rng(5).uniform(lo, hi, 500),
                        lo + h + np.arange(8) * 2 * h, np.nextafter([lo, hi], 0.0)])
    out, f, d = _table(lib, z)
    assert out == 0
    for x, a, b in zip(z, f, d):
        x = mp.mpf(float(x))
        F, G = mp.erfc(x) / 2, -mp.exp(-x * x) / mp.sqrt(mp.pi)
        assert abs((mp.mpf(float(a)) - F) / F) < 4 * 2.0 ** -53
        assert abs((mp.mpf(float(b)) - G) / G) < 4 * 2.0 ** -53


def test_points_beyond_the_table(lib):
    out, f, _ = _table(lib, np.array([4.0, -4.0, 1e300, np.inf, -np.inf, np.nan]))
    assert out == 6 and np.isnan(f).all()


@pytest.mark.parametrize("un", [-9.0, 3.9, 4.1, 9.0])
def test_flux_on_both_sides_of_the_table_end(lib, un):
    """p = rho / 2, so lam = 1 and erfc's argument is the normal velocity itself."""
    ff = np.tile([1.0, 0, 0, 0, 1 / 1.4], 6)
    P = np.concatenate([[1.4, 2e-3, 0.01, 1.0, 1, 1, 1.0, 0.9, 0.7], np.zeros(24), ff])
    rng = np.random.default_rng(3)
    q = lambda r: np.array([r, r * un, 0.1 * r, 0.2 * r, 0.5 * r / 0.4 + 0.5 * r * (un ** 2 + 0.05)])
    ql, qr, dql, dqr = q(1.0), q(1.1), rng.normal(size=(3, 5)) * 0.1, rng.normal(size=(3, 5)) * 0.1
    Fn, Ft = np.zeros(5), np.zeros(5)
    p = lambda a: np.ascontiguousarray(a).ctypes.data_as(D)
    assert lib.gks_gp_flux_host(p(P), p(ql), p(dql), p(qr), p(dqr), ctypes.c_double(0.01),
                                Fn.ctypes.data_as(D), Ft.ctypes.data_as(D)) == 0
    Fo = oracle.gp_flux(oracle.params_vec(flux_mode=1, tau_model=1, mu=2e-3), ql, dql, qr, dqr, 0.01)
    Fn_o, Ft_o = (4 * Fo[0] - Fo[1]) / 0.01, 4 * (Fo[1] - 2 * Fo[0]) / 1e-4
    # the tolerances of the other points of this flux (test_kinetic_host.py)
    np.testing.assert_allclose(Fn, Fn_o, rtol=0, atol=1e-11 * np.abs(Fn_o).max())
    np.testing.assert_allclose(Ft, Ft_o, rtol=0, atol=1e-10 * np.abs(Ft_o).max())
