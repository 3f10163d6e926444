"""The time-step bound where the FP32 estimate that chooses the cells to evaluate in FP64 is weakest,
against the oracle on the same states. The cells are of two kinds whose true bounds lie a few
percent apart, so that an estimate that is off by more than its margin of 2^-9 picks the wrong
kind and returns a step above the bound.

Tolerance: a few roundings of 2^-53 (FP64) or of the float-float state, 2^-47, raised by the
cancellation of the pressure, rho E over the internal energy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2203_09047_gb300 as gks  # noqa: E402
from paper_2203_09047_gb300 import build, inputs as I  # noqa: E402

PRECISIONS = [gks.GKS_PREC_FP64, gks.GKS_PREC_MIXED, gks.GKS_PREC_MIXED_FP64UPD]


@pytest.fixture(scope="module")
def cubes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gks.load_library()
    m = I.layered_box_mesh(8, "hex", jitter=0.0)  # every cell has the same size
    return m, oracle.Mesh(m)


def check(cubes, rho, U, e, prec, **prm):
    """rho [n], U [n, 3], internal energy per mass e [n]."""
    m, om = cubes
    q = np.ascontiguousarray(np.stack([rho, *(rho[:, None] * U).T,
                                       rho * (e + 0.5 * (U * U).sum(1))]))
    S = gks.Solver(m, precision=prec, **prm)
    S.set_state(q)
    ref = om.max_dt(oracle.params_vec(**prm), q, 0.5)
    cond = float((1.0 + 0.5 * (U * U).sum(1) / e).max())
    tol = 8 * cond * 2.0 ** (-53 if prec == gks.GKS_PREC_FP64 else -46) + 1e-11
    assert abs(S.max_dt(0.5) - ref) <= tol * ref


def two_kinds(n):
    return np.arange(n) % 2 == 0


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("gm1", [1e-3, 3e-7, 1e-7])
def test_gamma_near_one(cubes, prec, gm1):
    """Sound speed 1 at rest against a stream at 1.03: gamma - 1 has to be that of the FP64 gamma
    (rounded to FP32 first, gamma - 1 = 3e-7 becomes 3.6e-7)."""
    n, a, g = 512, two_kinds(512), 1.0 + gm1
    U = np.zeros((n, 3))
    U[~a, 0] = 1.03
    check(cubes, np.ones(n), U, np.where(a, 1.0 / (g * (g - 1.0)), 1.0), prec, gamma=g)


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("rho,c", [(1e-10, 1.9545e-12), (1e-10, 2.6e-12)])
def test_states_whose_products_are_subnormal_in_fp32(cubes, prec, rho, c):
    """rho E of a few units of the smallest FP32 number: such cells are evaluated in FP64."""
    n, a = 512, two_kinds(512)
    U = np.zeros((n, 3))
    U[~a, 1] = 0.8 * c
    e = c * c / (1.4 * 0.4)
    check(cubes, np.full(n, rho), U, np.where(a, e, 0.02 * e), prec)


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("mach,warm,mu_pow", [(540.0, 0.998, 0.7), (540.0, 0.9995, 0.7),
                                              (30.0, 0.9995, 0.7), (60.0, 0.999, 40.0), (2.0, 1.01, -300.0)])
def test_power_law_viscosity_of_fast_gas(cubes, prec, mach, warm, mu_pow):
    """A bound set by mu(T): the temperature of a fast gas loses rho E over the internal energy in
    FP32, the exponent multiplies that."""
    n, a = 512, two_kinds(512)
    rng = np.random.default_rng(3)
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    U = np.where(a, 0.0, mach * np.sqrt(1.4) * (0.95 + 0.05 * rng.random(n)))[:, None] * d
    check(cubes, np.ones(n), U, np.where(a, 1.0, warm) / 0.4, prec, mu=1e6, tau_model=3, T_ref=1.0,
          mu_pow=mu_pow)


@pytest.mark.parametrize("prec", PRECISIONS)
def test_large_ragged_mesh(prec):
    """Four cells per thread (from 155,648 cells on), the last block partly filled; the smallest
    bound in the first, the last and an inner cell."""
    m = I.layered_box_mesh(32, "hex", shape=(71, 69))
    om = oracle.Mesh(m, lazy=True)
    n = om.n_cells
    assert n >= 155648 and n % 1024
    rng = np.random.default_rng(64)
    rho, u = 1 + 0.3 * rng.random(n), 0.5 * rng.normal(size=(n, 3))
    q = I.primitive_to_conserved(rho, u, 1 + 0.3 * rng.random(n))
    S = gks.Solver(m, precision=prec, mu=1e-4, tau_model=2)
    for cell in (None, 0, n // 3, n - 1):
        x = q.copy()
        if cell is not None:
            x[4, cell] *= 300.0
        S.set_state(np.ascontiguousarray(x))
        ref = om.max_dt(oracle.params_vec(mu=1e-4, tau_model=2), np.ascontiguousarray(x), 0.5)
        assert abs(S.max_dt(0.5) - ref) <= (1e-13 if prec == gks.GKS_PREC_FP64 else 1e-11) * ref
