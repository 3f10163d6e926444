"""Quotients of the nonlinear weights at the ends of the FP64 range: the joint division of three of
them has to give what the single divisions give, or leave them to it. Forward and adjoint against
the oracle at the bars of the parity tests (1e-12; 1e-10 for the dot product)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2203_09047_gb300 as gks  # noqa: E402
from paper_2203_09047_gb300 import build, inputs as I  # noqa: E402


@pytest.fixture(scope="module")
def box():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gks.load_library()
    m = I.layered_box_mesh(8, "hybrid8", shape=(5, 6))
    return m, oracle.Mesh(m, min_stencil=18)


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("weps,p0", [(3e-94, 1e14), (1e-80, 1e20), (1e60, 1e-25), (1e-8, 1.0)])
def test_jump_beside_flat_candidates(box, weps, p0):
    """A pressure step: candidates on one side of it have indicator zero, so that three quotients
    tau / epsilon with tau of the order of p0^2 share a division (tau / epsilon^3 is out of range
    for the first two)."""
    m, om = box
    x = I.vertex_mean(m)
    n = om.n_cells
    q = I.primitive_to_conserved(np.ones(n), np.zeros((n, 3)),
                                 p0 * np.where(x[:, 2] < 1.0, 1.0, 1.5))
    dt = 0.01 / np.sqrt(p0)
    Lo, _ = om.residual(oracle.params_vec(weno_eps=weps), q, dt)
    L, _ = gks.Solver(m, min_stencil=18, weno_eps=weps).residual(q, dt)
    for v in range(5):
        if np.linalg.norm(Lo[v]) > 0:
            assert rel(L.cpu()[v], Lo[v]) < 1e-12


@pytest.mark.parametrize("weps", [1e-150, 1e-110, 1e120, 1e200])
def test_adjoint_at_extreme_epsilons(box, weps):
    """Smooth density in a gas at rest (the momenta and the energy have indicators zero)."""
    m, om = box
    x = I.vertex_mean(m)
    n = om.n_cells
    q = I.primitive_to_conserved(1 + 0.2 * np.sin(np.pi * x.sum(1)), np.zeros((n, 3)), np.ones(n))
    P = oracle.params_vec(weno_eps=weps)
    S = gks.Solver(m, min_stencil=18, weno_eps=weps)
    gL, gLt, dQ = I.normal_directions(q.shape, 3, 54)
    Lo, _, dL, dLt = om.residual_jvp(P, q, dQ, 0.01)
    L, _ = S.residual(q, 0.01)
    assert rel(L.cpu(), Lo) < 1e-12
    lhs = (S.residual_vjp(q, 0.01, gL, gLt).cpu().numpy() * dQ).sum()
    rhs = (gL * dL).sum() + (gLt * dLt).sum()
    assert abs(lhs - rhs) <= 1e-10 * abs(rhs), (lhs, rhs)
