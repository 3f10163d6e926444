"""The reconstruction's launch forms and weight options on the GPU, against the oracle: one launch
over all cell kinds (few tiles) and one per kind on forked streams (many), one kind, cell counts
that leave the last tile ragged, and the exponents of the nonlinear weights; forward in both
precisions at the tolerances of the parity tests, adjoint by the dot product with the oracle's
directional derivatives."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2203_09047_gb300 as gks  # noqa: E402
from paper_2203_09047_gb300 import build, inputs as I  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gks.load_library()


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


# layers, n, (nx, ny), min_stencil, weno_pow
FORMS = [("hybrid8", 8, (7, 5), 18, 1), ("hybrid8", 8, (6, 7), 0, 2), ("hybrid8", 8, (5, 6), 18, 3),
         ("hybrid8", 24, (21, 13), 18, 1), ("hex", 5, (5, 5), 0, 2), ("tet", 4, (4, 5), 20, 1),
         ("prism", 5, (4, 5), 0, 1)]


@pytest.mark.parametrize("layers,n,shape,min_stencil,wpow", FORMS)
def test_forms_against_oracle(layers, n, shape, min_stencil, wpow):
    m = I.layered_box_mesh(n, layers, shape=shape)
    om = oracle.Mesh(m, min_stencil=min_stencil)
    Q = I.perturbed_state(I.advection_state(m), seed=51, amp=0.03)
    p = dict(flux_mode=1, tau_model=2, mu=1e-3, weno_pow=wpow)
    dt = 0.01
    Lo, Lto = om.residual(oracle.params_vec(**p), Q, dt)
    S = gks.Solver(m, min_stencil=min_stencil, **p)
    L, Lt = S.residual(Q, dt)
    assert rel(L.cpu(), Lo) < 1e-12 and rel(Lt.cpu(), Lto) < 1e-12
    M = gks.Solver(m, min_stencil=min_stencil, precision=gks.GKS_PREC_MIXED, **p)
    assert rel(M.residual(Q, dt)[0].cpu(), Lo) < 2e-4
    gL, gLt, dQ = I.normal_directions(Q.shape, 3, 52)
    _, _, dL, dLt = om.residual_jvp(oracle.params_vec(**p), Q, dQ, dt)
    lhs = (S.residual_vjp(Q, dt, gL, gLt).cpu().numpy() * dQ).sum()
    rhs = (gL * dL).sum() + (gLt * dLt).sum()
    assert abs(lhs - rhs) <= 1e-10 * abs(rhs), (lhs, rhs)


@pytest.mark.parametrize("weps", [1e-150, 1e-110, 1e120, 1e200])
def test_extreme_weight_epsilon(weps):
    """Epsilons whose threefold product leaves the FP64 range, with variables whose indicators are
    zero (gas at rest): the weights take the general divisions."""
    m = I.layered_box_mesh(8, "hybrid8", shape=(5, 6))
    om = oracle.Mesh(m, min_stencil=18)
    Q = np.zeros((5, om.n_cells))
    Q[0] = 1.0 + 0.1 * I.uniform01(53, np.arange(om.n_cells, dtype=np.uint64))
    Q[4] = 2.5
    p = dict(weno_eps=weps)
    Lo, _ = om.residual(oracle.params_vec(**p), Q, 0.01)
    S = gks.Solver(m, min_stencil=18, **p)
    L, Lt = S.residual(Q, 0.01)
    assert rel(L.cpu(), Lo) < 1e-12 and np.isfinite(Lt.cpu().numpy()).all()
    gL, gLt, dQ = I.normal_directions(Q.shape, 3, 54)
    g = S.residual_vjp(Q, 0.01, gL, gLt).cpu().numpy()
    assert np.isfinite(g).all()
