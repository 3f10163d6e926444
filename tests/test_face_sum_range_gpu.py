"""Face fluxes near the end of the FP32 range: their sums over a cell are FP64 values (the residual of
the mixed precision and its FP64 update), so a partial sum of finite FP32 fluxes that is beyond
the FP32 range is not lost. Cells of 2.3e18 with faces of 5.3e36 and energy fluxes of about 42
per area give 2.2e38 per face. Bars of the parity tests for the mixed residual (2e-4)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2203_09047_gb300 as gks  # noqa: E402
from paper_2203_09047_gb300 import build, inputs as I  # noqa: E402

H = 2.0 ** 61


@pytest.fixture(scope="module")
def box():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gks.load_library()
    m = I.layered_box_mesh(6, "hex", hi=(6 * H,) * 3, jitter=0.02)
    return m, oracle.Mesh(m)


@pytest.mark.parametrize("signs", [(1, 1, 1), (-1, 1, 1), (1, -1, 1), (1, 1, -1)])
def test_partial_sums_beyond_fp32(box, signs):
    m, om = box
    n = om.n_cells
    u = np.tile(1.94 * np.array(signs), (n, 1))
    x = np.pi / (3 * H) * I.vertex_mean(m).sum(1)
    q = I.primitive_to_conserved(1 + 0.01 * np.sin(x), u, 4.4 + 0.02 * np.cos(x))
    dt = 0.05 * H
    Lo, Lto = om.residual(oracle.params_vec(), q, dt)
    L, Lt = gks.Solver(m, precision=gks.GKS_PREC_MIXED).residual(q, dt)
    L = L.cpu().numpy()
    assert np.isfinite(L).all() and np.isfinite(Lt.cpu().numpy()).all()
    assert np.linalg.norm(L - Lo) < 2e-4 * np.linalg.norm(Lo)
    S = gks.Solver(m, precision=gks.GKS_PREC_MIXED_FP64UPD)
    S.set_state(q)
    S.step(dt, 1)
    d = om.step(oracle.params_vec(), q, dt, 1) - q
    assert np.linalg.norm(S.get_state().cpu().numpy() - q - d) < 2e-4 * np.linalg.norm(d)
