"""The FP32 smooth flux with two Gauss points per thread (meshes of 60,000 faces and more) at
boundary planes, with each collision time, the Prandtl correction and the positivity fallback:
sampled cells against the oracle at the bar of the mixed residual (2e-4). And its second point:
each half of a pair is the flux of its own point."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2203_09047_gb300 as gks  # noqa: E402
from paper_2203_09047_gb300 import build, inputs as I  # noqa: E402

MIXED_TOL_L = 2e-4


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gks.load_library()


@pytest.fixture(scope="module")
def boxes():
    """Slip walls in x, no-slip walls in y, far field in z; and a box of slip walls."""
    out = []
    for bc, lo, hi in (((1, 2, 3), (0, 0, 0), (1, 1, 1)), ((1, 1, 1), (-1, -1, -1), (1, 1, 1))):
        m = I.layered_box_mesh(24, "hybrid8", lo=lo, hi=hi, bc=bc, shape=(20, 19))
        mesh = gks.Mesh(m)
        assert mesh.n_faces >= 60000
        out.append((m, mesh, oracle.Mesh(m, lazy=True)))
    return out


def sample(m, seed, near=None):
    """Cells at every plane of the box (or where `near` holds) and anywhere."""
    x, rng = I.vertex_mean(m), np.random.default_rng(seed)
    lo, hi = np.array(m["lo"]), np.array(m["hi"])
    cells = [rng.choice(len(x), 40, replace=False)]
    masks = [near] if near is not None else \
        [(np.abs(x[:, a] - e[a]) < 0.04) for a in range(3) for e in (lo, hi)]
    for k in masks:
        cells.append(rng.choice(np.nonzero(k)[0], 25 if near is None else 150, replace=False))
    return np.unique(np.concatenate(cells)).astype(np.int32)


UW = np.zeros((6, 3))
UW[4] = (0.2, 0.0, 0.05)
TW = np.array([0, 0, 0, 0, 0.8, 0])


@pytest.mark.parametrize("prm", [dict(tau_model=0), dict(tau_model=1), dict(tau_model=2, mu=2e-3),
                                 dict(tau_model=3, mu=2e-3, T_ref=0.7, mu_pow=0.7),
                                 dict(tau_model=2, mu=2e-3, Pr=0.72)])
def test_boundary_planes_match_oracle(boxes, prm):
    m, mesh, om = boxes[0]
    prm = dict(flux_mode=0, wall_u=UW, wall_T=TW, farfield=(1.0, 0.1, 0.0, 0.3, 1 / 1.4), **prm)
    q = I.primitive_to_conserved(np.ones(mesh.n_cells),
                                 np.tile([0.1, 0.05, 0.2], (mesh.n_cells, 1)),
                                 np.full(mesh.n_cells, 1 / 1.4))
    q = I.perturbed_state(q, seed=50, amp=0.02)
    cells = sample(m, 51)
    Lo, _ = om.residual_cells(oracle.params_vec(**prm), q, 0.002, cells)
    S = gks.Solver(mesh, precision=gks.GKS_PREC_MIXED, **prm)
    L = S.residual(q, 0.002)[0].cpu().numpy()[:, cells].T
    assert np.linalg.norm(L - Lo) < MIXED_TOL_L * np.linalg.norm(Lo)


@pytest.mark.parametrize("tau_model", [0, 1])
def test_positivity_fallback_matches_oracle(boxes, tau_model):
    m, mesh, om = boxes[1]
    x = I.vertex_mean(m)
    q = I.explosion_state(m)
    prm = dict(flux_mode=0, tau_model=tau_model)
    with pytest.raises(gks.GksError) as e:
        gks.Solver(mesh, precision=gks.GKS_PREC_MIXED, **prm).residual(q, 1e-3)
    assert e.value.status == gks.GKS_E_NONPHYSICAL
    cells = sample(m, 52, np.abs(np.sqrt((x * x).sum(1)) - 0.4) < 0.08)
    Lo, _ = om.residual_cells(oracle.params_vec(gp_fallback=1, **prm), q, 1e-3, cells)
    S = gks.Solver(mesh, precision=gks.GKS_PREC_MIXED, gp_fallback=1, **prm)
    L = S.residual(q, 1e-3)[0].cpu().numpy()[:, cells].T
    assert np.linalg.norm(L - Lo) < MIXED_TOL_L * np.linalg.norm(Lo)


def face_f32(x, tau_model, sides, Pr=1.0):
    """The scalar and the packed flux at points x [n, 45] (test_packed_flux_gpu.py)."""
    lib, n = gks.load_library(), len(x)
    P = np.concatenate([[1.4, 2e-3, 0.01, 1.0, 0, tau_model, Pr, 0.9, 0.7], np.zeros(24),
                        np.tile([1.0, 0, 0, 0, 1 / 1.4], 6)])
    f = lib.gks_gp_face_f32_sides if sides else lib.gks_gp_face_f32_pair
    t, o = torch.from_numpy(x).cuda(), torch.zeros((n, 21), device="cuda")
    assert f(P.ctypes.data_as(ctypes.c_void_p), n, ctypes.c_void_p(t.data_ptr()),
             ctypes.c_void_p(o.data_ptr())) == 0
    return o.cpu().numpy()


def points(n, seed):
    rng = np.random.default_rng(seed)
    x = np.zeros((n, 45), dtype=np.float32)
    for s in (0, 20):
        x[:, s:s + 5] = np.array([1.0, 0.2, -0.3, 0.1, 2.6]) + 0.1 * rng.normal(size=(n, 5))
        x[:, s + 5:s + 20] = 0.3 * rng.normal(size=(n, 15))
    nrm = rng.normal(size=(n, 3))
    x[:, 40:43] = nrm / np.linalg.norm(nrm, axis=1, keepdims=True)
    x[:, 43:] = 0.25, 2e-3
    return x


@pytest.mark.parametrize("tau_model,Pr", [(0, 1.0), (1, 1.0), (2, 0.72), (3, 1.0)])
def test_smooth_form_of_small_meshes(tau_model, Pr):
    """Both sides of a point in the two halves, at the bar of test_packed_flux_gpu.py."""
    o = face_f32(points(2048, 56), tau_model, True, Pr).astype(np.float64)
    assert (o[:, 20] == 3).all()
    for h in (slice(0, 5), slice(5, 10)):
        a, b = o[:, 10:20][:, h], o[:, :10][:, h]
        assert (np.abs(a - b) / np.abs(b).max(axis=1, keepdims=True)).max() < 1e-4


@pytest.mark.parametrize("tau_model", [0, 2])
def test_halves_are_independent(tau_model):
    """Points 2 j and 2 j + 1 share a pair: replacing one of them by another point, or by a
    non-physical one, leaves the other's bits, and only the non-physical one is refused."""
    x = points(512, 55)
    ref = face_f32(x, tau_model, False)
    assert (ref[:, 20] == 3).all()
    for odd in (0, 1):
        for bad in (False, True):
            y = x.copy()
            y[odd::2, :43] = np.roll(x[odd::2, :43], 1, axis=0)
            if bad:
                y[odd::2, 24] = -1.0  # the right side's energy
            o = face_f32(y, tau_model, False)
            np.testing.assert_array_equal(o[1 - odd::2], ref[1 - odd::2])
            if bad:
                assert (o[odd::2, 20] == 0).all() and (o[odd::2, 10:20] == 0).all()
            else:
                np.testing.assert_array_equal(o[odd::2], np.roll(ref[odd::2], 1, axis=0))
