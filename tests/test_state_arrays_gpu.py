"""Caller arrays: the kernels read and write aligned device arrays in place and take everything
else through staging copies; the results are the same bits either way. And the time-step bound,
which evaluates in FP64 only the cells that an FP32 estimate leaves open, against the oracle over
states far from unity."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2203_09047_gb300 as gks  # noqa: E402
from paper_2203_09047_gb300 import build, inputs as I  # noqa: E402


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    m = I.layered_box_mesh(8, "hybrid8", shape=(7, 5))
    return m, oracle.Mesh(m), I.perturbed_state(I.advection_state(m), seed=61, amp=0.03)


class Array:
    """A [5, n] float64 array in one kind of memory: its address and its values."""

    def __init__(self, kind, n, q=None):
        self.kind, self.n = kind, n
        q = np.zeros((5, n)) if q is None else q
        raw = torch.from_numpy(np.ascontiguousarray(q).reshape(-1).view(np.uint8).copy())
        if kind == "device":
            self.t = raw.cuda()
        elif kind == "pinned":
            self.t = raw.pin_memory()
        elif kind == "host":
            self.t = raw
        else:  # device memory 4 bytes off a value's alignment
            self.t = torch.zeros(raw.numel() + 8, dtype=torch.uint8, device="cuda")
            self.t[4:4 + raw.numel()] = raw.cuda()
        self.ptr = self.t.data_ptr() + (4 if kind == "unaligned" else 0)

    def values(self):
        b = self.t[4:-4] if self.kind == "unaligned" else self.t
        return b.cpu().numpy().view(np.float64).reshape(5, self.n)


@pytest.mark.parametrize("prec", [gks.GKS_PREC_FP64, gks.GKS_PREC_MIXED])
@pytest.mark.parametrize("kind", ["pinned", "host", "unaligned"])
def test_staged_arrays_give_the_same_bits(setup, kind, prec):
    m, om, Q = setup
    lib = gks.load_library()
    S = gks.Solver(m, precision=prec, min_stencil=18, flux_mode=1, tau_model=2, mu=1e-3)
    g = I.normal_directions(Q.shape, 2, 62)
    out = {}
    for k in ("device", kind):
        q, gl, glt = Array(k, S.n_cells, Q), Array(k, S.n_cells, g[0]), Array(k, S.n_cells, g[1])
        o = [Array(k, S.n_cells) for _ in range(4)]
        P = ctypes.c_void_p
        assert lib.gks_residual(S.h, P(q.ptr), 0.01, P(o[0].ptr), P(o[1].ptr)) == 0
        assert lib.gks_residual_vjp(S.h, P(q.ptr), 0.01, P(gl.ptr), P(glt.ptr), P(o[2].ptr)) == 0
        assert lib.gks_set_state(S.h, P(q.ptr)) == 0
        assert lib.gks_step(S.h, 0.005, 1) == 0
        assert lib.gks_get_state(S.h, P(o[3].ptr)) == 0
        torch.cuda.synchronize()
        out[k] = [x.values().copy() for x in o]
    for a, b in zip(out["device"], out[kind]):
        np.testing.assert_array_equal(a, b)
        assert np.abs(a).max() > 0


@pytest.mark.parametrize("prec", [gks.GKS_PREC_FP64, gks.GKS_PREC_MIXED, gks.GKS_PREC_MIXED_FP64UPD])
@pytest.mark.parametrize("rho,p,mach,power", [(1.0, 1.0, 1.0, 0), (1.2, 1e5, 0.1, 0),
                                              (1e-4, 10.0, 30.0, 1), (1e-20, 1e-3, 2.0, 0),
                                              (1e20, 1e3, 0.5, 0)])
def test_time_step_bound(setup, prec, rho, p, mach, power):
    m, om, _ = setup
    rng = np.random.default_rng(63)
    n = om.n_cells
    r = rho * (1 + 0.3 * rng.random(n))
    pr = p * (1 + 0.3 * rng.random(n))
    u = mach * np.sqrt(1.4 * p / rho) * rng.normal(size=(n, 3)) / 2
    Q = I.primitive_to_conserved(r, u, pr)
    prm = dict(mu=1e-3 * rho, tau_model=3 if power else 2, T_ref=p / rho, mu_pow=0.7)
    S = gks.Solver(m, precision=prec, **prm)
    S.set_state(Q)
    ref = om.max_dt(oracle.params_vec(**prm), np.ascontiguousarray(Q), 0.5)
    # FP64: the oracle's formula up to rounding; the float-float state carries 2^-47, which the
    # pressure of the fastest gas (kinetic over internal energy up to 500) raises to 4e-12
    assert abs(S.max_dt(0.5) - ref) <= (1e-13 if prec == gks.GKS_PREC_FP64 else 1e-11) * ref


@pytest.mark.parametrize("prec", [gks.GKS_PREC_FP64, gks.GKS_PREC_MIXED, gks.GKS_PREC_MIXED_FP64UPD])
def test_time_step_bound_reports_nonphysical_states(setup, prec):
    m, om, Q = setup
    for row, value in ((0, -1.0), (4, 1e-3), (4, np.nan)):
        bad = Q.copy()
        bad[row, -1] = value
        S = gks.Solver(m, precision=prec)
        S.set_state(bad)
        with pytest.raises(gks.GksError) as e:
            S.max_dt(0.5)
        assert e.value.status == gks.GKS_E_NONPHYSICAL
