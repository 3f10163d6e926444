"""Solvers of their own in several host threads: the launch of one does not depend on the shared
memory that another asked for its kernels, so meshes with different stencils can be driven at the
same time."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2203_09047_gb300 as gks  # noqa: E402
from paper_2203_09047_gb300 import build, inputs as I  # noqa: E402


def test_two_meshes_in_two_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gks.load_library()
    jobs = []
    for min_stencil in (0, 40, 52):  # three sizes of shared memory of the same kernels
        m = I.layered_box_mesh(5, "hex", shape=(5, 4))
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            S = gks.Solver(m, stream=st, min_stencil=min_stencil)
            Q = torch.from_numpy(I.perturbed_state(I.advection_state(m), seed=7)).cuda()
            g = torch.ones_like(Q)
            ref = (*S.residual(Q, 0.01), S.residual_vjp(Q, 0.01, g, g))
        st.synchronize()
        jobs.append((st, S, Q, g, ref))
    errors = []

    def work(st, S, Q, g, ref):
        try:
            with torch.cuda.stream(st):
                for _ in range(1500):
                    out = (*S.residual(Q, 0.01), S.residual_vjp(Q, 0.01, g, g))
            st.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(out, ref))
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
