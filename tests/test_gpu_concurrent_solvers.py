"""Solvers stepped at the same time, each on a stream of its own by a thread of its own."""
import threading
import time

import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_overlap_leaves_room_for_other_solvers():
    """Eight solvers of a few tiles each: every one gives the bits of a solver
    stepped alone, and together they take no longer with the overlap than without
    (by more than half; their launches would run one after another, 2.3 times as
    long, if each took every SM)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_13631_gb300 import Solver, hlbm_set_overlap
    from paper_2006_13631_gb300.build import build

    build()
    A, om, tau = inputs.harmonic_params(20.0, 0.5, 200.0, tau=0.55)
    w = inputs.Workload("together", 128, 128, 20.0, 0.4, 64.3, 64.2, tau, 24, inputs.MOTION_HARMONIC, A=A, omega=om,
                        dtype="f32", noise_amp=1e-6, seed=3,
                        mesh_args=dict(n_L=17, n_T=2, n_layers=9, h1=0.3, d_out=4.0))
    mesh, rho = w.mesh(), w.rho_init()
    alone = Solver(w, mesh=mesh, rho_init=rho)
    alone.step(3 * 300)
    streams = [torch.cuda.Stream() for _ in range(8)]
    seconds = []
    for on in (True, False):
        solvers = [Solver(w, mesh=mesh, rho_init=rho, stream=st.cuda_stream) for st in streams]
        for s in solvers:
            hlbm_set_overlap(s.h, on)
        best = 1e9
        for _ in range(3):
            threads = [threading.Thread(target=s.step, args=(300,)) for s in solvers]
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        seconds.append(best)
        for s in solvers:
            assert s.status == 0
            for a, b in zip(tuple(s.fields()) + s.force(), tuple(alone.fields()) + alone.force()):
                assert np.array_equal(a, b)
            s.close()
    assert seconds[0] <= 1.5 * seconds[1], seconds
