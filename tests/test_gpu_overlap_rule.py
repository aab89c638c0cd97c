"""The lattice on the SMs without a tile: taken only where it ends in time."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ms(s, steps=40):
    s.step(10)
    best = 1e9
    for _ in range(3):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        s.step(steps)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) / steps)
    return best


# beside patches of 17 and of 40 tiles: lattices that the idle SMs stream within
# the sub-steps, and lattices for which they would take two to three times as long
@pytest.mark.parametrize("n,mesh_args,L,n_sub", [
    (512, dict(n_L=40, n_layers=10, h1=0.3), 24.0, 24), (2048, dict(n_L=64, n_layers=15, h1=0.25), 32.0, 64),
    (2896, dict(n_L=64, n_layers=15, h1=0.25), 32.0, 24), (4096, dict(n_L=40, n_layers=10, h1=0.3), 24.0, 24),
    (4096, dict(n_L=64, n_layers=15, h1=0.25), 32.0, 64)])
def test_overlap_changes_no_bit_and_costs_no_time(n, mesh_args, L, n_sub):
    """Equal fields with the overlap on and off, and a step no slower with it on
    (by more than a quarter: runs of one side differ by 2 %)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_13631_gb300 import Solver, hlbm_set_overlap
    from paper_2006_13631_gb300.build import build

    build()
    A, om, tau = inputs.harmonic_params(L, 0.5, 200.0, tau=0.53)
    w = inputs.Workload("overlap", n, n, L, L / 50.0, 0.5 * n + 0.3, 0.5 * n + 0.2, tau, n_sub, inputs.MOTION_HARMONIC,
                        A=A, omega=om, dtype="f32", noise_amp=1e-6, seed=3, mesh_args=dict(n_T=2, d_out=5.0, **mesh_args))
    mesh, rho = w.mesh(), w.rho_init()
    got, ms = [], []
    for on in (True, False):
        s = Solver(w, mesh=mesh, rho_init=rho)
        hlbm_set_overlap(s.h, on)
        s.step(5)
        got.append(tuple(s.fields()) + s.force())
        ms.append(_ms(s))
        assert s.status == 0
        s.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert ms[0] <= 1.25 * ms[1], ms
