"""Packs of a sweep whose solvers are changed after packing."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_13631_gb300.build import build

    build()


def _workloads(dtype, count=2, n_L=78, n_layers=15):
    out = []
    for k in range(count):
        A, om, tau = inputs.harmonic_params(20.0, 0.2 + 0.05 * k, 500.0, tau=0.6)
        out.append(inputs.Workload(f"p{k}", 192, 192, 20.0, 0.4, 96.3, 96.2, tau, 50, inputs.MOTION_HARMONIC, A=A,
                                   omega=om, dtype=dtype, noise_amp=1e-6, seed=k,
                                   mesh_args=dict(n_L=n_L, n_T=2, n_layers=n_layers, h1=0.25, d_out=4.0)))
    return out


def _same(a, b):
    assert a.status == 0 and b.status == 0
    for x, y in zip(tuple(a.fields()) + a.force(), tuple(b.fields()) + b.force()):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("changed", [1, 2])
def test_depth_set_on_packed_solvers(dtype, changed):
    """hlbm_set_fv_depth rebuilds a solver's tiles as for a launch of its own (in
    FP64 one per SM): the sweep goes on, with the results of solvers stepped alone."""
    from paper_2006_13631_gb300 import Solver, Sweep, hlbm_set_fv_depth

    ws = _workloads(dtype)
    packed, alone = [Solver(w) for w in ws], [Solver(w) for w in ws]
    sw = Sweep(packed)
    assert sw.pack() == 1
    sw.step(2)
    for s in packed[:changed]:
        hlbm_set_fv_depth(s.h, 1)
    sw.step(3)
    for s in alone:
        s.step(5)
    torch.cuda.synchronize()
    for a, b in zip(packed, alone):
        _same(a, b)
    assert sw.pack() == 1
    sw.step(2)
    for s in alone:
        s.step(2)
    torch.cuda.synchronize()
    for a, b in zip(packed, alone):
        _same(a, b)
    sw.close()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_packs_take_the_depth_asked_for(dtype):
    from paper_2006_13631_gb300 import Solver, Sweep, hlbm_set_fv_depth

    ws = _workloads(dtype)
    packed, alone = [Solver(w) for w in ws], [Solver(w) for w in ws]
    for s in packed:
        hlbm_set_fv_depth(s.h, 3)
    sw = Sweep(packed)
    assert sw.pack() == 1
    assert [s.info()["fv_depth"] for s in packed] == [3, 3]
    sw.step(3)
    for s in alone:
        s.step(3)
    torch.cuda.synchronize()
    for a, b in zip(packed, alone):
        _same(a, b)
    sw.close()


def test_fv_time_of_a_pack():
    """Several timed steps of a packed sweep: every solver of the pack gets the
    time of the shared launches."""
    from paper_2006_13631_gb300 import Solver, Sweep

    solvers = [Solver(w) for w in _workloads("f32")]
    sw = Sweep(solvers)
    assert sw.pack() == 1
    ms = sw.fv_time(3)
    assert ms[0] > 0 and ms[0] == ms[1]
    assert all(s.status == 0 and s.info()["time"] == 3 for s in solvers)
    sw.close()


def test_depth_set_on_one_solver_of_a_tensor_memory_pack():
    """Five solvers whose tiles are too large for the deep kernel: the changed one
    has the deep kernel's tables afterwards and the others do not."""
    from paper_2006_13631_gb300 import Solver, Sweep, hlbm_set_fv_depth

    ws = []
    for k in range(5):
        A, om, tau = inputs.harmonic_params(64.0, 0.2 + 0.01 * k, 500.0, tau=0.52)
        ws.append(inputs.Workload(f"t{k}", 256, 192, 64.0, 1.28, 128.3, 96.2, tau, 25, inputs.MOTION_HARMONIC, A=A,
                                  omega=om, dtype="f32", mesh_args=dict(n_L=400, n_T=2, n_layers=50, h1=0.07, d_out=4.0)))
    mesh = ws[0].mesh()
    n_sub = inputs.stable_substeps(mesh, ws[0].tau_s - 0.5, minimum=25)
    for w in ws:
        w.n_sub = n_sub
    packed, alone = [Solver(w, mesh=mesh) for w in ws], [Solver(w, mesh=mesh) for w in ws]
    sw = Sweep(packed)
    assert sw.pack() == 1 and {s.info()["fv_kernel"] for s in packed} == {3}
    sw.step(1)
    hlbm_set_fv_depth(packed[0].h, 2)
    assert [s.info()["fv_kernel"] for s in packed] == [4, 3, 3, 3, 3]
    sw.step(2)
    for s in alone:
        s.step(3)
    torch.cuda.synchronize()
    for a, b in zip(packed, alone):
        _same(a, b)
    sw.close()
