"""Paths of the FV kernels chosen by size, precision and patch, at the sizes
where they can go wrong, against the oracle or against the general path."""
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


def _case(dtype, mesh_args, n_sub=24, L=20.0, n=128):
    A, om, tau = inputs.harmonic_params(L, 0.5, 100.0)
    w = inputs.Workload("paths", n, n - 12, L, L / 50.0, 0.5 * n + 0.3, 0.5 * n - 5.8, tau, n_sub,
                        inputs.MOTION_HARMONIC, A=A, omega=om, dtype=dtype, noise_amp=1e-6, seed=3, mesh_args=mesh_args)
    w.n_sub = inputs.stable_substeps(w.mesh(), tau - 0.5, minimum=n_sub)
    return w


SMALL = dict(n_L=17, n_T=2, n_layers=9, h1=0.3, d_out=4.0)
MEDIUM = dict(n_L=110, n_T=2, n_layers=20, h1=0.15, d_out=4.0)
LARGE = dict(n_L=200, n_T=4, n_layers=45, h1=0.08, d_out=4.0)


@pytest.mark.parametrize("dtype,tol", [("f64", 1e-9), ("f32", 2e-3)])
@pytest.mark.parametrize("mesh_args", [SMALL, MEDIUM], ids=["small", "medium"])
def test_adjoint_from_recorded_and_rerecorded_substeps(mesh_args, dtype, tol):
    """The adjoint whose forward steps record the FV sub-steps (deep tiles) and the
    one that records them again in global memory (global-memory kernel): the same
    gradient up to the order of the atomic sums (FP64: 1e-16 per term over 1e6
    terms, cancelling; FP32: 1e-7 likewise)."""
    from paper_2006_13631_gb300 import hlbm as H

    H.use_torch_allocator()
    w = _case(dtype, mesh_args)
    got = []
    for kern in (0, 1):
        w.fv_kernel = kern
        grid, patch, motion = H.workload_inputs(w)
        got.append(H.hlbm_theta_adjoint(grid, patch, w.tau_s, motion, 9, 0.0, 8.5 / w.period, 1.0, 0.5, 4))
    (t0, g0, _, _), (t1, g1, _, _) = got
    assert t0 == t1
    assert np.abs(g0 - g1).max() <= tol * np.abs(g1).max()


def test_adjoint_of_a_patch_of_more_nodes_than_resident_quads():
    """The reverse pass that strides over the nodes with grid barriers, against
    central differences of the CUDA path in tau_s (no node moves; FP64, the
    quotient's error is the square of the 1e-5 step and 1e-13 / 1e-5)."""
    from paper_2006_13631_gb300 import hlbm as H

    H.use_torch_allocator()
    w = _case("f64", LARGE)
    assert w.mesh().n_nodes > 152 * 4 * 24
    mesh, rho = w.mesh(), w.rho_init()
    steps, fit = 6, 5.5 / w.period
    grid, patch, motion = H.workload_inputs(w, mesh, rho)
    _, g, _, _ = H.hlbm_theta_adjoint(grid, patch, w.tau_s, motion, steps, 0.0, fit, 1.0, 0.5, 3)
    L = []
    for sign in (-1.0, 1.0):
        h = H.hlbm_create(grid, patch, w.tau_s * (1.0 + sign * 1e-5), motion, 0)
        H.hlbm_step(h, steps)
        re, im, _ = H.hlbm_gamma_window(h, w.omega, 0.0, fit)
        L.append(re + 0.5 * im)
        H.hlbm_destroy(h)
    quotient = (L[1] - L[0]) / (2e-5 * w.tau_s)
    assert abs(g[2] - quotient) <= 1e-5 * abs(quotient)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("mesh_args", [SMALL, MEDIUM, LARGE], ids=["small", "medium", "large"])
def test_outer_node_sums_agree_bit_for_bit(mesh_args, dtype):
    """outer_fv: the deep tiles (automatic choice, every exchange interval) and the
    shared- and global-memory kernels run the same arithmetic."""
    from paper_2006_13631_gb300 import Solver, hlbm_set_fv_depth

    w = _case(dtype, mesh_args, n_sub=25)
    w.outer_fv = 1
    mesh, rho = w.mesh(), w.rho_init()
    got = []
    for kern in (1, 2, 0):
        w.fv_kernel = kern
        try:
            s = Solver(w, mesh=mesh, rho_init=rho)
        except Exception:
            assert kern == 2 and dtype == "f64"  # tiles too large for the shared-memory kernel
            continue
        if kern == 0 and mesh_args is not LARGE:
            assert s.info()["fv_kernel"] == 4
        for depth in (1, 2, 3, 4) if s.info()["fv_kernel"] == 4 else (0, 0, 0, 0):
            if depth:
                hlbm_set_fv_depth(s.h, depth)
            s.step(3)
        assert s.status == 0
        got.append(tuple(s.fields()) + (s.patch_f(), s.force()[1]))
        s.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)


# the sizes next to each line of the dispatch: FP64 tiles of 18 and of 19 nodes
# (exchange interval 2 and 1), of at most 160 and of 161 (four lanes per node or
# one), FP32 tiles of few computed slots and of more than 384 (two lanes or one)
@pytest.mark.parametrize("dtype,n_L,n_layers,h1,nodes,depth", [
    ("f64", 75, 14, 0.3, 2716, 2), ("f64", 78, 14, 0.25, 2748, 1), ("f64", 240, 40, 0.08, None, 1),
    ("f64", 250, 40, 0.08, 24380, 1), ("f32", 74, 13, 0.3, 2436, 2), ("f32", 400, 50, 0.06, 46600, 2),
    ("f32", 420, 55, 0.06, 54612, 2)])
def test_deep_forms_agree_bit_for_bit(dtype, n_L, n_layers, h1, nodes, depth):
    """The forms of the deep kernel and the global-memory kernel run the same
    arithmetic: equal fields after a few steps."""
    from paper_2006_13631_gb300 import Solver

    w = _case(dtype, dict(n_L=n_L, n_T=2, n_layers=n_layers, h1=h1, d_out=4.0), n_sub=25)
    mesh, rho = w.mesh(), w.rho_init()
    assert nodes is None or mesh.n_nodes == nodes
    got = []
    for kern in (1, 0):
        w.fv_kernel = kern
        s = Solver(w, mesh=mesh, rho_init=rho)
        if kern == 0:
            assert s.info()["fv_kernel"] == 4
            if s.info()["n_tiles"] == 152:
                assert s.info()["fv_depth"] == depth
        s.step(4)
        assert s.status == 0
        got.append(tuple(s.fields()) + (s.patch_f(), s.force()[1]))
        s.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
