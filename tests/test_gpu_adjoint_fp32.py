"""The FP32 adjoint where its forward run overlaps the lattice with the patch."""
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
    from paper_2006_13631_gb300 import use_torch_allocator

    build()
    use_torch_allocator()


@pytest.mark.parametrize("every", [16, 64])
def test_segment_restored_into_the_window_of_the_last_step(every):
    """The last segment starts in the same window as the step after the run, so
    that the lattice precomputed for that step would fit the restored one by its
    rectangle: it must not be taken for it.  Against the global-memory kernel,
    which precomputes nothing.  The two runs take the same forward bits and add
    the adjoint in other orders: each component within 1e-3, the size of the
    FP32 adjoint's own rounding error on this case (5e-4 against FP64)."""
    from paper_2006_13631_gb300 import hlbm_theta_adjoint, workload_inputs

    w = inputs.workload("lamina-1024-gradient")
    mesh, steps = w.mesh(), 160
    got = []
    for kern in (0, 1):
        w.fv_kernel = kern
        grid, patch, motion = workload_inputs(w, mesh)
        got.append(hlbm_theta_adjoint(grid, patch, w.tau_s, motion, steps, 0.0, (steps - 0.5) / w.period, 1.0, 0.5,
                                      every)[:2])
    (t0, g0), (t1, g1) = got
    assert t0 == t1
    assert (np.abs(g0 - g1) <= 1e-3 * np.abs(g1)).all(), (g0, g1)
