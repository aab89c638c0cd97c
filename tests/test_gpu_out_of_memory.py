"""What the library does without when the device has no room for it (its own
cudaMalloc, no allocator installed)."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def own_allocator():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_13631_gb300 import _native as N
    from paper_2006_13631_gb300 import hlbm as H
    from paper_2006_13631_gb300.build import build

    build()
    N.load().hlbm_set_allocator(N.ALLOC_FN(), N.FREE_FN(), None)
    torch.cuda.empty_cache()
    yield H
    if H._callbacks is not None:
        N.load().hlbm_set_allocator(H._callbacks[0], H._callbacks[1], None)


def test_adjoint_whose_records_do_not_fit(own_allocator):
    """The FV records of a segment (some 7 GB here) are optional: with 3 GB free
    they are made again step by step, with the same gradient up to the order of
    the atomic sums (1e-16 per term over 1e6 terms, cancelling)."""
    H = own_allocator
    w = inputs.workload("lamina-256-f64")
    w.omega *= 1.0131
    w.n_sub = 400
    mesh, steps = w.mesh(), 48
    assert 3 << 30 < 16 * 8 * w.n_sub * mesh.n_nodes * steps <= 8 << 30
    grid, patch, motion = H.workload_inputs(w, mesh)

    def gradient():
        return H.hlbm_theta_adjoint(grid, patch, w.tau_s, motion, steps, 0.5, 1.25, 1.0, 0.5, steps)[:2]

    t0, g0 = gradient()
    held = torch.empty(torch.cuda.mem_get_info()[0] - (3 << 30), dtype=torch.uint8, device="cuda")
    try:
        t1, g1 = gradient()
    finally:
        del held
        torch.cuda.empty_cache()
    assert t0 == t1
    assert np.abs(g0 - g1).max() <= 1e-9 * np.abs(g0).max()
