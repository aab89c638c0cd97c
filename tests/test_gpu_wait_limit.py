"""How long a wait that runs out keeps the GPU busy."""
import os
import re

import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2006_13631_gb300", "csrc")


@pytest.mark.parametrize("dtype,fv_kernel", [("f32", 4), ("f64", 4), ("f32", 3), ("f32", 2), ("f32", 1)])
def test_wait_limit_is_about_a_second(dtype, fv_kernel):
    """The time of a step whose waits run out after the injected 4096 polls gives
    the time of a poll, and with it that of the limit of ordinary steps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_13631_gb300 import Solver, hlbm_inject_fault
    from paper_2006_13631_gb300.build import build

    build()
    src = open(os.path.join(CSRC, "hlbm_dev.cuh")).read()
    limit = 1 << int(re.search(r"kSpinLimit = 1L << (\d+);", src).group(1))
    w = inputs.workload("lamina-small-f32")
    w.dtype, w.fv_kernel = dtype, fv_kernel
    s = Solver(w)
    s.step(3)
    torch.cuda.synchronize()
    hlbm_inject_fault(s.h, 1, s.info()["n_tiles"] // 2)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    e[0].record()
    s.step(1)
    e[1].record()
    torch.cuda.synchronize()
    assert s.status & 32
    assert e[0].elapsed_time(e[1]) * 1e-3 * limit / 4096 < 1.5
    s.close()
