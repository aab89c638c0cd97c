"""Parameter sums of the adjoint at one node: each FP32 product goes into the
FP64 sum by itself."""
import ctypes as C
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "adj_node.cuh"
using namespace hk;
// one warp: the factor's term of ffsT, then of adj_psi and adj_kneq at eight outer nodes (quads)
__global__ void k_sums(const float* terms, double* out) {
    float st[12] = {}, lf[9], ls[12];
    for (int i = 0; i < 9; ++i) st[3 + i] = terms[i], lf[i] = 1.0f;
    double lk = 0.0;
    ffsT(st, 1.0f, 0.5f, lf, ls, lk);
    if (threadIdx.x == 0) out[0] = lk;
    Dev<float> d{};
    d.rho0 = 1.0f, d.kneq = 0.5f, d.dt_u = 1.0f;
    const AQuad<float> Q = aquad<float>();
    ANode<float> N{};
    N.valid = true;
    N.kind = HLBM_NODE_OUTER;
    for (int j = 3; j < 6; ++j) N.s0[j] = N.s1[j] = terms[j - 3];  // the lane's pair and the rest one
    ARec<float> r{};
    r.rho = 1.0f;
    float pa, pb, p0, l_inv = 0.0f, l_v = 0.0f;
    double l_kneq = 0.0;
    adj_psi(d, Q, N, r, 0.5f, 0.0f, 0.0f, 1.0f, 1.0f, Q.q == 0 ? 1.0f : 0.0f, pa, pb, p0, l_inv, l_kneq, l_v);
    adj_kneq(N, l_kneq);
    if (threadIdx.x < 2) out[1 + threadIdx.x] = l_kneq;
}
extern "C" int sums(const float* terms, double* out) {
    k_sums<<<1, 32>>>(terms, out);
    return (int)cudaDeviceSynchronize();
}
"""


def test_products_of_mixed_signs(tmp_path):
    """2^25 + 1 - 2^25 = 1 in FP64; an FP32 sum of the three rounds the 1 away."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_13631_gb300 import build as B

    src, lib = tmp_path / "sums.cu", tmp_path / "sums.so"
    src.write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.FLAGS, *B.ARCH, "-I" + B.CSRC, "-shared", str(src), "-o", str(lib)], check=True)
    big = 2.0 ** 25
    terms = torch.tensor([big, 1.0, -big, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0], device="cuda")
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    fn = C.CDLL(os.fspath(lib)).sums
    assert fn(C.c_void_p(terms.data_ptr()), C.c_void_p(out.data_ptr())) == 0
    # lane 0 of a quad has the pair's two products and the rest one, the others the pair's
    assert out.tolist() == [1.0, 1.0, big + 1.0]
