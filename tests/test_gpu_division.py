"""The sweeps' FP32 quotient and reciprocal (div_face, rcp_face) against exact
values and CUDA's own division: every mantissa at several exponents, and random
operands over the whole range they are written for.  Bound (derived beside the
functions): a relative error of 2^-24 + 2^-44, so at most one unit in the last
place from the correctly rounded result."""
import ctypes as C
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BOUND = 2.0 ** -24 + 2.0 ** -44 + 2.0 ** -51      # the last term: the check's own rounding in FP64

SOURCE = r"""
#include "fw_kernels.cuh"
namespace {
__global__ void k_divide(const float *c, const float *x, float *q, float *r, float *q0, float *r0, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = fwgb::div_face(c[i], x[i]);
    r[i] = fwgb::rcp_face(x[i]);
    q0[i] = __fdiv_rn(c[i], x[i]);
    r0[i] = __frcp_rn(x[i]);
}
}
extern "C" int divide(const float *h, float *out, int n)   // h: c, x; out: four arrays
{
    float *d = nullptr;
    const size_t b = n * sizeof(float);
    if (cudaMalloc(&d, 6 * b) != cudaSuccess) return 1;
    int rc = cudaMemcpy(d, h, 2 * b, cudaMemcpyHostToDevice) != cudaSuccess;
    if (!rc) {
        k_divide<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * (size_t)n, d + 3 * (size_t)n, d + 4 * (size_t)n,
                                           d + 5 * (size_t)n, n);
        rc = cudaMemcpy(out, d + 2 * (size_t)n, 4 * b, cudaMemcpyDeviceToHost) != cudaSuccess;
    }
    cudaFree(d);
    return rc;
}
"""


@pytest.fixture(scope="module")
def divide(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2606_11103_gb300 import build
    d = tmp_path_factory.mktemp("divide")
    (d / "divide.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O3", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
                    "-shared", "-I" + build.CSRC, str(d / "divide.cu"), "-o", str(d / "divide.so"), "-lcudart"],
                   check=True)
    fn = C.CDLL(str(d / "divide.so")).divide

    def run(c, x):
        h = np.ascontiguousarray(np.stack([c, x]), np.float32)
        out = np.empty((4, h.shape[1]), np.float32)
        assert fn(h.ctypes.data_as(C.c_void_p), out.ctypes.data_as(C.c_void_p), h.shape[1]) == 0
        return h[0], h[1], out

    return run


def check(c, x, out):
    q, r, q0, r0 = out
    c64, x64 = c.astype(np.float64), x.astype(np.float64)
    err_q = np.abs(q.astype(np.float64) * x64 / c64 - 1).max()
    err_r = np.abs(r.astype(np.float64) * x64 - 1).max()
    ulp = max(int(np.abs(a.view(np.int32).astype(np.int64) - b.view(np.int32)).max()) for a, b in ((q, q0), (r, r0)))
    print("relative error c/x %.3f, 1/x %.3f of 2^-24; %.2e, %.2e not correctly rounded" %
          (err_q * 2 ** 24, err_r * 2 ** 24, np.mean(q != q0), np.mean(r != r0)))
    assert err_q <= BOUND and err_r <= BOUND and ulp <= 1


@pytest.mark.parametrize("exponent", [-100, -50, 0, 9, 10, 33, 50, 99])
@pytest.mark.parametrize("c", [-1.0, -2.1343e-8, 3.0e-9])
def test_every_mantissa(divide, exponent, c):
    x = np.arange(1 << 23, dtype=np.int32) + np.int32((exponent + 127) << 23)
    x = x.view(np.float32)
    check(*divide(np.full(x.size, c * 2.0 ** (exponent // 2)), x))       # both operands and the quotient in range


def test_random_operands(divide):
    rng = np.random.default_rng(0)
    x = np.exp2(rng.uniform(-100, 100, 1 << 22))
    c = np.exp2(rng.uniform(-100, 100, 1 << 22)) * rng.choice([-1, 1], 1 << 22)
    keep = np.abs(np.log2(np.abs(c / x))) < 100
    check(*divide(c[keep], x[keep]))
