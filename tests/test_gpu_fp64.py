"""The FP64 helpers of the fluxes against extended precision.  recip and
recip_sqrt improve the hardware's approximation by one third-order Householder
step; with an approximation of 18 bits or better the terms left out are below
2^-54, and the roundings (the last multiply-add, and for recip_sqrt the
product x y, which enters with weight 1/2) add at most 2^-53 + 2^-54: the
relative error stays below 2^-52.  The limiter and the comparisons on bit
patterns must equal the arithmetic ones exactly."""
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include <vector>
#include "mrlt_impl.cuh"
using namespace mrlt;
__global__ void k(const double* x, const double* z, double* o, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    o[i] = recip(x[i]);
    o[n + i] = recip_sqrt(fabs(x[i]));
    o[2 * n + i] = minmod(x[i], z[i]);
    o[3 * n + i] = less(x[i], z[i]);
}
int main(int, char** a)
{
    const int n = atoi(a[1]);
    std::vector<double> h(6 * (size_t)n);
    FILE* f = fopen(a[2], "rb");
    if (!f || fread(h.data(), 8, 2 * (size_t)n, f) != 2 * (size_t)n) return 1;
    fclose(f);
    double* d = nullptr;
    if (cudaMalloc(&d, 48 * (size_t)n) != cudaSuccess) return 2;
    cudaMemcpy(d, h.data(), 16 * (size_t)n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * (size_t)n, n);
    if (cudaMemcpy(h.data(), d + 2 * (size_t)n, 32 * (size_t)n, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    f = fopen(a[3], "wb");
    fwrite(h.data(), 8, 4 * (size_t)n, f);
    return fclose(f);
}
"""


def test_fp64_helpers(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_08717_gb300 import build as b
    (tmp_path / "t.cu").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.check_call([b._nvcc()] + b.ARCH + ["-O3", "-std=c++17", "-I" + b.CSRC, "-o", exe, str(tmp_path / "t.cu")])
    rng = np.random.default_rng(0)
    n = 1 << 20
    x = np.ldexp(rng.uniform(1, 2, n), rng.integers(-900, 900, n)) * rng.choice([-1.0, 1.0], n)
    x[: n // 2] = rng.uniform(0.01, 100.0, n // 2)
    z = np.where(rng.random(n) < 0.1, x, np.roll(x, 1) * rng.choice([-1.0, 1.0], n))
    z[:1000] = 0.0
    np.concatenate([x, z]).tofile(tmp_path / "in")
    subprocess.check_call([exe, str(n), str(tmp_path / "in"), str(tmp_path / "out")])
    r, q, m, lt = np.fromfile(tmp_path / "out").reshape(4, n)
    X = x.astype(np.longdouble)
    assert np.finfo(np.longdouble).nmant >= 63
    assert np.abs(r.astype(np.longdouble) * X - 1).max() <= 2.0 ** -52
    assert np.abs(q.astype(np.longdouble) * np.sqrt(np.abs(X)) - 1).max() <= 2.0 ** -52
    same = np.signbit(x) == np.signbit(z)
    assert np.array_equal(m, np.where(same, np.where(np.abs(x) < np.abs(z), x, z), 0.0))
    assert np.array_equal(lt, (x < z).astype(float))
