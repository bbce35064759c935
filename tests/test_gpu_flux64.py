"""The FP64 limiter and fluxes on special values and against plain formulas."""
import itertools
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run(body, columns, nout): body computes o[0..nout) from x[0..ncol) of one row"""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_08717_gb300 import build as b

    def go(body, cols, nout):
        d = tmp_path_factory.mktemp("flux64")
        n, nc = cols.shape
        (d / "t.cu").write_text(r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "mrlt_impl.cuh"
using namespace mrlt;
__global__ void k(const double* in, double* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* x = in + (size_t)i * %d;
    double* o = out + (size_t)i * %d;
    %s
}
int main(int, char** a)
{
    const int n = atoi(a[1]);
    std::vector<double> x(%d * (size_t)n), o(%d * (size_t)n);
    FILE* f = fopen(a[2], "rb");
    if (!f || fread(x.data(), 8, x.size(), f) != x.size()) return 1;
    fclose(f);
    double *dx = nullptr, *dd = nullptr;
    if (cudaMalloc(&dx, 8 * x.size()) != cudaSuccess || cudaMalloc(&dd, 8 * o.size()) != cudaSuccess) return 2;
    cudaMemcpy(dx, x.data(), 8 * x.size(), cudaMemcpyHostToDevice);
    k<<<(n + 127) / 128, 128>>>(dx, dd, n);
    if (cudaMemcpy(o.data(), dd, 8 * o.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    f = fopen(a[3], "wb");
    fwrite(o.data(), 8, o.size(), f);
    return fclose(f);
}
""" % (nc, nout, body, nc, nout))
        exe = str(d / "t")
        subprocess.check_call([b._nvcc()] + b.ARCH + ["-O3", "-std=c++17", "-I" + b.CSRC, "-o", exe, str(d / "t.cu")])
        np.ascontiguousarray(cols, np.float64).tofile(d / "in")
        subprocess.check_call([exe, str(n), str(d / "in"), str(d / "out")])
        return np.fromfile(d / "out").reshape(n, nout)

    return go


def test_minmod_special_values(run):
    """every pair of special and plain values: 0 for opposite signs, else the
    smaller magnitude, and b where either is a NaN (a b <= 0 and |a| < |b| are
    false); a zero's sign is free"""
    v = [np.nan, -np.nan, np.inf, -np.inf, 0.0, -0.0, 1.0, -1.0, 2.5, -2.5, 1e-320, -1e-320, 1e-150, 1e300, -1e300]
    ab = np.array(list(itertools.product(v, v)))
    # through a sum, as the limiter's arguments are
    got = run("o[0] = minmod(x[0] + 0.0, x[1] + 0.0);", ab, 1)[:, 0]
    a, b = ab.T
    opposite = np.sign(a) * np.sign(b) <= 0.0
    want = np.where(np.isnan(a) | np.isnan(b), b, np.where(opposite, 0.0, np.where(np.abs(a) < np.abs(b), a, b)))
    assert np.array_equal(got, want, equal_nan=True), [(x, g, w) for x, g, w in zip(ab, got, want) if not (g == w or (g != g and w != w))]
