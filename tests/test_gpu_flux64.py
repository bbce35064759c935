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


def test_reciprocals_over_all_of_fp64(run):
    """recip is the correctly rounded 1 / x and recip_sqrt CUDA's rsqrt (one
    unit in the last place), for subnormals, the largest numbers, zero and
    infinity too"""
    x = np.concatenate([[0.0, np.inf, 5e-324, 1e-310, 2.3e-308, 1.7e308, 1.0, 3.0],
                        np.ldexp(np.random.default_rng(1).uniform(1, 2, 4096), np.arange(4096) % 2040 - 1040)])
    r, q = run("o[0] = recip(x[0]); o[1] = recip_sqrt(x[0]);", x[:, None], 2).T
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / x
        root = (1.0 / np.sqrt(x.astype(np.longdouble))).astype(np.float64)
    assert np.array_equal(r, want)
    f = np.isfinite(root)
    assert np.array_equal(q[~f], root[~f])
    assert (np.abs(q[f] - root[f]) <= np.spacing(root[f])).all()


def test_comparisons_on_bit_patterns(run):
    """-0 lies below +0 in less() and counts as negative; no zero is positive"""
    v = [-np.inf, -3.0, -1e-320, -0.0, 0.0, 1e-320, 3.0, np.inf]
    ab = np.array(list(itertools.product(range(8), range(8))))
    val = np.array(v)[ab]
    got = run("o[0] = less(x[0], x[1]); o[1] = below_abs(x[0], x[1]); o[2] = negative(x[0]); o[3] = positive(x[0]);", val, 4)
    assert np.array_equal(got[:, 0], ab[:, 0] < ab[:, 1])
    assert np.array_equal(got[:, 1], np.abs(val[:, 0]) < np.abs(val[:, 1]))
    assert np.array_equal(got[:, 2], ab[:, 0] <= 3)
    assert np.array_equal(got[:, 3], ab[:, 0] >= 5)


GAM = 1.4


def _states(n, seed):
    """left and right (rho, u, v, p): mixed, both supersonic one way or the
    other, one side or both without a positive pressure, exactly sonic, and
    densities and pressures so small that gamma p rho is subnormal"""
    rng = np.random.default_rng(seed)
    s = np.empty((n, 2, 4))
    s[:, :, 0] = 10.0 ** rng.uniform(-2, 1, (n, 2))
    s[:, :, 3] = 10.0 ** rng.uniform(-2, 2, (n, 2))
    s[:, :, 1:3] = rng.normal(size=(n, 2, 2)) * 10.0 ** rng.uniform(-1, 1, (n, 1, 1))
    k = np.arange(n) % 8
    c = np.sqrt(GAM * s[:, :, 3] / s[:, :, 0]).max(axis=1)
    s[k == 1, :, 1] = c[k == 1, None] * rng.uniform(1.5, 4, (np.count_nonzero(k == 1), 2))
    s[k == 2, :, 1] = -c[k == 2, None] * rng.uniform(1.5, 4, (np.count_nonzero(k == 2), 2))
    s[k == 3, 0, 3] *= -rng.uniform(0, 1, np.count_nonzero(k == 3))
    s[k == 4, 1, 3] = 0.0
    s[n // 2:][k[n // 2:] == 5, :, 3] *= -1.0
    tiny = k == 6
    s[tiny, :, 0] *= 1e-158
    s[tiny, :, 3] *= 1e-153
    s[tiny, :, 1:3] *= 300.0  # speeds of the order of the speed of sound
    return s


def _plain_hll(s):
    """HLL by its definition; a side without a sound speed leaves the speeds to the other"""
    q = s.astype(np.longdouble)
    r, u, v, p = np.moveaxis(q, 2, 0)
    E = p / (q.dtype.type(GAM) - 1) + r * (u * u + v * v) / 2
    g = np.longdouble(GAM)
    c = np.where(p > 0, np.sqrt(np.where(p > 0, g * p / r, 1)), np.nan)
    sL, sR = np.fmin.reduce(u - c, axis=1), np.fmax.reduce(u + c, axis=1)
    U = np.stack([r, r * u, r * v, E], axis=2)
    F = U * u[..., None]
    F[..., 1] += p
    F[..., 3] += p * u
    a, b = sL[:, None], sR[:, None]
    mid = (b * F[:, 0] - a * F[:, 1] + a * b * (U[:, 1] - U[:, 0])) / (b - a)
    f = np.where(a >= 0, F[:, 0], np.where(b <= 0, F[:, 1], mid))
    w = np.nanmax(np.abs(u) + np.where(np.isnan(c), 0, c), axis=1)[:, None]
    R = r.sum(axis=1)
    m = (r * (np.abs(u) + np.abs(v))).sum(axis=1)
    P = np.abs(p).sum(axis=1)
    size = np.stack([w[:, 0] * R, w[:, 0] * m + P, w[:, 0] * m, w[:, 0] * (np.abs(E).sum(axis=1) + P)], axis=1)
    return f, size


def _plain_ausm(s):
    """AUSM+ by its definition (interface speed min of a*^2 / max(a*, +-u); a
    side without a critical speed leaves it to the other)"""
    q = s.astype(np.longdouble)
    r, u, v, p = np.moveaxis(q, 2, 0)
    g = np.longdouble(GAM)
    H = g / (g - 1) * p / r + (u * u + v * v) / 2
    a2 = 2 * (g - 1) / (g + 1) * H
    ast = np.where(a2 > 0, np.sqrt(np.abs(a2)), np.nan)
    un = np.stack([u[:, 0], -u[:, 1]], axis=1)
    a = np.fmin.reduce(ast * ast / np.where(np.isnan(ast), np.nan, np.maximum(ast, un)), axis=1)
    M = u / a[:, None]
    sg = np.array([1, -1], np.longdouble)
    t = M * M - 1
    mach = np.where(np.abs(M) >= 1, (M + sg * np.abs(M)) / 2, sg * ((M + sg) ** 2 / 4 + t * t / 8))
    pres = np.where(np.abs(M) >= 1, (1 + sg * np.sign(M)) / 2,
                    (M + sg) ** 2 / 4 * (2 - sg * M) + sg * 3 * M * t * t / 16)
    mh = a * mach.sum(axis=1)
    ph = (pres * p).sum(axis=1)
    fl, fr = np.where(mh > 0, mh, 0) * r[:, 0], np.where(mh < 0, mh, 0) * r[:, 1]
    f = np.stack([fl + fr, fl * u[:, 0] + fr * u[:, 1] + ph, fl * v[:, 0] + fr * v[:, 1], fl * H[:, 0] + fr * H[:, 1]], axis=1)
    f[np.isnan(a)] = np.nan
    w = a + np.abs(u).max(axis=1)
    R = r.sum(axis=1)
    m = (r * (np.abs(u) + np.abs(v))).sum(axis=1)
    P = np.abs(p).sum(axis=1)
    h = g / (g - 1) * np.abs(p) / r + (u * u + v * v) / 2
    size = np.stack([w * R, w * m + P, w * m, w * (r * h).sum(axis=1)], axis=1)
    return f, size


@pytest.mark.parametrize("name,plain,roundings", [("hll64", _plain_hll, 64), ("ausm_plus64", _plain_ausm, 128)])
def test_fluxes_equal_their_definitions(run, name, plain, roundings):
    """HLL: the wave speeds carry at most 4 roundings of W = max(|u| + c), and
    s_R - s_L >= W where both sides enter, so the weights carry 16 and the
    speeds w (u_n - s), of size 2 W, some 50 roundings of W.  AUSM+: the Mach
    numbers carry 6, the splits (slopes up to 2) and their sum 40, the mass
    flux 50 and the pressure 12.  Each is doubled for the products that follow.
    Where gamma p rho is subnormal, HLL's sound speeds also carry its rounding to
    a multiple of 2^-1074."""
    n = 1 << 15
    s = _states(n, 5)
    body = """
    Grid g{};
    g.phys[0] = %r;
    g.igm = 1.0 / (g.phys[0] - 1.0);
    g.cstar = 2.0 * (g.phys[0] - 1.0) / (g.phys[0] + 1.0);
    %s<2, 4>(g, 0, x, x + 4, o);
    double y[8] = {x[0], x[2], x[1], x[3], x[4], x[6], x[5], x[7]}; // the same along y
    %s<2, 4>(g, 1, y, y + 4, o + 4);
    """ % (GAM, name, name)
    got = run(body, s.reshape(n, 8), 8)
    want, size = plain(s)
    nan = np.isnan(want.astype(np.float64)).any(axis=1)
    assert np.isnan(got[nan][:, [0, 3]]).all()
    assert 0 < np.count_nonzero(nan) < n // 8
    x = GAM * s[:, :, 0] * s[:, :, 3]
    sub = 4.0 * 2.0 ** -1074 / np.where(x > 0, x, np.inf).min(axis=1) if name == "hll64" else np.zeros(n)
    tol = (roundings * 2.0 ** -53 + sub)[~nan, None] * size[~nan]
    for f in (got[:, :4], got[:, [4, 6, 5, 7]]):
        err = np.abs(f[~nan] - want[~nan]) / size[~nan]
        print(name, "largest error in units of 2^-53:", float(err.max() * 2.0 ** 53))
        assert (np.abs(f[~nan] - want[~nan]) <= tol).all()
