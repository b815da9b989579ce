"""The device functions that stand in for FP64 operations (they hold this chip's FP64 pipe for 64 cycles an instruction): each
against the operation itself or extended precision, over dense arguments and the edges of its ranges.  Compiled here from the
library's headers."""
import ctypes as C
import os
import struct
import subprocess

import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "exp64.cuh"
enum { F32_TO_F64, F64_TO_F32, SYM_UNIT, COUNT, DIV_COUNT, RCP, RSQRT, EXP, IMAGE_SHORT, IMAGE, KEY, PLAIN_RCP, PLAIN_RSQRT, CAST_DOWN, CAST_UP };
__global__ void apply(int f, long long n, const double* x, const double* y, double p0, double p1, int lo, int hi, double* out) {
    __shared__ SysDesc sd;
    if (threadIdx.x == 0) { sd.box_L = p0; sd.inv_L = p1; sd.img_lo = lo; sd.img_hi = hi; }
    __syncthreads();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double a = x[i], b = y[i];
    double r = 0.0;
    switch (f) {
        case F32_TO_F64: r = f32_to_f64(__int_as_float((int)__double_as_longlong(a))); break;
        case CAST_UP: r = (double)__int_as_float((int)__double_as_longlong(a)); break;
        case F64_TO_F32: r = __longlong_as_double((long long)(unsigned)__float_as_int(f64_to_f32(a))); break;
        case CAST_DOWN: r = __longlong_as_double((long long)(unsigned)__float_as_int((float)a)); break;
        case SYM_UNIT: r = sym_unit((unsigned)__double_as_longlong(a), (unsigned)__double_as_longlong(b)); break;
        case COUNT: r = count_to_f64((int)a); break;
        case DIV_COUNT: r = div_count(a, b, 1.0 / b); break;
        case RCP: r = rcp64(a); break;
        case PLAIN_RCP: r = 1.0 / a; break;
        case RSQRT: r = rsqrt64(a); break;
        case PLAIN_RSQRT: r = 1.0 / sqrt(a); break;
        case EXP: r = exp64_neg(a); break;
        case IMAGE_SHORT: r = mimage64_short(sd, a); break;
        case IMAGE: r = mimage64(a, sd.box_L, sd.inv_L); break;
        case KEY: r = key_value(order_key(a)); if (order_key(a) < order_key(b) != a < b && !(a == 0.0 && b == 0.0)) r = 1e300; break;
    }
    out[i] = r;
}
template <int N> __global__ void sums(const double* x, double* out) {   // x: [32][N]; out: [N]
    double v[N];
    for (int q = 0; q < N; ++q) v[q] = x[threadIdx.x * N + q];
    int first = 0, count = N;
    warp_sums<N>(v, &first, &count);
    if (count == 1) out[first] = v[0];
}
extern "C" int run(int f, long long n, const double* x, const double* y, double p0, double p1, int lo, int hi, double* out, void* st) {
    apply<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)st>>>(f, n, x, y, p0, p1, lo, hi, out);
    return (int)cudaGetLastError();
}
extern "C" int run_sums(int n, const double* x, double* out, void* st) {
    cudaStream_t s = (cudaStream_t)st;
    switch (n) {
        case 1: sums<1><<<1, 32, 0, s>>>(x, out); break;
        case 2: sums<2><<<1, 32, 0, s>>>(x, out); break;
        case 3: sums<3><<<1, 32, 0, s>>>(x, out); break;
        case 6: sums<6><<<1, 32, 0, s>>>(x, out); break;
        case 18: sums<18><<<1, 32, 0, s>>>(x, out); break;
    }
    return (int)cudaGetLastError();
}
"""
NAMES = ("f32_to_f64", "f64_to_f32", "sym_unit", "count", "div_count", "rcp", "rsqrt", "exp", "image_short", "image", "key",
         "plain_rcp", "plain_rsqrt", "cast_down", "cast_up")
N = 1 << 18
LD = np.longdouble


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    d = tmp_path_factory.mktemp("device_functions")
    (d / "f.cu").write_text(SOURCE)
    so = str(d / "f.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", so, str(d / "f.cu"), "-lcudart"], check=True)
    lib = C.CDLL(so)
    vp, dbl = C.c_void_p, C.c_double
    lib.run.argtypes = [C.c_int, C.c_longlong, vp, vp, dbl, dbl, C.c_int, C.c_int, vp, vp]
    lib.run_sums.argtypes = [C.c_int, vp, vp, vp]

    def run(name, x, y=None, L=0.0, lo=0, hi=0):
        x = np.ascontiguousarray(x, np.float64)
        y = np.zeros_like(x) if y is None else np.ascontiguousarray(np.broadcast_to(y, x.shape), np.float64)
        xt, yt = (torch.from_numpy(a.view(np.int64).copy()).cuda() for a in (x, y))   # as bits: NaN payloads stay
        out = torch.empty_like(xt)
        assert lib.run(NAMES.index(name), x.size, xt.data_ptr(), yt.data_ptr(), L, 1.0 / L if L else 0.0, lo, hi, out.data_ptr(),
                       torch.cuda.current_stream().cuda_stream) == 0
        return out.cpu().numpy().view(np.float64)
    run.lib = lib
    return run


def _bits(a):
    return np.ascontiguousarray(a).view(np.int64)


def _doubles(rng, n=N):
    """Random bit patterns (every exponent, NaN and infinities), and the neighbours of powers of two."""
    b = rng.integers(-(1 << 63), (1 << 63) - 1, n, dtype=np.int64)
    p = 2.0 ** np.arange(-1074, 1024)
    edge = np.concatenate([p, np.nextafter(p, 0), np.nextafter(p, np.inf), -p, [0.0, -0.0, np.inf, -np.inf, np.nan, -np.nan]])
    return np.concatenate([b.view(np.float64), edge])


def test_conversions_bit_for_bit(dev):
    rng = np.random.default_rng(1)
    f = np.concatenate([rng.integers(0, 1 << 32, N, dtype=np.int64), np.arange(0, 1 << 32, 1 << 23, dtype=np.int64),
                        np.arange(0, 1 << 32, 1 << 23, dtype=np.int64) + 1, [0x7fffffff, 0xffffffff, 0x7f800001, 0x00000001]])
    f = f.view(np.float64)
    assert np.array_equal(_bits(dev("f32_to_f64", f)), _bits(dev("cast_up", f)))
    x = _doubles(rng)
    with np.errstate(invalid="ignore"):   # on, beside and between FP32 values
        near = rng.integers(0, 1 << 32, N, dtype=np.int64).astype(np.uint32).view(np.float32).astype(np.float64)
    u = np.abs(np.spacing(near.astype(np.float32)).astype(np.float64)) / 2
    with np.errstate(invalid="ignore", over="ignore"):
        x = np.concatenate([x, near, near + u, near - u, np.nextafter(near + u, np.inf), np.nextafter(near + u, -np.inf)])
    assert np.array_equal(_bits(dev("f64_to_f32", x)), _bits(dev("cast_down", x)))


def test_units_and_counts_exact(dev):
    rng = np.random.default_rng(2)
    a, b = (np.concatenate([rng.integers(0, 1 << 32, N, dtype=np.int64), [0, 0xffffffff, 0x80000000, 0x7fffffff, 64, 63, 0x80000040]]) for _ in range(2))
    n = ((a >> 6) << 26) | (b >> 6)
    assert np.array_equal(_bits(dev("sym_unit", a.view(np.float64), b.view(np.float64))), _bits((2 * n + 1 - (1 << 52)).astype(np.float64) * 2.0 ** -52))
    k = np.arange(1, (1 << 20) + 1, dtype=np.float64)
    assert np.array_equal(dev("count", k), k)


def test_division_by_a_count_rounded_correctly(dev):
    rng = np.random.default_rng(3)
    n = rng.integers(1, 513, N).astype(np.float64)
    x = rng.choice([-1.0, 1.0], N) * rng.uniform(1, 2, N) * 2.0 ** rng.integers(-900, 900, N)
    q = np.rint(rng.uniform(-1e12, 1e12, N))   # and multiples, and their neighbours
    for v in (x, q * n, np.nextafter(q * n, 0), np.nextafter(x, 0), rng.integers(1, 1 << 53, N).astype(np.float64), np.zeros(N)):
        assert np.array_equal(dev("div_count", v, n), v / n)


def test_reciprocals_within_their_roundings(dev):
    rng = np.random.default_rng(4)
    x = _doubles(rng)
    for name, roundings in (("rcp", 1), ("rsqrt", 2)):
        got, plain = dev(name, x), dev("plain_" + name, x)
        hi = (_bits(x) >> 32).astype(np.int32).astype(np.int64)
        short = (hi >= 0x00200000) & (hi < 0x7fc00000)     # the rest takes the plain operation
        assert np.array_equal(_bits(got[~short]), _bits(plain[~short]))
        v, g = x[short], got[short]
        exact = 1 / v.astype(LD) if name == "rcp" else 1 / np.sqrt(v.astype(LD))
        assert np.all(np.abs(g.astype(LD) - exact) <= roundings * np.spacing(g).astype(LD)), name
        v = np.random.default_rng(5).uniform(0.25, 4.0, 4 * N)
        g = dev(name, v)
        exact = 1 / v.astype(LD) if name == "rcp" else 1 / np.sqrt(v.astype(LD))
        assert np.all(np.abs(g.astype(LD) - exact) <= roundings * np.spacing(g).astype(LD)), name


def test_exponential_of_what_is_not_positive(dev):
    """Within one rounding where the result is normal, one subnormal spacing below."""
    rng = np.random.default_rng(6)
    x = -np.concatenate([rng.uniform(0, 745.5, 4 * N), rng.uniform(0, 1, N), rng.uniform(708, 745.5, N), np.exp(rng.uniform(-700, 0, N)),
                         np.arange(0, 746 * 64) * np.log(2) / 64, [0.0, 745.13321910194, 745.14, 745.25, 745.2499999, 1e3, 1e308, np.inf]])
    g = dev("exp", x)
    exact = np.exp(x.astype(LD))
    assert np.all(np.abs(g.astype(LD) - exact) <= np.spacing(np.maximum(g, 5e-324)).astype(LD))
    assert np.array_equal(dev("exp", np.array([0.0, -0.0, -np.inf, -746.0])), [1.0, 1.0, 0.0, 0.0]) and np.isnan(dev("exp", np.array([np.nan])))[0]


@pytest.mark.parametrize("L", [8.0, 20.0, 30.0, 40.0, 13.7, 1e-3, 1e9, struct.unpack("<d", struct.pack("<Q", 0x4034000affffffff))[0],
                               struct.unpack("<d", struct.pack("<Q", 0x4034000affffffff - (1 << 52)))[0]])
def test_minimum_images_bit_for_bit(dev, L):
    """All displacements, and those about an image's edges; sides whose half ends in zeros or in ones among them."""
    hi = lambda v: int(struct.unpack("<q", struct.pack("<d", v))[0] >> 32)
    rng = np.random.default_rng(7)
    steps = np.array([struct.unpack("<q", struct.pack("<d", m * L))[0] for m in (0.5, 1.0, 1.5, 2.0, 2.5)])
    near = (steps[:, None] + np.concatenate([np.arange(-40, 41), rng.integers(-(1 << 34), 1 << 34, 4000)])[None]).reshape(-1).view(np.float64)
    x = np.concatenate([near, -near, rng.uniform(-3, 3, N) * L, rng.normal(size=N) * L * 1e6, [0.0, -0.0, np.inf, -np.inf, np.nan]])
    lo, up = hi(0.5 * L), hi(1.5 * L) - 1
    a, b = dev("image_short", x, L=L, lo=lo, hi=up), dev("image", x, L=L, lo=lo, hi=up)
    differ = ~((a == b) | (np.isnan(a) & np.isnan(b)))
    assert not differ.any(), (x[differ][:5], a[differ][:5], b[differ][:5])
    open_x = _doubles(rng)
    a = dev("image_short", open_x, lo=0x7fffffff, hi=0x7fffffff)
    assert np.all((a == open_x) | np.isnan(open_x))


def test_keys_order_as_their_values(dev):
    rng = np.random.default_rng(8)
    x, y = (v[~np.isnan(v)][:N] for v in (_doubles(rng), _doubles(rng)))
    n = min(x.size, y.size)
    assert np.array_equal(_bits(dev("key", x[:n], y[:n])), _bits(x[:n]))


@pytest.mark.parametrize("n", [1, 2, 3, 6, 18])
def test_warp_sums_of_several_values(dev, n):
    x = np.random.default_rng(n).integers(-1000, 1000, (32, n)).astype(np.float64)
    out = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
    xt = torch.from_numpy(x).cuda()
    assert dev.lib.run_sums(n, xt.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    assert np.array_equal(out.cpu().numpy(), x.sum(0))
