"""The arithmetic that stands for CUDA's own in the hot kernels, each against CUDA's or
against exact integers: the reciprocal (1 ulp of 1.0 / d, over all exponents and its
cut-offs), the double of a float (the same bits, subnormal numbers, infinities and NaN
among them), the rounding of wide integer sums to a double (nearest, ties to even,
weights that cancel), the 62-bit fixed point of a double and the BF16 magnitude.
A small kernel around the library's own headers is compiled for it."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_0912_1459_gb300 import build

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

DEV = torch.device("cuda:0")
SRC = r"""
#include "dgemm_tc.cuh"
using namespace cds;
__global__ void k_recip(const double* d, int64_t n, double* a, double* b) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) { a[i] = recip(d[i]); b[i] = 1.0 / d[i]; }
}
__global__ void k_double(uint32_t first, int64_t n, unsigned long long* wrong) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float x = __uint_as_float(first + (uint32_t)i);
        const double a = double_of(x), b = (double)x;
        if (x != x ? a == a : __double_as_longlong(a) != __double_as_longlong(b)) atomicAdd(wrong, 1ull);
    }
}
__global__ void k_wide(const long long* hi, const long long* lo, const int32_t* e, int64_t n, double* out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = dx::to_double(hi[i], lo[i], e[i]);
}
__global__ void k_fixed(const double* x, const int32_t* ex, int64_t n, long long* q, int32_t* m) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) { q[i] = dx::fixed62(x[i], ex[i]); m[i] = (int32_t)dx::magnitude(x[i], ex[i]); }
}
static unsigned grid(int64_t n) { return (unsigned)((n + 255) / 256); }
extern "C" void t_recip(const double* d, int64_t n, double* a, double* b) { k_recip<<<grid(n), 256>>>(d, n, a, b); }
extern "C" void t_double(uint32_t f, int64_t n, unsigned long long* w) { k_double<<<4096, 256>>>(f, n, w); }
extern "C" void t_wide(const long long* h, const long long* l, const int32_t* e, int64_t n, double* o) {
    k_wide<<<grid(n), 256>>>(h, l, e, n, o);
}
extern "C" void t_fixed(const double* x, const int32_t* ex, int64_t n, long long* q, int32_t* m) {
    k_fixed<<<grid(n), 256>>>(x, ex, n, q, m);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("conversions")
    (d / "c.cu").write_text(SRC)
    out = str(d / "c.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-cudart", "static", str(d / "c.cu"), "-o",
                    out], check=True, capture_output=True)
    torch.zeros(1, device=DEV)
    return ctypes.CDLL(out)


def p(t):
    return ctypes.c_void_p(t.data_ptr())


def test_recip(lib):
    rng = np.random.default_rng(0)
    mant = np.concatenate([rng.integers(0, 1 << 52, 4000), [0, 1, 2, (1 << 52) - 1, (1 << 52) - 2, 1 << 51],
                           (np.arange(1024) << 42) | rng.integers(0, 2, 1024)]).astype(np.uint64)
    bits = (np.arange(2048, dtype=np.uint64)[:, None] << np.uint64(52)) | mant[None, :]
    d = np.concatenate([bits.ravel().view(np.float64), -bits[::37].ravel().view(np.float64)])
    x = torch.from_numpy(d).to(DEV)
    a, b = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    lib.t_recip(p(x), ctypes.c_int64(x.numel()), p(a), p(b))
    torch.cuda.synchronize()
    nan = torch.isnan(b)
    assert torch.equal(torch.isnan(a), nan)
    ulps = (a.view(torch.int64) - b.view(torch.int64)).abs()[~nan]
    assert ulps.max().item() <= 1
    special = (x.view(torch.int64) >> 52) & 2047
    plain = ((special < 2) | (special >= 2044)) & ~nan
    assert torch.equal(a[plain], b[plain])


def test_double_of_every_float(lib):
    wrong = torch.zeros(1, dtype=torch.int64, device=DEV)
    torch.cuda.synchronize()
    lib.t_double(ctypes.c_uint32(0), ctypes.c_int64(1 << 32), p(wrong))
    torch.cuda.synchronize()
    assert wrong.item() == 0


def nearest(v):
    """The double nearest to an integer times a power of two (Fraction), ties to even."""
    return float(v)                       # Fraction -> float rounds correctly


def test_wide_sums(lib):
    rng = np.random.default_rng(1)
    vals = [(0, 0, 0), (1, 0, -5), (-1, 1 << 32, 3), (0, -1, 0), (1, -(1 << 32), 0), (1 << 40, 1, 7),
            ((1 << 62), (1 << 62), -100), (-(1 << 62), -(1 << 62), 100), (1 << 21, 1 << 21, 0)]
    for k in range(20, 62):               # ties and their neighbours at every width
        for low in (-1, 0, 1):
            vals += [((1 << k) | 1, low, -k), (-(1 << k) - 3, low, k), (0, (1 << k) + low, 2)]
            for half in range(k - 21, k - 20):
                if half >= 0:
                    vals += [((1 << k) + (1 << half), low, 0), ((1 << k) + 3 * (1 << half), low, 0),
                             (-(1 << k) - (1 << half), low, 0)]
    vals += [(int(h) >> int(s), int(lo) >> int(t), int(e)) for h, lo, s, t, e in zip(
        rng.integers(-(1 << 62), 1 << 62, 20000), rng.integers(-(1 << 62), 1 << 62, 20000),
        rng.integers(0, 60, 20000), rng.integers(0, 60, 20000), rng.integers(-800, 700, 20000))]
    h, lo, e = (np.array(c, dtype=t) for c, t in zip(zip(*vals), (np.int64, np.int64, np.int32)))
    th, tl, te = (torch.from_numpy(c).to(DEV) for c in (h, lo, e))
    out = torch.empty(len(vals), dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    lib.t_wide(p(th), p(tl), p(te), ctypes.c_int64(len(vals)), p(out))
    got = out.cpu().numpy()
    for (a, b, c), g in zip(vals, got):
        v = Fraction((a << 32) + b)
        v = v * (1 << c) if c >= 0 else v / (1 << -c)
        assert nearest(v) == g, (a, b, c)


def test_fixed_point_and_magnitude(lib):
    rng = np.random.default_rng(2)
    ex = rng.integers(-400, 401, 30000).astype(np.int32)
    x = np.ldexp(rng.uniform(0.5, 1.0, 30000), ex - rng.integers(0, 80, 30000)) * rng.choice([-1.0, 1.0], 30000)
    edge = [(0.0, 0), (-0.0, 0), (1.0 - 2.0 ** -53, 0), (-(1.0 - 2.0 ** -53), 0), (0.5, 0), (2.0 ** -63, 0),
            (2.0 ** -64, 0), (3 * 2.0 ** -64, 0), (-(2.0 ** -63), 0), (5e-324, 0), (2.0 ** -126, 0), (2.0 ** -127, 0)]
    x = np.concatenate([x, [v for v, _ in edge]])
    ex = np.concatenate([ex, [e for _, e in edge]]).astype(np.int32)
    tx, te = torch.from_numpy(x).to(DEV), torch.from_numpy(ex).to(DEV)
    q = torch.empty(len(x), dtype=torch.int64, device=DEV)
    m = torch.empty(len(x), dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    lib.t_fixed(p(tx), p(te), ctypes.c_int64(len(x)), p(q), p(m))
    q, m = q.cpu().numpy(), m.cpu().numpy()
    mag = (m.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    for v, e, a, b in zip(x, ex, q, mag):
        f = abs(Fraction(float(v))) * Fraction(2) ** (62 - int(e))
        r = int(f + Fraction(1, 2)) if f >= Fraction(1, 2) else 0
        assert abs(int(a)) == r and (a == 0 or (a < 0) == (v < 0)), (v, e)
        t = abs(Fraction(float(v))) / Fraction(2) ** int(e)
        assert Fraction(float(b)) <= t and (t < Fraction(2) ** -126 or Fraction(float(b)) > t * (1 - Fraction(1, 128)))
