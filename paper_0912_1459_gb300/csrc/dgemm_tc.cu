// Exact-slice FP64 GEMM on the tensor cores (dgemm_tc.cuh).
//
// Tile 128 x 64, eight FP32 accumulators of 64 columns, one per weight
// u = s + t (all 512 TMEM columns).  B's digit tiles lie one after another in
// shared memory, so one MMA of N = 64 j multiplies digit s of A with digits
// t .. t + j - 1 of B into the accumulators s + t .. s + t + j - 1: the 36
// digit products of a k-step are 12 MMAs (N up to 256), and A's digits are
// read from shared memory 12 times instead of 36.
// Exact sums: a chunk of 256 columns adds at most 256 (u + 1) products into
// weight u; with |d_0| <= 64 and |d| <= 128 elsewhere that is at most 2^24 for
// u <= 4, so those sums are exact in FP32; for u >= 5 a sum can only pass
// 2^24 when the low digits of 200 columns all agree, and then loses units of
// 2^-52 of the scales.  After each chunk the epilogue adds the sums as
// integers, weights 0..3 and 4..7 in one int64 each, and rounds once per
// result, to nearest, when it forms the FP64 value with integer operations:
// the FP64 pipe (2 lanes a clock and SM) is not used at all.
#include "dgemm_tc.cuh"
#include "tcgen05.cuh"

namespace cds {
namespace dx {

using namespace tc;

constexpr int NSTAGE = 4;
constexpr int A_DIGIT = kRowsA * 32;               // 4 KB
constexpr int B_DIGIT = kRowsB * 32;               // 2 KB
constexpr int A_STEP = kDigits * A_DIGIT;          // 32 KB
constexpr int B_STEP = kDigits * B_DIGIT;          // 16 KB
constexpr int STAGE = A_STEP + B_STEP;
constexpr int CHUNK = 16;                          // k-steps per exact chunk (256 columns)
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 64 + 32 * EPI_WARPS;
constexpr size_t SMEM = 1024 + NSTAGE * STAGE + 128;
constexpr int kMagicI = 0x4B400000;                // bits of 1.5 * 2^23
constexpr float kMagicF = 12582912.f;
constexpr int kMaxExp = 400;

struct Args {
    const uint8_t *a, *b;
    const int32_t *exa, *exb;
    int64_t m, per, per_pad;     // rows of A, rows per group of B
    int32_t ksteps, mtiles, tpg; // tpg: tiles per group of B
    int32_t g0, ng;
    Out out;
};

// K-major, 32-byte swizzle, 8-row groups 256 bytes apart.
__device__ __forceinline__ uint64_t desc32(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) |
           ((uint64_t)(256 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
}
__device__ __forceinline__ constexpr uint32_t idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(kRowsA >> 4) << 24);
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4]) {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ bool epi_any(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 1, 256, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v)
        : "memory");
    return r != 0;
}

// (hi 2^32 + lo) 2^e as a double, rounded to nearest (ties to even).
__device__ __forceinline__ double to_double(long long hi, long long lo, int e) {
    unsigned long long l = (unsigned long long)lo + ((unsigned long long)hi << 32);
    long long h = (hi >> 32) + (lo >> 63) + (l < (unsigned long long)lo ? 1 : 0);
    const bool neg = h < 0;
    if (neg) {
        l = ~l + 1ull;
        h = ~h + (l == 0 ? 1 : 0);
    }
    unsigned long long top = (unsigned long long)h, rest = l;
    if (top == 0) { top = rest; rest = 0; e -= 64; }
    if (top == 0) return 0.0;
    const int lz = __clzll((long long)top);
    if (lz) {
        top = (top << lz) | (rest >> (64 - lz));
        rest <<= lz;
    }
    // value = (top + rest 2^-64) 2^(64 - lz + e), top's leading bit set
    unsigned long long mant = top >> 11;
    const unsigned long long low = top & 0x7ffull;
    const bool up = low > 0x400ull || (low == 0x400ull && (rest != 0 || (mant & 1ull)));
    // exponent of the leading bit: 127 - lz + e; the mantissa's leading bit adds 1
    const unsigned long long bexp = (unsigned long long)(127 - lz + e + 1023 - 1);
    unsigned long long bits = (bexp << 52) + mant + (up ? 1ull : 0ull);
    if (neg) bits |= 0x8000000000000000ull;
    return __longlong_as_double((long long)bits);
}

__global__ void __launch_bounds__(THREADS, 1)
k_dx_gemm(const Args g, const int32_t* __restrict__ active, const int32_t* __restrict__ flag,
          int32_t* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    if (*flag) return;   // the plain FP64 kernel takes the call
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + NSTAGE * STAGE);
    uint64_t* empty = full + NSTAGE;
    uint64_t* tfull = empty + NSTAGE;
    uint64_t* tempty = tfull + 1;
    uint32_t* tmem_slot = (uint32_t*)(tempty + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t ntiles_n = g.ng * g.tpg;
    const int64_t ntiles = (int64_t)g.mtiles * ntiles_n;
    volatile int32_t* verr = err;

    if (threadIdx.x == 0) {
        for (int i = 0; i < NSTAGE; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        mbar_init(tfull, 1);
        mbar_init(tempty, EPI_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- producer: two contiguous copies per k-step ----------------
            int stage = 0;
            uint32_t phase = 0;
            int32_t last_parity[NSTAGE];
            for (int i = 0; i < NSTAGE; ++i) last_parity[i] = -1;
            bool ok = true;
            for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
                const int32_t nt = (int32_t)(tile % ntiles_n), mt = (int32_t)(tile / ntiles_n);
                const int32_t grp = g.g0 + nt / g.tpg;
                if (active && !active[grp]) continue;
                const uint8_t* pa = g.a + (int64_t)mt * g.ksteps * A_STEP;
                const uint8_t* pb = g.b + ((int64_t)grp * g.tpg + nt % g.tpg) * g.ksteps * B_STEP;
                for (int ks = 0; ks < g.ksteps; ++ks) {
                    if (!mbar_wait(&empty[stage], phase ^ 1u, verr)) { ok = false; break; }
                    mbar_arrive_expect_tx(&full[stage], (uint32_t)STAGE);
                    last_parity[stage] = (int32_t)phase;
                    const uint32_t st = smem_u32(smem + stage * STAGE);
                    bulk_load(st, pa + (int64_t)ks * A_STEP, A_STEP, &full[stage]);
                    bulk_load(st + A_STEP, pb + (int64_t)ks * B_STEP, B_STEP, &full[stage]);
                    if (++stage == NSTAGE) { stage = 0; phase ^= 1u; }
                }
            }
            for (int i = 0; i < NSTAGE; ++i)
                if (last_parity[i] >= 0) mbar_wait(&full[i], (uint32_t)last_parity[i], verr, false);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---------------- MMA issuer ----------------
            int stage = 0;
            uint32_t phase = 0, aphase = 0;
            bool ok = true;
            for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
                const int32_t nt = (int32_t)(tile % ntiles_n);
                if (active && !active[g.g0 + nt / g.tpg]) continue;
                for (int ks = 0; ks < g.ksteps; ++ks) {
                    const bool first = ks % CHUNK == 0;
                    if (first) {
                        if (!mbar_wait(tempty, aphase ^ 1u, verr)) { ok = false; break; }
                        fence_after();
                    }
                    if (!mbar_wait(&full[stage], phase, verr)) { ok = false; break; }
                    fence_after();
                    const uint32_t sa = smem_u32(smem + stage * STAGE), sb = sa + A_STEP;
#pragma unroll
                    for (int s = 0; s < kDigits; ++s) {
                        const uint32_t en = (s == 0 && first) ? 0u : 1u;
                        const int n1 = s <= 4 ? 4 : kDigits - s;
                        mma_f16(tmem + s * kRowsB, desc32(sa + s * A_DIGIT), desc32(sb),
                                idesc(n1 * kRowsB), en);
                        if (s < 4)
                            mma_f16(tmem + (s + 4) * kRowsB, desc32(sa + s * A_DIGIT),
                                    desc32(sb + 4 * B_DIGIT), idesc((4 - s) * kRowsB), en);
                    }
                    mma_commit(&empty[stage]);
                    if (++stage == NSTAGE) { stage = 0; phase ^= 1u; }
                    if (ks % CHUNK == CHUNK - 1 || ks == g.ksteps - 1) {
                        mma_commit(tfull);
                        aphase ^= 1u;
                    }
                }
            }
        }
    } else {
        // ---------------- epilogue: 8 warps, (row, 32 columns) per thread ----------------
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const int row = quad * 32 + lane;
        const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)half * 32u;
        const int nch = (g.ksteps + CHUNK - 1) / CHUNK;
        // every converted sum carries the magic constant's bits
        const long long bias =
            (long long)nch * (long long)kMagicI * ((1LL << 24) + (1LL << 16) + (1LL << 8) + 1LL);
        uint32_t aphase = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
            const int32_t nt = (int32_t)(tile % ntiles_n), mt = (int32_t)(tile / ntiles_n);
            const int32_t gl = nt / g.tpg, grp = g.g0 + gl;
            if (active && !active[grp]) continue;
            long long H[32], L[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) { H[j] = -bias; L[j] = -bias; }
            for (int ch = 0; ch < nch; ++ch) {
                const bool bad = !mbar_wait(tfull, aphase, verr) || *verr;
                if (epi_any(bad)) { ok = false; break; }
                aphase ^= 1u;
                fence_after();
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    float v[kDigits][4];
#pragma unroll
                    for (int u = 0; u < kDigits; ++u) tmem_ld4(ta + u * kRowsB + c * 4, v[u]);
                    tmem_wait_ld();
                    float mx = 0.f;
#pragma unroll
                    for (int u = 0; u < kDigits; ++u)
#pragma unroll
                        for (int j = 0; j < 4; ++j) mx = fmaxf(mx, fabsf(v[u][j]));
                    int iv[kDigits][4];
                    if (__any_sync(0xffffffffu, mx >= 4194304.f)) {
#pragma unroll
                        for (int u = 0; u < kDigits; ++u)
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                iv[u][j] = __float2int_rn(v[u][j]) + kMagicI;
                    } else {   // |v| < 2^22: the integer is in the low bits of v + 1.5 2^23
#pragma unroll
                        for (int u = 0; u < kDigits; ++u)
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                iv[u][j] = __float_as_int(v[u][j] + kMagicF);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int o = c * 4 + j;
                        H[o] += ((long long)iv[0][j] << 24) + ((long long)iv[1][j] << 16) +
                                ((long long)iv[2][j] << 8) + iv[3][j];
                        L[o] += ((long long)iv[4][j] << 24) + ((long long)iv[5][j] << 16) +
                                ((long long)iv[6][j] << 8) + iv[7][j];
                    }
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty);
            }
            if (!ok) break;
            // the next tile's MMAs run while the results are formed and stored
            const int64_t m = (int64_t)mt * kRowsA + row;
            const int32_t c0 = (nt % g.tpg) * kRowsB + half * 32;
            const int ncols = (int)min((int64_t)32, g.per - c0);
            if (m < g.m && ncols > 0) {
                const int ea = g.exa[m] - 68;
                const int32_t* eb = g.exb + (int64_t)grp * g.per_pad + c0;
                double* dst = g.out.p + (m / g.out.kdiv) * g.out.m_hi + (m % g.out.kdiv) * g.out.m_lo +
                              (int64_t)gl * g.out.g_s + (int64_t)c0 * g.out.n_s;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (j < ncols) dst[j * g.out.n_s] = to_double(H[j], L[j], ea + eb[j]);
            }
        }
    }

    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(512u));
    }
}

// ---------------------------------------------------------------------------
// slicing: one warp per row, a lane takes 8 consecutive columns (a 16-byte
// piece of each digit's row), two passes over the row (largest entry, digits)
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long fixed62(double x, int ex) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    int e = (int)((b >> 52) & 0x7ffull);
    unsigned long long m = b & 0xfffffffffffffull;
    if (e) m |= 1ull << 52;
    else e = 1;
    const int sh = e - 1013 - ex;   // q = m 2^sh, sh <= 9
    if (sh >= 0) m <<= sh;
    else if (sh > -54) m = (m + (1ull << (-sh - 1))) >> -sh;
    else m = 0;
    return (b >> 63) ? -(long long)m : (long long)m;
}

template <int R, typename Src>
__global__ void __launch_bounds__(256)
k_dx_slice(const Src src, int64_t groups, int64_t per, int64_t per_pad, int32_t kdim,
           int32_t ksteps, uint8_t* __restrict__ img, int32_t* __restrict__ exps,
           int32_t* __restrict__ flag) {
    const int64_t idx = blockIdx.x * 8LL + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (idx >= groups * per) return;
    const int64_t g = idx / per, r = idx - g * per;
    unsigned long long mx = 0;
    for (int k = lane; k < kdim; k += 32) {
        const unsigned long long a =
            (unsigned long long)__double_as_longlong(src.get(g, r, k)) & 0x7fffffffffffffffull;
        mx = a > mx ? a : mx;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = w > mx ? w : mx;
    }
    int ex = mx ? (int)(mx >> 52) - 1022 : 0;   // every |x| < 2^ex
    const int64_t ir = g * per_pad + r;
    if (lane == 0) {
        exps[ir] = ex;
        if (ex > kMaxExp || ex < -kMaxExp) *flag = 1;
    }
    if (ex > kMaxExp) return;
    const int64_t tile = ir / R;
    const int rr = (int)(ir % R);
    const int off = (rr >> 3) * 256 + (rr & 7) * 32, swz = (rr >> 2) & 1;
    for (int c = lane; c < 2 * ksteps; c += 32) {
        uint32_t w[kDigits][4];
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
#pragma unroll
            for (int j = 0; j < 4; ++j) w[s][j] = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = c * 8 + j;
            long long q = k < kdim ? fixed62(src.get(g, r, k), ex) : 0;
#pragma unroll
            for (int s = kDigits - 1; s >= 0; --s) {
                const int d = s ? (int)(signed char)(q & 0xff) : (int)q;
                q = (q - d) >> 8;
                // float(d) through the low bits of 1.5 2^23 + d; its upper half is the BF16
                const float f = __int_as_float(kMagicI + d) - kMagicF;
                w[s][j >> 1] |= (__float_as_uint(f) >> 16) << (16 * (j & 1));
            }
        }
        uint8_t* dst = img + ((tile * ksteps + (c >> 1)) * kDigits) * (int64_t)(R * 32) + off +
                       (((c & 1) ^ swz) << 4);
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
            *reinterpret_cast<uint4*>(dst + (int64_t)s * (R * 32)) =
                make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
}

template <typename Src>
static int slice_any(const Src& src, const Operand& o, int R, int32_t kdim, int32_t* flag,
                     cudaStream_t stream) {
    const int64_t rows = o.groups * o.per;
    if (rows <= 0 || kdim <= 0) return CDS_OK;
    const unsigned grid = (unsigned)((rows + 7) / 8);
    if (R == kRowsA)
        k_dx_slice<kRowsA, Src><<<grid, 256, 0, stream>>>(src, o.groups, o.per, o.per_pad, kdim,
                                                          o.ksteps, o.img, o.ex, flag);
    else
        k_dx_slice<kRowsB, Src><<<grid, 256, 0, stream>>>(src, o.groups, o.per, o.per_pad, kdim,
                                                          o.ksteps, o.img, o.ex, flag);
    CDS_LAUNCH_CHECK();
    return CDS_OK;
}

int slice_rows(const RowMajor& src, const Operand& o, int R, int32_t kdim, int32_t* flag,
               cudaStream_t stream) {
    return slice_any(src, o, R, kdim, flag, stream);
}
int slice_packed(const PackedRows& src, const Operand& o, int R, int32_t kdim, int32_t* flag,
                 cudaStream_t stream) {
    return slice_any(src, o, R, kdim, flag, stream);
}
int slice_columns(const Columns& src, const Operand& o, int R, int32_t kdim, int32_t* flag,
                  cudaStream_t stream) {
    return slice_any(src, o, R, kdim, flag, stream);
}

__global__ void k_nan_on_error(const int32_t* __restrict__ err, double* __restrict__ p, int64_t n) {
    if (*err == 0) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = __longlong_as_double(0x7ff8000000000000LL);
}

int nan_on_error(const int32_t* err, double* p, int64_t n, cudaStream_t stream) {
    if (n <= 0) return CDS_OK;
    k_nan_on_error<<<(unsigned)std::min<int64_t>((n + 255) / 256, 2 * device_sms()), 256, 0, stream>>>(
        err, p, n);
    CDS_LAUNCH_CHECK();
    return CDS_OK;
}

int gemm(const Operand& A, const Operand& B, int64_t g0, int64_t g1, const Out& out,
         const int32_t* active, const int32_t* flag, int32_t* err, cudaStream_t stream) {
    if (A.groups != 1 || A.ksteps != B.ksteps) return CDS_ERR_ARG;
    if (A.per <= 0 || B.per <= 0 || g1 <= g0 || A.ksteps <= 0) return CDS_OK;
    Args a;
    a.a = A.img;
    a.b = B.img;
    a.exa = A.ex;
    a.exb = B.ex;
    a.m = A.per;
    a.per = B.per;
    a.per_pad = B.per_pad;
    a.ksteps = A.ksteps;
    const int64_t mtiles = A.per_pad / kRowsA, tpg = B.per_pad / kRowsB, ng = g1 - g0;
    if (mtiles > INT32_MAX || tpg * ng > INT32_MAX || tpg * g1 > INT32_MAX) return CDS_ERR_UNSUPPORTED;
    a.mtiles = (int32_t)mtiles;
    a.tpg = (int32_t)tpg;
    a.g0 = (int32_t)g0;
    a.ng = (int32_t)ng;
    a.out = out;
    CDS_CUDA_TRY(cudaFuncSetAttribute(k_dx_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)SMEM));
    const int grid = (int)std::min<int64_t>(mtiles * tpg * ng, device_sms());
    k_dx_gemm<<<grid, THREADS, SMEM, stream>>>(a, active, flag, err);
    CDS_LAUNCH_CHECK();
    return CDS_OK;
}

}  // namespace dx
}  // namespace cds
