// Exact-slice FP64 GEMM on the tensor cores (dgemm_tc.cuh).
//
// Tile 128 x 64, eight FP32 accumulators of 64 columns, one per weight
// u = s + t (all 512 TMEM columns).  B's digit tiles lie one after another in
// shared memory, so one MMA of N = 64 j multiplies digit s of A with digits
// t .. t + j - 1 of B into the accumulators s + t .. s + t + j - 1: the 36
// digit products of a k-step are 12 MMAs (N up to 256), and A's digits are
// read from shared memory 12 times instead of 36.
// Exact sums: a chunk of 240 columns adds at most 240 (u + 1) products into
// weight u; with |d_0| <= 64 and |d| <= 128 elsewhere that is below 2^24 for
// u <= 4, so those sums are exact in FP32.  Weight 5 passes 2^24 only where the
// digits d_1 .. d_4 of the whole chunk are near 128 and agree, and S is then above
// 2^-1; its units (2^-52 of the scales) are then below the bound above.  After each
// chunk the epilogue adds the sums as
// integers, weights 0..3 and 4..7 in one int64 each, and rounds once per
// result, to nearest, when it forms the FP64 value with integer operations:
// the FP64 pipe (2 lanes a clock and SM) is not used at all.
//
// k_dx_guard, the second pass, is one MMA per k-step and tile beside the 12 above and
// reads an eighth of their bytes: 50 us beside 700 for the integrals of 10 orbitals of
// 240 functions, 720 vectors.  Results that it takes again cost K FMAs on the FP64 units
// each, as every result did before the slices; with factors graded in opposite senses, all
// of them: one energy of an orbital of 840 functions 6.8 ms, then 173 (165 with the fused
// FP64 kernel).
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
constexpr int CHUNK = 15;                          // k-steps per exact chunk (240 columns)
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

__global__ void __launch_bounds__(THREADS, 1)
k_dx_gemm(const Args g, const int32_t* __restrict__ active, int32_t* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
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
template <int R, typename Src>
__global__ void __launch_bounds__(256)
k_dx_slice(const Src src, int64_t groups, int64_t per, int64_t per_pad, int32_t kdim,
           int32_t ksteps, uint8_t* __restrict__ img, uint8_t* __restrict__ mag,
           int32_t* __restrict__ exps) {
    const int64_t idx = blockIdx.x * 8LL + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (idx >= groups * per) return;
    const int64_t g = idx / per, r = idx - g * per;
    const auto x_of = src.row(g, r);
    unsigned long long mx = 0;
    for (int k = lane; k < kdim; k += 32) {
        const unsigned long long a =
            (unsigned long long)__double_as_longlong(x_of[k]) & 0x7fffffffffffffffull;
        mx = a > mx ? a : mx;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = w > mx ? w : mx;
    }
    int ex = mx ? (int)(mx >> 52) - 1022 : 0;   // every |x| < 2^ex
    const bool plain = ex > kMaxExp || ex < -kMaxExp;   // left to the second pass: digits, magnitudes 0
    if (plain) ex = 0;
    const int64_t ir = g * per_pad + r;
    if (lane == 0) exps[ir] = ex;
    const int64_t tile = ir / R;
    const int rr = (int)(ir % R);
    const int off = (rr >> 3) * 256 + (rr & 7) * 32, swz = (rr >> 2) & 1;
    for (int c = lane; c < 2 * ksteps; c += 32) {
        uint32_t w[kDigits][4], wm[4] = {0, 0, 0, 0};
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
#pragma unroll
            for (int j = 0; j < 4; ++j) w[s][j] = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = c * 8 + j;
            const double x = k < kdim && !plain ? x_of[k] : 0.0;
            long long q = fixed62(x, ex);
            // a row of zeros counts as one of ones: its results are exact
            const uint32_t m = mx == 0 ? (k < kdim ? 0x3f80u : 0u) : magnitude(x, ex);
            wm[j >> 1] |= m << (16 * (j & 1));
#pragma unroll
            for (int s = kDigits - 1; s >= 0; --s) {
                const int d = s ? (int)(signed char)(q & 0xff) : (int)q;
                q = (q - d) >> 8;
                // float(d) through the low bits of 1.5 2^23 + d; its upper half is the BF16
                const float f = __int_as_float(kMagicI + d) - kMagicF;
                w[s][j >> 1] |= (__float_as_uint(f) >> 16) << (16 * (j & 1));
            }
        }
        const int piece = off + (((c & 1) ^ swz) << 4);
        const int64_t step = tile * ksteps + (c >> 1);
        *reinterpret_cast<uint4*>(mag + step * (int64_t)(R * 32) + piece) = make_uint4(wm[0], wm[1], wm[2], wm[3]);
        uint8_t* dst = img + step * kDigits * (int64_t)(R * 32) + piece;
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
            *reinterpret_cast<uint4*>(dst + (int64_t)s * (R * 32)) =
                make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
}

template <typename Src>
static int slice_any(const Src& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream) {
    const int64_t rows = o.groups * o.per;
    if (rows <= 0 || kdim <= 0) return CDS_OK;
    const unsigned grid = (unsigned)((rows + 7) / 8);
    auto kern = R == kRowsA ? k_dx_slice<kRowsA, Src> : k_dx_slice<kRowsB, Src>;
    kern<<<grid, 256, 0, stream>>>(src, o.groups, o.per, o.per_pad, kdim, o.ksteps, o.img, o.mag, o.ex);
    CDS_LAUNCH_CHECK();
    return CDS_OK;
}

int slice(const RowMajor& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream) {
    return slice_any(src, o, R, kdim, stream);
}
int slice(const PanelRows& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream) {
    return slice_any(src, o, R, kdim, stream);
}
int slice(const PackedRows& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream) {
    return slice_any(src, o, R, kdim, stream);
}
int slice(const Columns& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream) {
    return slice_any(src, o, R, kdim, stream);
}

// ---------------------------------------------------------------------------
// second pass: S = sum |a||b| of every result, and the FP64 sum where it is small
// ---------------------------------------------------------------------------
constexpr int G_STAGES = 4;
constexpr int G_STEPS = 4;                         // k-steps per stage
constexpr int G_STAGE = G_STEPS * (A_DIGIT + B_DIGIT);   // 24 KB
constexpr size_t G_SMEM = 1024 + G_STAGES * G_STAGE + 128;
constexpr uint32_t G_COLS = 2 * kRowsB;            // two accumulators
constexpr float kLeastS = 1.f / 32.f;              // K 2^-58.9 <= K 2^-53 S with room to spare

struct GuardArgs {
    const uint8_t *a, *b;
    int64_t m, per;
    int32_t ksteps, mtiles, tpg, g0, ng, kdim;
    Out out;
};

// Sums of eight values over the warp (9 adds): lanes 4 i .. 4 i + 3 return value i.
__device__ __forceinline__ double warp_sums8(double (&v)[8]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = 4; n >= 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const double send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    double s = v[0];
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    return s + __shfl_xor_sync(0xffffffffu, s, 1);
}

template <typename SrcA, typename SrcB>
__global__ void __launch_bounds__(THREADS, 2)
k_dx_guard(const GuardArgs g, const SrcA srca, const SrcB srcb, const int32_t* __restrict__ active,
           int32_t* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + G_STAGES * G_STAGE);
    uint64_t* empty = full + G_STAGES;
    uint64_t* tfull = empty + G_STAGES;
    uint64_t* tempty = tfull + 2;
    uint32_t* tmem_slot = (uint32_t*)(tempty + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t ntiles_n = g.ng * g.tpg;
    const int64_t ntiles = (int64_t)g.mtiles * ntiles_n;
    volatile int32_t* verr = err;

    if (threadIdx.x == 0) {
        for (int i = 0; i < G_STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], EPI_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(G_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- producer: two contiguous copies per stage ----------------
            int stage = 0;
            uint32_t phase = 0;
            int32_t last_parity[G_STAGES];
            for (int i = 0; i < G_STAGES; ++i) last_parity[i] = -1;
            bool ok = true;
            for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
                const int32_t nt = (int32_t)(tile % ntiles_n), mt = (int32_t)(tile / ntiles_n);
                const int32_t grp = g.g0 + nt / g.tpg;
                if (active && !active[grp]) continue;
                const uint8_t* pa = g.a + (int64_t)mt * g.ksteps * A_DIGIT;
                const uint8_t* pb = g.b + ((int64_t)grp * g.tpg + nt % g.tpg) * g.ksteps * B_DIGIT;
                for (int ks = 0; ks < g.ksteps; ks += G_STEPS) {
                    if (!mbar_wait(&empty[stage], phase ^ 1u, verr)) { ok = false; break; }
                    const uint32_t n = (uint32_t)min(G_STEPS, g.ksteps - ks);
                    mbar_arrive_expect_tx(&full[stage], n * (A_DIGIT + B_DIGIT));
                    last_parity[stage] = (int32_t)phase;
                    const uint32_t st = smem_u32(smem + stage * G_STAGE);
                    bulk_load(st, pa + (int64_t)ks * A_DIGIT, n * A_DIGIT, &full[stage]);
                    bulk_load(st + G_STEPS * A_DIGIT, pb + (int64_t)ks * B_DIGIT, n * B_DIGIT, &full[stage]);
                    if (++stage == G_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            for (int i = 0; i < G_STAGES; ++i)
                if (last_parity[i] >= 0) mbar_wait(&full[i], (uint32_t)last_parity[i], verr, false);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---------------- MMA issuer ----------------
            int stage = 0, buf = 0;
            uint32_t phase = 0, aphase = 0;
            bool ok = true;
            for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
                const int32_t nt = (int32_t)(tile % ntiles_n);
                if (active && !active[g.g0 + nt / g.tpg]) continue;
                if (!mbar_wait(&tempty[buf], aphase ^ 1u, verr)) break;
                fence_after();
                for (int ks = 0; ks < g.ksteps; ks += G_STEPS) {
                    if (!mbar_wait(&full[stage], phase, verr)) { ok = false; break; }
                    fence_after();
                    const uint32_t sa = smem_u32(smem + stage * G_STAGE), sb = sa + G_STEPS * A_DIGIT;
                    const int n = min(G_STEPS, g.ksteps - ks);
                    for (int i = 0; i < n; ++i)
                        mma_f16(tmem + (uint32_t)buf * kRowsB, desc32(sa + i * A_DIGIT),
                                desc32(sb + i * B_DIGIT), idesc(kRowsB), (ks | i) ? 1u : 0u);
                    mma_commit(&empty[stage]);
                    if (++stage == G_STAGES) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                mma_commit(&tfull[buf]);
                if (++buf == 2) { buf = 0; aphase ^= 1u; }
            }
        }
    } else {
        // ---------------- epilogue: 8 warps, (row, 32 columns) per thread ----------------
        const int quad = warp & 3, half = (warp - 2) >> 2;
        int buf = 0;
        uint32_t aphase = 0;
        for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const int32_t nt = (int32_t)(tile % ntiles_n), mt = (int32_t)(tile / ntiles_n);
            const int32_t gl = nt / g.tpg, grp = g.g0 + gl;
            if (active && !active[grp]) continue;
            const bool bad = !mbar_wait(&tfull[buf], aphase, verr) || *verr;
            if (epi_any(bad)) break;
            fence_after();
            const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * kRowsB + half * 32);
            const int64_t m0 = (int64_t)mt * kRowsA + quad * 32;
            const int32_t c0 = (nt % g.tpg) * kRowsB + half * 32;
            const int ncols = (int)min((int64_t)32, g.per - c0);
            const bool mok = m0 + lane < g.m;
            uint32_t again = 0;                      // columns of this thread's row
#pragma unroll
            for (int c = 0; c < 32; c += 16) {
                float s[16];
                tmem_ld16(ta + c, s);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (mok && c + j < ncols && !(s[j] >= kLeastS)) again |= 1u << (c + j);
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
            if (++buf == 2) { buf = 0; aphase ^= 1u; }
            // The results with a small S again.  Rows with many of them, where B's rows lie
            // across: a lane per column, four rows at a time, one FMA chain per result (320
            // functions, localised orbitals, 80 % of the results: whole transform 45 -> 20 ms, 36 with
            // every product on the FP64 units).
            if constexpr (SrcB::kAcross) {
                uint32_t many = __ballot_sync(0xffffffffu, __popc(again) >= 8);
                while (many) {
                    constexpr int NR = 4;
                    const int n = min(NR, __popc(many));
                    const int first = __ffs((int)many) - 1;
                    decltype(srca.row(0, 0)) xa[NR];
                    double* dst[NR];
                    uint32_t cols[NR];
#pragma unroll
                    for (int j = 0; j < NR; ++j) {
                        const int rl = many ? __ffs((int)many) - 1 : first;
                        many &= many - 1u;
                        const int64_t m = m0 + rl;
                        xa[j] = srca.row(0, m);
                        dst[j] = g.out.p + (m / g.out.kdiv) * g.out.m_hi + (m % g.out.kdiv) * g.out.m_lo +
                                 (int64_t)gl * g.out.g_s;
                        cols[j] = __shfl_sync(0xffffffffu, again, rl);
                        if (lane == rl) again = 0;
                    }
                    const int col = c0 + min(lane, ncols - 1);
                    const auto xb = srcb.row(grp, col);
                    double v[NR] = {};
#pragma unroll 4
                    for (int k = 0; k < g.kdim; ++k) {
                        const double y = xb[k];
#pragma unroll
                        for (int j = 0; j < NR; ++j) v[j] = fma(xa[j][k], y, v[j]);
                    }
#pragma unroll
                    for (int j = 0; j < NR; ++j)
                        if (j < n && (cols[j] >> lane & 1u)) dst[j][(int64_t)col * g.out.n_s] = v[j];
                }
            }
            // else the whole warp at up to eight of one row
            for (uint32_t rows = __ballot_sync(0xffffffffu, again != 0); rows; rows &= rows - 1) {
                const int rl = __ffs((int)rows) - 1;
                const int64_t m = m0 + rl;
                double* dst = g.out.p + (m / g.out.kdiv) * g.out.m_hi + (m % g.out.kdiv) * g.out.m_lo +
                              (int64_t)gl * g.out.g_s;
                const auto xa = srca.row(0, m);
                uint32_t cols = __shfl_sync(0xffffffffu, again, rl);
                while (cols) {
                    constexpr int NC = 8;
                    const int n = min(NC, __popc(cols));
                    const uint32_t first = (uint32_t)__ffs((int)cols) - 1u;
                    decltype(srcb.row(0, 0)) xb[NC];
                    int mine = 0;                    // the column whose sum this lane ends up with
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        const uint32_t c = cols ? (uint32_t)__ffs((int)cols) - 1u : first;
                        cols &= cols - 1u;
                        xb[j] = srcb.row(grp, c0 + (int)c);
                        if (j == (lane >> 2)) mine = (int)c;
                    }
                    double v[NC] = {};
                    for (int k = lane; k < g.kdim; k += 32) {
                        const double x = xa[k];
#pragma unroll
                        for (int j = 0; j < NC; ++j) v[j] = fma(x, xb[j][k], v[j]);
                    }
                    const double sum = warp_sums8(v);
                    if ((lane & 3) == 0 && (lane >> 2) < n) dst[(int64_t)(c0 + mine) * g.out.n_s] = sum;
                }
            }
        }
    }

    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G_COLS));
    }
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

template <typename SrcA, typename SrcB>
static int gemm_any(const Operand& A, const SrcA& srca, const Operand& B, const SrcB& srcb, int32_t kdim,
                    int64_t g0, int64_t g1, const Out& out, const int32_t* active, int32_t* err,
                    cudaStream_t stream) {
    if (A.groups != 1 || A.ksteps != B.ksteps || A.ksteps != ksteps_of(kdim)) return CDS_ERR_ARG;
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
    const int64_t tiles = mtiles * tpg * ng;
    k_dx_gemm<<<(int)std::min<int64_t>(tiles, device_sms()), THREADS, SMEM, stream>>>(a, active, err);
    CDS_LAUNCH_CHECK();
    const GuardArgs ga{A.mag, B.mag, a.m, a.per, a.ksteps, a.mtiles, a.tpg, a.g0, a.ng, kdim, out};
    auto guard = k_dx_guard<SrcA, SrcB>;
    CDS_CUDA_TRY(cudaFuncSetAttribute(guard, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G_SMEM));
    guard<<<(int)std::min<int64_t>(tiles, 2 * device_sms()), THREADS, G_SMEM, stream>>>(ga, srca, srcb, active,
                                                                                       err);
    CDS_LAUNCH_CHECK();
    return CDS_OK;
}

int gemm(const Operand& A, const RowMajor& a, const Operand& B, const RowMajor& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream) {
    return gemm_any(A, a, B, b, kdim, g0, g1, out, active, err, stream);
}
int gemm(const Operand& A, const PanelRows& a, const Operand& B, const RowMajor& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream) {
    return gemm_any(A, a, B, b, kdim, g0, g1, out, active, err, stream);
}
int gemm(const Operand& A, const PackedRows& a, const Operand& B, const Columns& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream) {
    return gemm_any(A, a, B, b, kdim, g0, g1, out, active, err, stream);
}
int gemm(const Operand& A, const RowMajor& a, const Operand& B, const Columns& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream) {
    return gemm_any(A, a, B, b, kdim, g0, g1, out, active, err, stream);
}

}  // namespace dx
}  // namespace cds
