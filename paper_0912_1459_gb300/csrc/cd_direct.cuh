// The FP64 Cholesky decomposition as one cooperative launch (included by cd.cu,
// after cd_steps.cuh): every step of it, from the first pivot to the stop test.
//
// Left-looking like the two launches per step it replaces (k_cd_project,
// k_cd_update), whose step took 18 us at 300 pairs, nearly all of it launches and the
// serial end, and 30 us at 28,920 pairs and 377 vectors, where the FP64 units (2
// FMA/clk/SM) bound the projections.  Here
//  - CTA c keeps pairs [c pc, (c + 1) pc): residuals and pair data in registers,
//    the first rows in shared memory;
//  - the integral column, L^k and the residuals are the same FP64 operations;
//  - the projections sum_K L^K_I L^K_P are taken in integers: beside its FP64 row
//    every L^K_I is kept as a 56-bit number below the pair's scale 2^e > sqrt(D0_I)
//    >= |L^K_I|, q = hi 2^26 + lo, and hi hi' and hi lo' + lo hi' are summed exactly
//    in 64 bits (three 32-bit multiply-adds into 64 bits).  In units of the scales'
//    product the sum of K terms is off by at most sqrt(K) 2^-56 (the rounding of q, by
//    Cauchy-Schwarz: sum_K (L^K_I)^2 <= D0_I) + K 2^-62 (lo lo', |lo| <= 2^25): 2^-51 at
//    K = 400, 2^-49 at the largest K; unrelated digits leave about 2^-56 + sqrt(K) 2^-64.
//    The FP64 chain may round its K partial sums to 2^-53 of that product each.  The
//    vectors against extended precision, largest error before -> now: 300 pairs x 104
//    2.8e-14 -> 2.3e-14, 1,176 x 139 9.1e-14 -> 5.5e-14, 1,830 x 117 (a chain of
//    centres) 7.3e-14 -> 5.3e-14, 2,485 x 51 2.2e-13 -> 8.4e-14; rms and relative errors
//    likewise.  No overflow: |sum hi hi'| <= 2^60, |sum hi lo'| <= 2^55 sqrt(K);
//  - while one group of warps forms the integral column on the FP64 units, the
//    others take the projections on the integer units;
//  - the exchange of the residual maxima, the pivot choice and its ties are those
//    of cd_steps.cuh: tagged words, one 128-byte line per CTA, every CTA decides.
// Every wait is bounded and sets the error word instead of hanging.
// Measured, whole decompositions, a launch per step -> this: 300 pairs x 120 vectors 1.98
// -> 0.68 ms, 15,576 x 293 6.5 -> 2.1, 28,920 x 372 11.0 -> 3.8, 56,616 x 456 21.2 -> 11.0,
// 113,526 x 408 28.7 -> 17.2.  A step of the third takes 10 us: 5 the projections (the
// 64-bit multiply-adds; the integral column beside them 3), 1 the block maxima, 2 the
// exchange, 1 the choice of the pivot, 1 the pivot's data.  Rows beyond shared memory
// come from L2: read upwards only, 41,616 x 452 took 17 ms, in turn 14, and with the
// addresses advanced instead of formed anew 8.9.  Side by side, 100 molecules of 300
// pairs 5.8 -> 3.5, 12 of 2,485 to 66,430 pairs 102 -> 72.
#pragma once

namespace cds {

constexpr int kDirMaxPer = 3;               // pairs per thread of the column group
constexpr int kDirGroup = 256;              // widest column group
constexpr int kDirMaxCtas = 160;            // five lines per lane of a deciding warp
constexpr int kDirBoys = (kBoysPoints * kBoysStride + 1) / 2 * 2;   // whole 16-byte units
constexpr int kDirBits = 26;                // bits of lo
constexpr int kDirTop = 30;                 // bits of hi
constexpr int kDirMinExp = -960;
constexpr int kDirMaxRank = 4096;           // 2 x 2^55 x sqrt(4096) < 2^63
constexpr size_t kDirSmemMax = 220 * 1024;

// How the pairs of one molecule, or of several side by side, are laid out: pc per CTA.
struct DirectShape {
    int per, width, groups, pc, threads;
};
inline DirectShape direct_shape(int64_t each) {   // at least `each` pairs per CTA
    DirectShape s;
    s.per = (int)std::max<int64_t>(1, (each + kDirGroup - 1) / kDirGroup);
    s.width = (int)(((each + s.per - 1) / s.per + 31) / 32 * 32);
    s.pc = s.width * s.per;
    // Projection groups: enough threads to poll every line and to keep loads in flight, within
    // the block's registers.  These / one / two / three everywhere: 28,920 pairs x 372 3.41 /
    // 4.62 / 3.68 / 3.78 ms, 41,616 x 452 8.4 / 14.2 / 9.6 / 8.4, 5,050 x 200 1.00 / 1.10 / 0.99 /
    // 0.97, 300 x 120 0.67 / 0.69 / 0.65 / 0.65.
    s.groups = s.width <= 64 ? 7 : s.width <= 96 ? 6 : s.width <= 128 ? 5 : s.width <= 192 ? 3 : 2;
    s.threads = s.width * (1 + s.groups) + 32;
    return s;
}
inline int direct_ctas(int64_t n, const DirectShape& s) { return (int)((n + s.pc - 1) / s.pc); }

struct CdDirectArgs {
    int64_t n;
    DirectShape sh;
    int32_t cta0, ctas;    // its CTAs of the launch
    int32_t max_rank, kcap, srows;
    double* L;
    int2* Q;               // [kcap][n] rows as (hi, lo)
    double* sc;            // [n] 2^(e - 30)
    double* D;
    const uint8_t* cand;
    PairSoA pd;
    unsigned long long* words[2];   // [ctas][16]
    int32_t* piv;
    CdCtrl* ctrl;
    int32_t* err;
};

// The words of one launch: two sets of a 128-byte line per CTA, on lines of their own
// (they are read 16 bytes at a time) whatever the caller's workspace starts at.
constexpr size_t kDirWords = 2 * 16 * (size_t)kDirMaxCtas;
constexpr size_t kDirWordsRoom = kDirWords + 16;
inline unsigned long long* dir_words(unsigned long long* room) {
    return reinterpret_cast<unsigned long long*>(align_up((size_t)room, 128));
}

__host__ __device__ inline size_t direct_smem(const DirectShape& s, int32_t kcap, int32_t srows) {
    return (size_t)kDirBoys * 8 + (size_t)(kcap + 1) / 2 * 2 * 8 + (size_t)s.groups * s.pc * 16 +
           (size_t)s.pc * 6 * 8 + (size_t)srows * s.pc * 8;
}

__device__ __forceinline__ void ld_relaxed2(const unsigned long long* p, unsigned long long& x,
                                            unsigned long long& y) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void named_sync(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int count) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// TABLE: several molecules side by side (one shape), each on its own CTAs; else one.
template <int PER, bool TABLE>
__global__ void __launch_bounds__(kDirGroup * kDirMaxPer + 32, 1)
k_cd_direct(const __grid_constant__ CdDirectArgs one, const CdDirectArgs* table, int count) {
    extern __shared__ __align__(128) char dyn[];
    __shared__ CdDirectArgs s_args;
    __shared__ long long s_key[2][kDirMaxCtas];
    __shared__ uint32_t s_ix[2][kDirMaxCtas];
    __shared__ int2 s_fresh[2][kDirMaxCtas];
    __shared__ long long s_wmax[8], s_wmin[8];
    __shared__ uint32_t s_widx[8];
    __shared__ int2 s_new;
    __shared__ long long s_okey;
    __shared__ uint32_t s_oidx;
    __shared__ int s_amb, s_fail, s_best;
    __shared__ double s_rdp, s_dp;
    __shared__ long long s_pick;

    const int tid = threadIdx.x, lane = tid & 31;
    if constexpr (TABLE) {
        if (tid == 0) {
            int i = 0;
            while (i + 1 < count && table[i + 1].cta0 <= (int)blockIdx.x) ++i;
            s_args = table[i];
        }
        __syncthreads();
    }
    const CdDirectArgs& a = TABLE ? s_args : one;
    const int W = a.sh.width, G = a.sh.groups, pc = a.sh.pc, ncta = a.ctas;
    double* s_boys = reinterpret_cast<double*>(dyn);
    int2* s_lp = reinterpret_cast<int2*>(s_boys + kDirBoys);
    longlong2* s_part = reinterpret_cast<longlong2*>(s_lp + (a.kcap + 1) / 2 * 2);   // [G][pc]
    double* s_pd = reinterpret_cast<double*>(s_part + G * pc);   // [6][pc]: p, P, K/p, 2^(e - 30)
    int2* s_row = reinterpret_cast<int2*>(s_pd + 6 * pc);        // [srows][pc]

    const int cta = (int)blockIdx.x - a.cta0;
    const bool column = tid < W, decider = tid >= W * (1 + G);
    const int nwc = W >> 5;                      // warps of the column group
    CdCtrl* c = a.ctrl;
    if (c->done) return;
    const int64_t n = a.n, base = (int64_t)cta * pc;
    const double scale = c->scale, de = c->delta_eff, band = kTieRel * scale;
    const long long de_key = __double_as_longlong(de), band_bits = __double_as_longlong(band);
    const long long neg_key = key_of(-kNotPdRel * scale);
    long long P = c->P;
    double dp = c->DP;
    int from_line = -1;                          // the line that holds the newest row at P
    unsigned meets = 0;
    for (int i = tid; i < kBoysPoints * kBoysOrder; i += blockDim.x)
        s_boys[i / kBoysOrder * kBoysStride + i % kBoysOrder] = kBoysTaylor[i / kBoysOrder][i % kBoysOrder];
    if (tid == 0) { s_fail = 0; s_amb = 0; s_new = make_int2(0, 0); }
    // this thread's pairs (column group)
    double dreg[PER];
    bool creg[PER];
    if (column) {
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int64_t I = base + r * W + tid;
            const bool ok = I < n;
            dreg[r] = ok ? a.D[I] : 0.0;
            creg[r] = ok && a.cand[I];
            double* own = s_pd + r * W + tid;
            own[0] = ok ? a.pd.p[I] : 1.0;
            own[pc] = ok ? a.pd.Px[I] : 0.0;
            own[2 * pc] = ok ? a.pd.Py[I] : 0.0;
            own[3 * pc] = ok ? a.pd.Pz[I] : 0.0;
            own[4 * pc] = ok ? a.pd.Kp[I] : 0.0;
            // sqrt(D0_I), from the pair's factors where D0_I = 2 pi^(5/2) (K/p)^2 / sqrt(2 p)
            // itself leaves the normal range (pairs of centres far apart, L^K_I of 1e-150 and less)
            const double root = dreg[r] < 1e-290 ? own[4 * pc] * sqrt(kTwoPi52 * rsqrt(2.0 * own[0]))
                                                 : sqrt(dreg[r]);
            int e = 0;
            if (root > 0.0 && root < INFINITY) frexp(root, &e);     // root < 2^e
            e = max(e, kDirMinExp);                                 // 2^(e - 30) stays normal
            own[5 * pc] = ldexp(1.0, e - kDirTop);
            if (ok) a.sc[I] = own[5 * pc];
        }
    }
    __syncthreads();

    for (int32_t k = 0;; ++k) {
        const unsigned tag = (unsigned)k + 1u;
        const int par = k & 1;
        unsigned long long* words = par ? a.words[1] : a.words[0];
        if (column) {
            // the integral column at this thread's pairs
            double e[PER];
            {
                const double q = a.pd.p[P], qx = a.pd.Px[P], qy = a.pd.Py[P], qz = a.pd.Pz[P],
                             kq = a.pd.Kp[P];
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    double x, sm;
                    const double* own = s_pd + r * W + tid;
                    eri_xs(own[0], own[pc], own[2 * pc], own[3 * pc], q, qx, qy, qz, x, sm);
                    const double kk = own[4 * pc] * kq;
                    e[r] = eri_is_far(x, sm) ? eri_far(kk, x) : eri_near<kBoysStride>(kk, x, sm, s_boys);
                }
            }
            if (k > 0) {
                const double scP = __ldcg(a.sc + P);
                named_sync(1, W * (1 + G));
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    long long hh = 0, cr = 0;
                    for (int g = 0; g < G; ++g) {
                        const longlong2 v = s_part[g * pc + r * W + tid];
                        hh += v.x;
                        cr += v.y;
                    }
                    const double s = (double)hh + (double)cr * (1.0 / (1 << kDirBits));
                    e[r] -= s * s_pd[5 * pc + r * W + tid] * scP;
                }
            }
            named_sync(5, W + 32);               // 1 / sqrt(D_P)
            const double rDP = s_rdp;
            long long mx = -1, mn = LLONG_MAX, ck[PER];
            double l[PER];
            int2 qv[PER];
            uint32_t mi = kIdxNone;
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int64_t I = base + r * W + tid;
                ck[r] = -1;
                l[r] = e[r] * rDP;
                // 2^(56 - e) from the exponent of 2^(e - 30)
                const long long es = __double_as_longlong(s_pd[5 * pc + r * W + tid]) >> 52;
                const double up = __longlong_as_double((2 * 1023 + kDirBits - es) << 52);
                const long long q = __double2ll_rn(l[r] * up);
                const int lo = (int)((unsigned)q << (32 - kDirBits)) >> (32 - kDirBits);   // low bits, signed
                qv[r] = make_int2((int)((q - lo) >> kDirBits), lo);
                if (I < n) {
                    double d = dreg[r] - l[r] * l[r];
                    if (I == P) d = 0.0;
                    dreg[r] = d;
                    const long long bits = __double_as_longlong(d);
                    if (creg[r]) {
                        ck[r] = bits > 0 ? bits : 0LL;
                        if (ck[r] > mx) { mx = ck[r]; mi = (uint32_t)I; }
                    }
                    mn = min(mn, key_of(d));
                }
                if (k < a.srows) s_row[(int64_t)k * pc + r * W + tid] = qv[r];
            }
            const long long wm = redux_max(mx), wn = redux_min(mn);
            const uint32_t wi = __reduce_min_sync(0xffffffffu, mx == wm && mx >= 0 ? mi : kIdxNone);
            if (lane == 0) { s_wmax[tid >> 5] = wm; s_wmin[tid >> 5] = wn; s_widx[tid >> 5] = wi; }
            named_sync(3, W);
            const long long lm = lane < nwc ? s_wmax[lane] : -1, ln = lane < nwc ? s_wmin[lane] : LLONG_MAX;
            const uint32_t li = lane < nwc ? s_widx[lane] : kIdxNone;
            const long long bm = redux_max(lm);
            const uint32_t bi = __reduce_min_sync(0xffffffffu, lm == bm ? li : kIdxNone);
            const bool neg = __any_sync(0xffffffffu, ln < neg_key);
            const long long fk = band_floor_key(bm, band_bits);
            bool other = false;
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const uint32_t I = (uint32_t)(base + r * W + tid);
                other = other || (ck[r] >= fk && ck[r] > de_key && I != bi);
                if (I == bi) s_new = qv[r];
            }
            if (__any_sync(0xffffffffu, other) && lane == 0) s_amb = 1;
            if (tid == 0) {
                s_okey = neg ? LLONG_MAX : bm;   // too negative: above every number
                s_oidx = bm >= 0 ? bi : kIdxNone;
            }
            named_arrive(4, W + 32);             // the deciding warp stores the line
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int64_t I = base + r * W + tid;
                if (I < n) {
                    __stcs(a.L + (int64_t)k * n + I, l[r]);   // not read again here
                    a.Q[(int64_t)k * n + I] = qv[r];
                }
            }
        } else if (decider) {
            // the last row (at k = 0 the scales) before this step's words: fence and words by
            // the same threads, so a reader that acquires a word sees the rows behind it
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if (lane == 0) s_rdp = 1.0 / sqrt(dp);
            __syncwarp();
            named_arrive(5, W + 32);
            named_sync(4, W + 32);               // the column group's maximum
            const int2 f = s_new;
            const uint32_t v = lane == 0   ? (uint32_t)(s_okey >> 32)
                               : lane == 1 ? (uint32_t)s_okey
                               : lane == 2 ? (s_oidx | (s_amb ? kIdxAmbiguous : 0u))
                               : lane == 3 ? (uint32_t)f.x
                                           : (uint32_t)f.y;
            if (lane < 5) st_relaxed(words + (size_t)cta * 16 + lane, ((unsigned long long)v << 32) | tag);
            __syncwarp();
            if (lane == 0) s_amb = 0;
        } else {
            const int dt = tid - W;
            if (k > 0) {
                // the pivot's rows: the newest from its line (unless a tie scan, whose
                // meetings are fences, or the only CTA found the pivot)
                for (int K = dt; K < k; K += W * G)
                    s_lp[K] = (K == k - 1 && from_line >= 0) ? s_fresh[par ^ 1][from_line]
                                                             : __ldcg(a.Q + (int64_t)K * n + P);
                named_sync(2, W * G);
                const int g = dt / W, t = dt - g * W;
                long long hh[PER], cr[PER];
#pragma unroll
                for (int r = 0; r < PER; ++r) hh[r] = cr[r] = 0;
                const int ins = min(k, a.srows);
                auto add = [&](int r, int2 v, int2 lp) {
                    hh[r] += (long long)v.x * lp.x;
                    cr[r] += (long long)v.x * lp.y;
                    cr[r] += (long long)v.y * lp.x;
                };
                const int2* own = s_row + g * pc + t;
#pragma unroll 4
                for (int K = g; K < ins; K += G, own += G * pc) {
                    const int2 lp = s_lp[K];
#pragma unroll
                    for (int r = 0; r < PER; ++r) add(r, own[r * W], lp);
                }
                constexpr int kDepth = PER == 1 ? 16 : PER == 2 ? 8 : 4;
                // the rows beyond, upwards and downwards in turn: what a step reads last,
                // the next finds in L2
                int left = k - ins - g;
                const int2* lp = s_lp + (par ? k - 1 - g : ins + g);
                const int dl = par ? -G : G;
                const int2* row[PER];
                const int64_t dr = (int64_t)dl * n;
#pragma unroll
                for (int r = 0; r < PER; ++r)            // (dead lanes: any pair)
                    row[r] = a.Q + (int64_t)(par ? k - 1 - g : ins + g) * n + min(base + r * W + t, n - 1);
                for (; left > 0; left -= kDepth * G) {
                    int2 v[kDepth][PER];
#pragma unroll
                    for (int j = 0; j < kDepth; ++j)
#pragma unroll
                        for (int r = 0; r < PER; ++r) {
                            v[j][r] = j * G < left ? __ldcg(row[r]) : make_int2(0, 0);
                            row[r] += dr;
                        }
#pragma unroll
                    for (int j = 0; j < kDepth; ++j)
                        if (j * G < left) {
#pragma unroll
                            for (int r = 0; r < PER; ++r) add(r, v[j][r], *lp);
                            lp += dl;
                        }
                }
#pragma unroll
                for (int r = 0; r < PER; ++r)
                    s_part[g * pc + r * W + t] = make_longlong2(hh[r], cr[r]);
                named_arrive(1, W * (1 + G));
            }
            // every CTA's line of this step
            for (int j = dt; j < ncta; j += W * G) {
                const unsigned long long* f = words + (size_t)j * 16;
                unsigned long long w0, w1, w2, w3, w4, t0 = 0;
                for (unsigned it = 0;; ++it) {
                    ld_relaxed2(f, w0, w1);
                    ld_relaxed2(f + 2, w2, w3);
                    w4 = ld_acquire(f + 4);      // the rows behind the words
                    if ((unsigned)w0 == tag && (unsigned)w1 == tag && (unsigned)w2 == tag &&
                        (unsigned)w3 == tag && (unsigned)w4 == tag)
                        break;
                    if ((it & 255u) == 255u) {
                        const unsigned long long now = steps_timer();
                        if (!t0) t0 = now;
                        if (now - t0 > kStepsTimeoutNs || *(volatile int32_t*)a.err) {
                            atomicExch(a.err, (int32_t)CDS_ERR_TIMEOUT);
                            s_fail = 1;
                            break;
                        }
                    }
                }
                s_key[par][j] = (long long)((w0 & 0xffffffff00000000ull) | (w1 >> 32));
                s_ix[par][j] = (uint32_t)(w2 >> 32);
                s_fresh[par][j] = make_int2((int)(w3 >> 32), (int)(w4 >> 32));
            }
        }
        __syncthreads();
        if (s_fail) return;
        // the decision, alike in every warp of every CTA
        const int32_t made = k + 1;
        constexpr int kEach = kDirMaxCtas / 32;
        long long kk[kEach], A = -1;
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            const int j = lane + 32 * i;
            kk[i] = j < ncta ? s_key[par][j] : -1;
            A = max(A, kk[i]);
        }
        A = redux_max(A);
        int status = CDS_OK, from = -1;
        bool stop = true;
        if (A > 0x7ff0000000000000LL) {                     // a NaN's bits, or a negative residual
            status = CDS_ERR_NOT_PD;
        } else if (A <= de_key) {                           // G <= delta_eff (none: -1)
            status = CDS_OK;
        } else if (made >= a.max_rank) {
            status = CDS_ERR_RANK_CAP;
        } else {
            stop = false;
            // the lowest line whose maximum is in the band: with one line above the
            // band's (generous) integer floor that is the maximum's
            const long long fk = band_floor_key(A, band_bits);
            unsigned bl = 0xffffffffu;
            int cnt = 0;
#pragma unroll
            for (int i = 0; i < kEach; ++i) {
                const bool in = kk[i] >= fk && kk[i] > de_key;
                cnt += __popc(__ballot_sync(0xffffffffu, in));
                if (in && bl == 0xffffffffu) bl = (unsigned)(lane + 32 * i);
            }
            if (cnt != 1) {
                const double thr = __longlong_as_double(A) - band;
                const long long tk = thr > 0.0 ? __double_as_longlong(thr) : 0LL;
                bl = 0xffffffffu;
#pragma unroll
                for (int i = 0; i < kEach; ++i)
                    if (bl == 0xffffffffu && kk[i] >= tk && kk[i] > de_key) bl = (unsigned)(lane + 32 * i);
            }
            bl = __reduce_min_sync(0xffffffffu, bl);
            const uint32_t bx = s_ix[par][bl];
            dp = __longlong_as_double(s_key[par][bl]);
            if (bx & kIdxAmbiguous) {
                from = (int)bl;                             // several residuals in its band
            } else {
                P = (long long)(bx & kIdxNone);
                from_line = ncta > 1 ? (int)bl : -1;
            }
        }
        if (!stop && from >= 0) {   // the lowest index in the band, from the residuals themselves
            const double thr = __longlong_as_double(A) - band;
            const long long tk = thr > 0.0 ? __double_as_longlong(thr) : 0LL;
            int bl = from;
            for (;;) {
                // its owner stores the residuals; nobody scans before that, and nobody
                // changes residuals while another still scans
                if (column && bl == cta) {
#pragma unroll
                    for (int r = 0; r < PER; ++r) {
                        const int64_t I = base + r * W + tid;
                        if (I < n) a.D[I] = dreg[r];
                    }
                }
                if (tid == 0) s_best = INT_MAX;
                __syncthreads();
                if (tid == 0 && !steps_meet(c, ++meets * (unsigned)ncta, a.err)) s_fail = 1;
                __syncthreads();
                if (s_fail) return;
                for (int i = tid; i < pc; i += blockDim.x) {
                    const int64_t I = (int64_t)bl * pc + i;
                    if (I < n && a.cand[I]) {
                        const long long bits = __double_as_longlong(__ldcg(a.D + I));
                        if (bits > 0 && bits >= tk && bits > de_key) atomicMin(&s_best, (int)I);
                    }
                }
                __syncthreads();
                const int best = s_best;
                if (best != INT_MAX && tid == 0) { s_pick = best; s_dp = __ldcg(a.D + best); }
                if (tid == 0 && !steps_meet(c, ++meets * (unsigned)ncta, a.err)) s_fail = 1;
                __syncthreads();
                if (s_fail) return;
                if (best != INT_MAX) break;
                // the band reached below delta_eff: on to the next line that passes
                int nx = ncta;
                for (int j = bl + 1; j < ncta; ++j)
                    if (s_key[par][j] >= tk && s_key[par][j] > de_key) { nx = j; break; }
                if (nx == ncta) { stop = true; status = CDS_ERR_NOT_PD; break; }
                bl = nx;
            }
            if (!stop) { P = s_pick; dp = s_dp; }
            from_line = -1;
            __syncthreads();
        }
        if (stop) {
            if (column) {
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    const int64_t I = base + r * W + tid;
                    if (I < n) a.D[I] = dreg[r];
                }
            }
            if (cta == 0 && tid == 0) {
                c->status = status;
                c->done = 1;
                c->M = made;
            }
            return;
        }
        if (cta == 0 && tid == 0) a.piv[made] = (int32_t)P;
    }
}

// Rows that shared memory holds beside the rest.
inline int32_t direct_rows(const DirectShape& sh, int32_t kcap) {
    return (int32_t)std::min<size_t>(kcap, (kDirSmemMax - direct_smem(sh, kcap, 0)) / ((size_t)sh.pc * 8));
}

// One molecule (table null), or the count molecules of a table in device memory, of one
// shape, on ctas CTAs; smem: the most that one of them needs.  The caller has checked
// that the shape fits (direct_serves).
inline int launch_direct(const CdDirectArgs& one, const CdDirectArgs* table, int count, int ctas,
                         size_t smem, cudaStream_t stream) {
    void (*kern)(CdDirectArgs, const CdDirectArgs*, int) =
        table ? (one.sh.per == 1   ? k_cd_direct<1, true>
                 : one.sh.per == 2 ? k_cd_direct<2, true>
                                   : k_cd_direct<3, true>)
              : (one.sh.per == 1   ? k_cd_direct<1, false>
                 : one.sh.per == 2 ? k_cd_direct<2, false>
                                   : k_cd_direct<3, false>);
    CDS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDirSmemMax));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)one.sh.threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // its CTAs wait on one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, one, table, count));
    count_launches(1);
    return CDS_OK;
}

}  // namespace cds
