// Steps of the tensor-core Cholesky decomposition between two streaming passes,
// in one cooperative launch (included by cd.cu, after its helpers).
//
// A step is short: 2-3 us of arithmetic on the pairs of one SM, then a
// grid-wide maximum that the next step depends on.  As one kernel per step
// (the form this replaces: the update kernel, and the slicing and projection
// kernels returning at once) a step took 30 us at 217,000 live pairs, nearly all of
// it launches, cold loads and the serial end in the last block.  Here every CTA
// keeps its pairs and the steps go on inside the kernel until one needs a new
// pass or the decomposition stops:
//  - the update of cd_step_body, element by element the same arithmetic; the
//    pairs' data and their rows since the pass stay in shared memory, the
//    residuals in registers;
//  - each block of 512 pairs publishes {largest candidate residual, its lowest
//    index, flags, the new vector there} in 8-byte words that carry the step's
//    tag, so a reader sees data and arrival in one load (no counter, no second
//    round trip).  A CTA's words are one 128-byte line, written by one store: with
//    a line shared by several writers the readers' polls took it in turns with
//    the writes, 7 us a step;
//  - the fence behind a row (4-6 us when the column's warps waited for it) is made by
//    the deciding warp, which stores the words, while the others form the next column,
//    so a row is read by other CTAs from the step after the next on, and the newest
//    from the words;
//  - every CTA gathers all blocks' words and takes the same decision: stop test,
//    pivot, candidate slot.  A warp of its own decides, with integer keys, and
//    forms 1 / sqrt(D_P) while the others form the next column.
// Two word sets alternate: a CTA can publish step k + 2 only after every CTA has
// read step k.  When several residuals lie within the tie band of a block's
// maximum (a flag), its owner stores the block's residuals, all CTAs meet at a
// counter, scan them for the lowest index and meet again.
// Every wait is bounded and sets the error word instead of hanging.
// Measured, whole decompositions, update kernel per step -> this: 840 functions
// (899 steps, 54 passes) 42.3 -> 32.8 ms, 600 (1224 steps) 45.9 -> 30.7 ms, 240 (377
// steps) 10.4 -> 5.4 ms; the first 30.9 with the float pairs' conversions in integer
// operations here and in the digit store.  A step of it takes 13 us: 6 us the column,
// the rows since the pass and the residuals, 2 us the block maxima, 3 us the exchange.
#pragma once

namespace cds {

constexpr int kStepsMaxSub = 3;             // 256-thread sub-blocks per CTA
constexpr unsigned long long kStepsTimeoutNs = 2000000000ull;

struct CdStepsArgs {
    int64_t n;
    int32_t nblk, max_rank;
    int32_t srows;         // rows since the pass that shared memory holds
    double* L;             // compact vectors (float pairs)
    double* D;
    const uint8_t* cand;
    const float2* G;
    PairF2 pf;
    unsigned long long* words[2];   // [lines of 16]: per block key high, low, index and flags, the
                                    // new vector's pair; nsub blocks per line
    int32_t* piv;
    CdCtrl* ctrl;
    int32_t* err;
};

__device__ __forceinline__ unsigned long long steps_timer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ long long redux_max(long long v) {
    const int hi = __reduce_max_sync(0xffffffffu, (int)(v >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (int)(v >> 32) == hi ? (unsigned)v : 0u);
    return ((long long)hi << 32) | lo;
}
__device__ __forceinline__ long long redux_min(long long v) {
    const int hi = __reduce_min_sync(0xffffffffu, (int)(v >> 32));
    const unsigned lo = __reduce_min_sync(0xffffffffu, (int)(v >> 32) == hi ? (unsigned)v : 0xffffffffu);
    return ((long long)hi << 32) | lo;
}
__device__ __forceinline__ void sub_barrier(int sb) {
    asm volatile("bar.sync %0, 256;" ::"r"(1 + sb) : "memory");
}

// Key (bits of a positive double) at or below that of value - band, for the key
// of value >= 0: the band in units of value's last place, doubled for a lower binade.
__device__ __forceinline__ long long band_floor_key(long long key, long long band_bits) {
    const int e = (int)(key >> 52), eb = (int)(band_bits >> 52);
    if (e <= eb) return 0;
    const long long m = (band_bits & 0xfffffffffffffLL) | (1LL << 52);
    const long long ulps = e - eb < 53 ? (m >> (e - eb)) + 1 : 1;
    const long long f = key - 2 * ulps;
    return f > 0 ? f : 0;
}

constexpr uint32_t kIdxNone = 0x3fffffffu, kIdxAmbiguous = 0x40000000u, kIdxNegative = 0x80000000u;

// Shared memory of a CTA of nsub sub-blocks: the Boys table (rows padded to nine
// entries against bank conflicts), the gathered keys and indices, and, when
// every sub-block has one block (RES), its pairs' data and recent rows.
constexpr int kBoysStride = kBoysOrder + 1;
constexpr size_t kStepsBoys = ((size_t)kBoysMidPoints * kBoysStride * 8 + 127) / 128 * 128;
constexpr size_t kStepsSmemMax = 220 * 1024;
__host__ __device__ inline size_t steps_smem(int nblk, int nsub, bool res, int srows) {
    const size_t keys = ((size_t)nblk * 12 + 127) / 128 * 128;
    return kStepsBoys + keys + (res ? (size_t)nsub * kStepChunk * 8 * (5 + srows) : 0);
}

// One meeting of the CTAs at ctrl's counter (thread 0 of each; false: gave up).
__device__ __forceinline__ bool steps_meet(CdCtrl* c, unsigned target, int32_t* err) {
    __threadfence();
    atomicAdd(&c->_pad2, 1u);
    const unsigned long long t0 = steps_timer();
    for (unsigned it = 0; (int)(*(volatile unsigned*)&c->_pad2 - target) < 0; ++it)
        if ((it & 255u) == 255u && (steps_timer() - t0 > kStepsTimeoutNs || *(volatile int32_t*)err)) {
            atomicExch(err, (int32_t)CDS_ERR_TIMEOUT);
            return false;
        }
    __threadfence();
    return true;
}

// CTA cta of the ncta that work on one decomposition: blockDim.x = 256 threads per
// sub-block and a deciding warp.
template <bool RES>
__device__ __forceinline__ void cd_steps_body(const CdStepsArgs& a, int cta, int ncta, char* dyn) {
    __shared__ float2 s_lp[kBatchTC];
    __shared__ long long s_set[kSpecTC];
    __shared__ long long s_wmax[kStepsMaxSub][8], s_wmin[kStepsMaxSub][8];
    __shared__ uint32_t s_widx[kStepsMaxSub][8];
    // a block's results for the CTA's line; two sets, as a sub-block may be a turn
    // ahead of the warp that stores the line
    struct Block {
        long long bm;
        float2 fresh;
        uint32_t bi;
        int amb, neg;
    };
    __shared__ Block s_out[2][kStepsMaxSub];
    __shared__ long long s_gmax[kStepsMaxSub * 8 + 1];
    __shared__ uint32_t s_gj[kStepsMaxSub * 8 + 1];
    __shared__ int s_gflag[kStepsMaxSub * 8 + 1];
    __shared__ float2 s_rdp;
    __shared__ int s_fail;
    // the step's decision (written by the deciding warp)
    __shared__ long long s_pick;
    __shared__ double s_dp;
    __shared__ int s_status, s_stop, s_hit, s_from, s_bl, s_best;

    const int nblk = a.nblk;
    const int nsub = (int)(blockDim.x >> 8);
    float2* s_boys = reinterpret_cast<float2*>(dyn);
    dyn += kStepsBoys;
    long long* s_key = reinterpret_cast<long long*>(dyn);
    uint32_t* s_ix = reinterpret_cast<uint32_t*>(s_key + nblk);
    const int np = nsub * kStepChunk;            // pairs of this CTA (RES)
    float2* s_pf = reinterpret_cast<float2*>(dyn + ((size_t)nblk * 12 + 127) / 128 * 128);   // [5][np]
    float2* s_row = s_pf + 5 * np;               // [srows][np]

    const int tid = threadIdx.x, tt = tid & 255, sb = tid >> 8, lane = tid & 31;
    const int sw = tt >> 5;
    const bool decider = tid >= 256 * nsub;
    CdCtrl* c = a.ctrl;
    if (c->done) return;
    const int64_t n = a.n;
    float2* Lf = reinterpret_cast<float2*>(a.L);
    const double scale = c->scale, de = c->delta_eff, band = kTieRel * scale;
    const long long de_key = __double_as_longlong(de);
    const long long neg_key = key_of(-kNotPdRel * scale);
    const long long band_bits = __double_as_longlong(band);
    int32_t k = c->kstep;
    const int32_t k0 = c->k0;
    int32_t slot = c->slot, bl_prev = -1;
    long long P = c->P;
    unsigned int meets = (unsigned int)c->_pad4;     // meetings so far, all launches
    long long extra_sum = 0;
    for (int i = tid; i < kBoysMidPoints * kBoysOrder; i += blockDim.x)
        s_boys[i / kBoysOrder * kBoysStride + i % kBoysOrder] = kBoysTaylorF2[i / kBoysOrder][i % kBoysOrder];
    if (tid == 0) { s_rdp = c->rDPf; s_fail = 0; }
    if (tid < kSpecTC) s_set[tid] = c->STc[tid];
    if (tid < 2 * kStepsMaxSub) {
        s_out[tid & 1][tid >> 1].amb = 0;
        s_out[tid & 1][tid >> 1].fresh = make_float2(0.f, 0.f);
    }
    const int per = RES ? 1 : (nblk + ncta * nsub - 1) / (ncta * nsub);
    // RES: this thread's pairs
    double dreg[kStepPer];
    bool creg[kStepPer];
    if (RES && !decider) {
        const int b = cta * nsub + sb;
#pragma unroll
        for (int q = 0; q < kStepPer; ++q) {
            const int64_t I = (int64_t)b * kStepChunk + q * kUpdThreads + tt;
            const int j = sb * kStepChunk + q * kUpdThreads + tt;
            const bool ok = b < nblk && I < n;
            dreg[q] = ok ? a.D[I] : 0.0;
            creg[q] = ok && a.cand[I];
            s_pf[0 * np + j] = ok ? a.pf.p[I] : make_float2(1.f, 0.f);
            s_pf[1 * np + j] = ok ? a.pf.Px[I] : make_float2(0.f, 0.f);
            s_pf[2 * np + j] = ok ? a.pf.Py[I] : make_float2(0.f, 0.f);
            s_pf[3 * np + j] = ok ? a.pf.Pz[I] : make_float2(0.f, 0.f);
            s_pf[4 * np + j] = ok ? a.pf.Kp[I] : make_float2(0.f, 0.f);
        }
    }
    const PairF2 pfs = RES ? PairF2{s_pf, s_pf + np, s_pf + 2 * np, s_pf + 3 * np, s_pf + 4 * np} : a.pf;

    for (;;) {
        const int32_t extra = k - k0;
        const unsigned tag = (unsigned)k + 1u;
        unsigned long long* words = (k & 1) ? a.words[1] : a.words[0];
        // the pivot's column of the rows since the pass: the newest from the words of
        // its block (unless a tie scan, whose meetings are fences, or the only CTA
        // found the pivot), the others from the rows
        if (tid < extra) {
            if (bl_prev >= 0 && tid == extra - 1) {
                const unsigned long long* f = ((k & 1) ? a.words[0] : a.words[1]) +
                                              (size_t)(bl_prev / nsub) * 16 + bl_prev % nsub * 5 + 3;
                unsigned long long x, y, t0 = 0;
                for (unsigned it = 0;; ++it) {
                    x = ld_relaxed(f);
                    y = ld_relaxed(f + 1);
                    if ((unsigned)x == (unsigned)k && (unsigned)y == (unsigned)k) break;
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
                s_lp[tid] = make_float2(__uint_as_float((unsigned)(x >> 32)),
                                        __uint_as_float((unsigned)(y >> 32)));
            } else {
                s_lp[tid] = __ldcg(Lf + (int64_t)(k0 + tid) * n + P);
            }
        }
        PivotF2 pv;
        if (!decider) pv = pivot_f2(a.pf, P);
        __syncthreads();
        if (s_fail) return;
        if (!decider) {
            const float2* Gs = a.G + (int64_t)slot * n;
            bool have_rdp = false;
            for (int r = 0; r < per; ++r) {
                const int b = (r * ncta + cta) * nsub + sb;
                const bool on = b < nblk;            // the same in the whole sub-block
                const int64_t base = (int64_t)b * kStepChunk;
                float2 e[kStepPer];
                if (on) {
                    float2 acc[kStepPer];
#pragma unroll
                    for (int q = 0; q < kStepPer; ++q) {
                        const int64_t I = base + q * kUpdThreads + tt;
                        acc[q] = (k0 > 0 && I < n) ? Gs[I] : make_float2(0.f, 0.f);
                    }
                    const int ins = RES ? min(extra, a.srows) : 0;   // rows in shared memory
                    if constexpr (RES) {
                        const float2* row = s_row + sb * kStepChunk + tt;
                        for (int i = 0; i < ins; ++i, row += np) {
                            const float2 lp = s_lp[i];
#pragma unroll
                            for (int q = 0; q < kStepPer; ++q) df_fma(acc[q], row[q * kUpdThreads], lp);
                        }
                    }
                    constexpr int kDepth = 4;
                    for (int i0 = ins; i0 < extra; i0 += kDepth) {
                        float2 v[kStepPer][kDepth];
#pragma unroll
                        for (int q = 0; q < kStepPer; ++q) {
                            const int64_t I = base + q * kUpdThreads + tt;
#pragma unroll
                            for (int j = 0; j < kDepth; ++j)
                                v[q][j] = (I < n && i0 + j < extra) ? Lf[(int64_t)(k0 + i0 + j) * n + I]
                                                                    : make_float2(0.f, 0.f);
                        }
#pragma unroll
                        for (int j = 0; j < kDepth; ++j)
                            if (i0 + j < extra) {
                                const float2 lp = s_lp[i0 + j];
#pragma unroll
                                for (int q = 0; q < kStepPer; ++q) df_fma(acc[q], v[q][j], lp);
                            }
                    }
#pragma unroll
                    for (int q = 0; q < kStepPer; ++q) {
                        const int64_t I = base + q * kUpdThreads + tt;
                        const int64_t src = RES ? (int64_t)(sb * kStepChunk + q * kUpdThreads + tt) : I;
                        if (I < n)
                            e[q] = df_add(eri_elem_df<kBoysStride>(pfs, src, pv, s_boys), df_neg(acc[q]));
                    }
                }
                if (!have_rdp) {   // 1 / sqrt(D_P) from the deciding warp
                    asm volatile("bar.sync 5, %0;" ::"r"((int)blockDim.x) : "memory");
                    have_rdp = true;
                }
                if (!on) continue;
                const float2 rDPf = s_rdp;
                long long mx = -1, mn = LLONG_MAX, ck[kStepPer];
                float2 lf[kStepPer];
                uint32_t mi = kIdxNone;
#pragma unroll
                for (int q = 0; q < kStepPer; ++q) {
                    const int64_t I = base + q * kUpdThreads + tt;
                    ck[q] = -1;
                    lf[q] = make_float2(0.f, 0.f);
                    if (I < n) {
                        lf[q] = df_mul(e[q], rDPf);
                        if (RES && extra < a.srows)
                            s_row[(int64_t)extra * np + sb * kStepChunk + q * kUpdThreads + tt] = lf[q];
                        const float2 l2 = df_mul(lf[q], lf[q]);
                        double d = (RES ? dreg[q] : a.D[I]) - double_of(l2);
                        if (I == P) d = 0.0;
                        if (RES) dreg[q] = d;
                        else a.D[I] = d;
                        const long long bits = __double_as_longlong(d);
                        if (RES ? creg[q] : a.cand[I] != 0) {
                            ck[q] = bits > 0 ? bits : 0LL;
                            if (ck[q] > mx) { mx = ck[q]; mi = (uint32_t)I; }
                        }
                        mn = min(mn, key_of(d));
                    }
                }
                const long long wm = redux_max(mx), wn = redux_min(mn);
                const uint32_t wi =
                    __reduce_min_sync(0xffffffffu, mx == wm && mx >= 0 ? mi : kIdxNone);
                if (lane == 0) { s_wmax[sb][sw] = wm; s_wmin[sb][sw] = wn; s_widx[sb][sw] = wi; }
                sub_barrier(sb);
                const long long lm = s_wmax[sb][lane & 7], ln = s_wmin[sb][lane & 7];
                const uint32_t li = s_widx[sb][lane & 7];
                const long long bm = redux_max(lm);
                const uint32_t bi = __reduce_min_sync(0xffffffffu, lm == bm ? li : kIdxNone);
                const bool neg = __any_sync(0xffffffffu, ln < neg_key);
                Block& out = s_out[r & 1][sb];
                const long long floor_key = band_floor_key(bm, band_bits);
                bool other = false;
#pragma unroll
                for (int q = 0; q < kStepPer; ++q) {
                    const uint32_t I = (uint32_t)(base + q * kUpdThreads + tt);
                    other = other || (ck[q] >= floor_key && ck[q] > de_key && I != bi);
                    if (I == bi) out.fresh = lf[q];   // the new vector at the block's maximum
                }
                if (__any_sync(0xffffffffu, other) && lane == 0) out.amb = 1;
                if (tt == 0) { out.bm = bm; out.bi = bi; out.neg = neg; }
                // the deciding warp stores the line of this turn's blocks
                const int on_sub = min(nsub, nblk - (r * ncta + cta) * nsub);
                asm volatile("bar.sync 6, %0;" ::"r"(256 * on_sub + 32) : "memory");
#pragma unroll
                for (int q = 0; q < kStepPer; ++q) {
                    const int64_t I = base + q * kUpdThreads + tt;
                    if (I < n) Lf[(int64_t)k * n + I] = lf[q];
                }
            }
        } else {
            // the last row before this step's words: fence and words by the same threads, so a
            // reader that acquires a word sees the rows behind it
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if (k > k0 && lane == 0) {   // (the first step's comes with the state)
                const double rDP = 1.0 / sqrt(s_dp);
                const float h = (float)rDP;
                s_rdp = make_float2(h, (float)(rDP - (double)h));
            }
            __syncwarp();
            asm volatile("bar.arrive 5, %0;" ::"r"((int)blockDim.x) : "memory");
            // the CTA's blocks of each turn, one line by one store
            for (int r = 0; r < per; ++r) {
                const int on_sub = min(nsub, nblk - (r * ncta + cta) * nsub);
                if (on_sub <= 0) break;
                asm volatile("bar.sync 6, %0;" ::"r"(256 * on_sub + 32) : "memory");
                const int q = lane / 5, f = lane - 5 * q;
                if (q < on_sub) {
                    const Block& o = s_out[r & 1][q];
                    const uint32_t ix = (o.bm >= 0 ? o.bi : kIdxNone) | (o.amb ? kIdxAmbiguous : 0u) |
                                        (o.neg ? kIdxNegative : 0u);
                    const uint32_t v = f == 0   ? (uint32_t)(o.bm >> 32)
                                       : f == 1 ? (uint32_t)o.bm
                                       : f == 2 ? ix
                                       : f == 3 ? __float_as_uint(o.fresh.x)
                                                : __float_as_uint(o.fresh.y);
                    st_relaxed(words + (size_t)(r * ncta + cta) * 16 + lane, ((unsigned long long)v << 32) | tag);
                }
                __syncwarp();
                if (lane < kStepsMaxSub) s_out[r & 1][lane].amb = 0;
            }
        }
        // gather every block's words of this step; each warp keeps its largest key,
        // the block it is in, and whether another of its blocks is in that key's band
        {
            unsigned long long t0 = 0;
            long long g1 = -1, g2 = -1;      // this thread's two largest keys
            uint32_t gj = 0xffffffffu;
            bool gneg = false;
            for (int j = tid; j < nblk; j += blockDim.x) {
                const unsigned long long* f = words + (size_t)(j / nsub) * 16 + j % nsub * 5;
                unsigned long long w0, w1, w2;
                for (unsigned it = 0;; ++it) {
                    w0 = ld_relaxed(f);
                    w1 = ld_relaxed(f + 1);
                    w2 = ld_relaxed(f + 2);
                    if ((unsigned)w0 == tag && (unsigned)w1 == tag && (unsigned)w2 == tag) break;
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
                const long long key = (long long)((w0 & 0xffffffff00000000ull) | (w1 >> 32));
                s_key[j] = key;
                s_ix[j] = (uint32_t)(w2 >> 32);
                gneg = gneg || (w2 >> 63);
                if (key > g1) { g2 = g1; g1 = key; gj = (uint32_t)j; }
                else g2 = max(g2, key);
            }
            asm volatile("fence.acq_rel.gpu;" ::: "memory");   // the rows behind the words
            const long long wm = redux_max(g1);
            const uint32_t wj = __reduce_min_sync(0xffffffffu, g1 == wm ? gj : 0xffffffffu);
            const long long fk = band_floor_key(max(wm, 0LL), band_bits);
            const bool multi = __any_sync(0xffffffffu, (g1 >= fk && gj != wj) || g2 >= fk);
            gneg = __any_sync(0xffffffffu, gneg);
            if (lane == 0) {
                s_gmax[tid >> 5] = wm;
                s_gj[tid >> 5] = wj;
                s_gflag[tid >> 5] = (multi ? 1 : 0) | (gneg ? 2 : 0);
            }
        }
        __syncthreads();
        if (s_fail) return;
        const int32_t made = k + 1;
        if (decider) {   // the decision, alike in every CTA
            const int nw = (int)(blockDim.x >> 5);
            const long long gm = lane < nw ? s_gmax[lane] : -1;
            const int gf = lane < nw ? s_gflag[lane] : 0;
            const long long A = redux_max(gm);
            const bool neg = __any_sync(0xffffffffu, gf & 2);
            int status = CDS_OK, stop = 1, from = -1;
            unsigned bl = 0xffffffffu;
            long long pick = -1;
            if (neg || A > 0x7ff0000000000000LL) {          // a NaN's bits
                status = CDS_ERR_NOT_PD;
            } else if (A <= de_key) {                       // G <= delta_eff (none: -1)
                status = CDS_OK;
            } else if (made >= a.max_rank) {
                status = CDS_ERR_RANK_CAP;
            } else {
                // the lowest block whose maximum is in the band: with one block above
                // the band's (generous) integer floor that is the maximum's
                const long long fk = band_floor_key(A, band_bits);
                const unsigned in = __ballot_sync(0xffffffffu, gm >= fk && gm > de_key);
                const unsigned mu = __ballot_sync(0xffffffffu, gm >= fk && (gf & 1));
                if (__popc(in) == 1 && !(mu & in)) {
                    if (in & (1u << lane)) bl = s_gj[lane];
                } else {
                    const double thr = __longlong_as_double(A) - band;
                    const long long tk = thr > 0.0 ? __double_as_longlong(thr) : 0LL;
                    for (int j = lane; j < nblk; j += 32)
                        if (s_key[j] >= tk && s_key[j] > de_key) { bl = (unsigned)j; break; }
                }
                bl = __reduce_min_sync(0xffffffffu, bl);
                stop = 0;                                   // the maximum's block passes
                const uint32_t ix = s_ix[bl];
                if (ix & kIdxAmbiguous) from = (int)bl;     // several residuals in its band
                else pick = (long long)(ix & kIdxNone);
            }
            const unsigned m = __ballot_sync(0xffffffffu, !stop && s_set[lane] == pick);
            if (lane == 0) {
                s_status = status;
                s_stop = stop;
                s_from = from;
                s_bl = from < 0 && !stop && ncta > 1 ? (int)bl : -1;
                s_pick = pick;
                if (!stop) s_dp = __longlong_as_double(s_key[bl]);
                s_hit = (!stop && m && made - k0 < kBatchTC) ? 31 - __clz(m) : -1;
            }
        }
        __syncthreads();
        if (s_from >= 0) {   // the lowest index in the band, from the residuals themselves
            const double thr = [&] {
                long long A = -1;
                for (int j = 0; j < nblk; ++j) A = max(A, s_key[j]);
                return __longlong_as_double(A) - band;
            }();
            const long long tk = thr > 0.0 ? __double_as_longlong(thr) : 0LL;
            int bl = s_from;
            for (;;) {
                // its owner stores the block's residuals; nobody scans before that,
                // and nobody changes residuals while another still scans
                if (RES && !decider && bl == cta * nsub + sb) {
#pragma unroll
                    for (int q = 0; q < kStepPer; ++q) {
                        const int64_t I = (int64_t)bl * kStepChunk + q * kUpdThreads + tt;
                        if (I < n) a.D[I] = dreg[q];
                    }
                }
                if (tid == 0) s_best = INT_MAX;
                __syncthreads();
                if (tid == 0 && !steps_meet(c, ++meets * (unsigned)ncta, a.err)) s_fail = 1;
                __syncthreads();
                if (s_fail) return;
                for (int i = tid; i < kStepChunk; i += blockDim.x) {
                    const int64_t I = (int64_t)bl * kStepChunk + i;
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
                // the band reached below delta_eff: on to the next block that passes
                int nx = nblk;
                for (int j = bl + 1; j < nblk; ++j)
                    if (s_key[j] >= tk && s_key[j] > de_key) { nx = j; break; }
                if (nx == nblk) {
                    if (tid == 0) { s_stop = 1; s_status = CDS_ERR_NOT_PD; }
                    break;
                }
                bl = nx;
            }
            __syncthreads();
            if (decider) {
                const bool go = s_stop == 0;
                const unsigned m = __ballot_sync(0xffffffffu, go && s_set[lane] == s_pick);
                if (lane == 0) s_hit = (go && m && made - k0 < kBatchTC) ? 31 - __clz(m) : -1;
            }
            __syncthreads();
        }
        const bool stop = s_stop != 0;
        const long long pick = s_pick;
        const int hit = s_hit;
        if (!stop && hit >= 0) {
            extra_sum += made - k0;
            slot = hit;
            P = pick;
            bl_prev = s_bl;
            k = made;
            if (cta == 0 && tid == 0) a.piv[made] = (int32_t)pick;
            continue;
        }
        if (RES && !decider) {
#pragma unroll
            for (int q = 0; q < kStepPer; ++q) {
                const int64_t I = (int64_t)(cta * nsub + sb) * kStepChunk + q * kUpdThreads + tt;
                if (cta * nsub + sb < nblk && I < n) a.D[I] = dreg[q];
            }
        }
        if (cta != 0) return;
        // CTA 0 leaves the state for the next pass (or the host)
        if (!stop) {
            // the candidates after the pivot: the eligible blocks' maxima by (maximum
            // descending, block index ascending).  Each block's rank is the number of
            // blocks before it in that order; ranks below 31 are taken.
            if (tid < kSpecTC) s_set[tid] = tid == 0 ? pick : -1;
            __syncthreads();
            for (int j = tid; j < nblk; j += blockDim.x) {
                const uint32_t ix = s_ix[j] & kIdxNone;
                const long long key = s_key[j];
                const bool ok = ix != kIdxNone && (long long)ix != pick && key > de_key;
                if (!ok) continue;
                int rank = 0;
                for (int i = 0; i < nblk; ++i) {
                    const long long o = s_key[i];
                    if (o < key || (o == key && i >= j)) continue;
                    const uint32_t ox = s_ix[i] & kIdxNone;
                    rank += (ox != kIdxNone && (long long)ox != pick && o > de_key) ? 1 : 0;
                }
                if (rank < kSpecTC - 1) s_set[rank + 1] = (long long)ix;
            }
            __syncthreads();
            if (tid < kSpecTC) c->STc[tid] = s_set[tid];
        }
        if (tid == 0) {
            c->_pad4 = (int32_t)meets;
            c->extra += extra_sum;
            c->kstep = made;
            if (stop) {
                c->status = s_status;
                c->done = 1;
                c->M = made;
            } else {
                const double rDP = 1.0 / sqrt(s_dp);
                const float h = (float)rDP;
                c->P = pick;
                c->DP = s_dp;
                c->rDP = rDP;
                c->rDPf = make_float2(h, (float)(rDP - (double)h));
                a.piv[made] = (int32_t)pick;
                c->kdone = k0;   // the store holds the rows before the last pass's step
                c->k0 = made;
                c->slot = 0;
                c->pass = 1;
                c->passes += 1;
                c->streamed += made;
            }
        }
        return;
    }
}

template <bool RES>
__global__ void __launch_bounds__(256 * kStepsMaxSub + 32, 1) k_cd_steps_tc(const CdStepsArgs a) {
    extern __shared__ __align__(128) char dyn[];
    cd_steps_body<RES>(a, blockIdx.x, gridDim.x, dyn);
}

// Sub-blocks per CTA and CTAs for nblk blocks on nsm SMs: as many SMs as there are
// blocks, then up to three blocks side by side on each, then several in turn.
inline int steps_sub(int nblk, int nsm) {
    return std::max(1, std::min(kStepsMaxSub, (nblk + nsm - 1) / nsm));
}

inline int launch_steps(CdStepsArgs a, int nsm, cudaStream_t stream) {
    const int sub = steps_sub(a.nblk, nsm);
    const int ctas = std::max(1, std::min(nsm, (a.nblk + sub - 1) / sub));
    const bool res = a.nblk <= ctas * sub;
    // rows that fit beside the pairs' data
    const size_t fixed = steps_smem(a.nblk, sub, res, 0);
    a.srows = res ? (int)std::min<size_t>(kBatchTC, (kStepsSmemMax - fixed) / ((size_t)sub * kStepChunk * 8)) : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)(256 * sub + 32));
    cfg.dynamicSmemBytes = steps_smem(a.nblk, sub, res, a.srows);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // its CTAs wait on one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto kern = res ? k_cd_steps_tc<true> : k_cd_steps_tc<false>;
    CDS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kStepsSmemMax));
    CDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, a));
    return CDS_OK;
}

}  // namespace cds
