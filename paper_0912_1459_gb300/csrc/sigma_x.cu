// FP64 self-energy (paper Eq. SE) in two passes per group of orbitals:
//   1. the MO integrals X^t[x][(j, b)] = sum_J Lp^J_tx Lov^J_jb of the group, an
//      FP64-accurate tensor-core product (dgemm_tc.cu), into a scratch of
//      kScratch bytes or one orbital's integrals (0.8 GB at 840 functions);
//   2. k_sigma_x: numerators (2 X_xy - X_yx) X_xy and the energy denominators.
// The fused kernel this replaces formed the integrals with FP64 FMAs, which
// the part issues at 2 a clock and SM: 0.14 s for an orbital of that basis.
// Writing and reading the scratch costs 0.25 ms of HBM time per orbital.
// Where that and the sliced factors (18 bytes per element of Lov and Lp) would take more
// than kWorkspace bytes, or more than the caller's workspace, the spectators are taken in
// panels, as many at once as fit: the virtual ones of the first sum, then the occupied
// ones of the second, for each panel one orbital after another; the blocks add to
// their partial sums from panel to panel.
//
// Pass 2 is bound by the FP64 pipe as well, so its energies are grouped.  For
// a grid of more than kDirect energies with centre E0 and half width h, an
// element with denominator h (c + x), x = (E - E0) / h in [-1, 1], |c| > 1, is
//   1 / (c + x) = sgn(c) / sqrt(c^2 - 1) [1 + 2 sum_k v^k T_k(x)],
//   v = -sgn(c) (|c| - sqrt(c^2 - 1)),
// the Chebyshev expansion of a simple pole, so K moments sum n w v^k serve all
// energies of the grid: 2 K + 18 FP64 operations per element instead of 7 per
// element and energy.  K is chosen per 32 x 32 tile from the smallest |c| in it so
// that the remainder is below 2^-56 (10 to 32 terms for |c| from 290 down to
// 2.06); a tile with a pole nearer than that is evaluated energy by energy.
#include "dgemm_tc.cuh"
#include "sigma_x.cuh"
#include "tcgen05.cuh"

namespace cds {

namespace sx {

constexpr int TB = 32;                      // pair-index block, as k_sigma_fp64
constexpr int kItem = TB * TB;
constexpr int kDirect = 8;                  // energies evaluated one by one
constexpr int kZone = 64;                   // energies served by one set of moments
constexpr int kMom = 32;                    // moments at most
constexpr int kPartC = kMom + 2 * kZone;    // partials of a block, moment form
constexpr int kPartD = 2 * kDirect;         // partials of a block, direct form (2 for one energy)
constexpr int part_stride(int32_t nE) { return nE == 1 ? 2 : nE <= kDirect ? kPartD : kPartC; }
constexpr int kBlocks = 608;                // blocks of a launch: 4 per SM
constexpr int kThreads = 256;
constexpr int64_t kScratch = 512LL << 20;
constexpr size_t kWorkspace = (size_t)4 << 30;   // asked for at most

struct XTerm {
    int32_t nx, ns, nb, npb;
    int32_t xoff;              // row of x = 0 in an orbital's block of X
    int64_t per;               // items of a launch per orbital: the term's, or a panel's
    int64_t item0, cper;       // cached items: first of the launch, per orbital
    int64_t cs, cy;            // column of (s, y): s cs + y cy
    const double *eps_s, *eps_x;
};

struct XArgs {
    XTerm tm[2];
    const double* X;           // [orbital of the group][rows][ncols]
    int64_t tstride, ncols;
    const double* E;
    int32_t nE, t0;
    const int32_t* active;
    double* cache;             // numerators: written when X is given, else read
    double* part;
    int32_t add;               // a later panel: add to the partial sums
};

// Sum of each of N values over the warp with N - 1 + 5 - log2 N adds: value
// index of a lane = its top log2 N lane bits (bit 4 first).
template <int N>
__device__ __forceinline__ double warp_sums(double (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const double send = up ? v[i] : v[i + n];
            const double keep = up ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (; o; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// Terms of the expansion for a pole at |c| >= z: with rho = z + sqrt(z^2 - 1)
// the remainder after K terms is below rho^(3 - K) 2^-4 < 2^-56 relative, also
// for the derivative's k^2 at the ends of the interval.  0: evaluate directly.
__device__ __forceinline__ int terms_for(float z) {
    if (!(z >= 2.06f)) return 0;
    return z >= 290.f ? 10 : z >= 39.f ? 12 : z >= 10.1f ? 16 : z >= 5.05f ? 20
           : z >= 3.3f ? 24 : z >= 2.5f ? 28 : 32;
}

// MODE 1: one energy; 2: up to kDirect energies, each evaluated; 3: moments.
// Threads as in k_sigma_fp64: thread (tr, tc) holds the 2 x 2 elements x = A 32 + 2
// tr + i, y = B 32 + 2 tc + j.  A block takes items of one orbital in turn
// and keeps its sums in registers across them (fixed order), so it meets at
// barriers only at the end.
template <int MODE, bool FROM_CACHE>
__global__ void __launch_bounds__(kThreads, 2)
k_sigma_x(const XArgs a) {
    extern __shared__ float s_rng[];            // MODE 3: [blocks of both terms][min, max]
    __shared__ double s_sum[MODE == 3 ? 8 : 1][MODE == 3 ? 2 * kZone : 1];
    __shared__ double s_red[8][MODE == 3 ? kMom : kPartD];
    const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
    const int lane = tid & 31, w = tid >> 5;
    const int tl = blockIdx.y, t = a.t0 + tl;
    if (a.active && !a.active[t]) return;
    const int e_first = MODE == 3 ? blockIdx.z * kZone : 0;
    const int ne = MODE == 3 ? min(kZone, a.nE - e_first) : a.nE;
    const double* Et = a.E + (int64_t)t * a.nE + e_first;
    double E0 = 0.0, hinv = 0.0;
    float fh = 0.f;
    constexpr int NS = MODE == 1 ? 1 : MODE == 2 ? kDirect : 1;
    double sv[NS], dv[NS], Ee[NS];
    double mom[MODE == 3 ? kMom : 1];
    if constexpr (MODE == 3) {
        double lo = Et[0], hi = Et[0];
        for (int e = 1; e < ne; ++e) {
            const double v = Et[e];
            lo = v < lo ? v : lo;
            hi = v > hi ? v : hi;
        }
        E0 = 0.5 * (lo + hi);
        const double h = 0.5 * (hi - lo);
        hinv = 1.0 / h;
        fh = (float)h;
#pragma unroll
        for (int k = 0; k < kMom; ++k) mom[k] = 0.0;
        // range of e_x over each 32-block of both terms
        for (int b = w; b < a.tm[0].nb + a.tm[1].nb; b += kThreads / 32) {
            const XTerm& q = a.tm[b < a.tm[0].nb ? 0 : 1];
            const int x = (b < a.tm[0].nb ? b : b - a.tm[0].nb) * TB + lane;
            float mn = x < q.nx ? (float)q.eps_x[x] : INFINITY;
            float mx = x < q.nx ? (float)q.eps_x[x] : -INFINITY;
            if (mn != mn) mx = INFINITY;        // NaN: the range admits everything
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            }
            if (lane == 0) { s_rng[2 * b] = mn; s_rng[2 * b + 1] = mx; }
        }
        for (int i = tid; i < 8 * 2 * kZone; i += kThreads) s_sum[i / (2 * kZone)][i % (2 * kZone)] = 0.0;
        __syncthreads();
    } else {
#pragma unroll
        for (int e = 0; e < NS; ++e) {
            sv[e] = dv[e] = 0.0;
            Ee[e] = Et[min(e, ne - 1)];
        }
    }

    const int64_t n0 = a.tm[0].per, ntot = n0 + a.tm[1].per;
    for (int64_t it = blockIdx.x; it < ntot; it += gridDim.x) {
        const bool second = it >= n0;
        const XTerm& q = a.tm[second ? 1 : 0];
        const int nx = q.nx;
        const uint32_t r = (uint32_t)(second ? it - n0 : it);
        const int s = (int)(r / (uint32_t)q.npb);
        int A, B;
        block_pair(r - (uint32_t)s * (uint32_t)q.npb, q.nb, A, B);
        const int x0 = A * TB + tr * 2, y0 = B * TB + tc * 2;
        double num[4], base[4];
        const double es = q.eps_s[s];
        double* citem = a.cache ? a.cache + (q.item0 + (int64_t)t * q.cper + r) * kItem + tid : nullptr;
        {
            const double* X = a.X + (int64_t)tl * a.tstride + (int64_t)s * q.cs;
            double exv[2], eyv[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                exv[i] = x0 + i < nx ? q.eps_x[x0 + i] : 0.0;
                eyv[i] = y0 + i < nx ? q.eps_x[y0 + i] : 0.0;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int x = x0 + (k >> 1), y = y0 + (k & 1);
                const bool ok = x < nx && y < nx;
                if constexpr (FROM_CACHE) {
                    num[k] = citem[k * kThreads];
                } else {
                    const double x1 = ok ? X[(int64_t)(q.xoff + x) * a.ncols + (int64_t)y * q.cy] : 0.0;
                    const double x2 = ok ? X[(int64_t)(q.xoff + y) * a.ncols + (int64_t)x * q.cy] : 0.0;
                    // fused operations spelled out, so every form rounds alike
                    num[k] = A == B ? fma(2.0, x1, -x2) * x1
                                    : 2.0 * fma(x1, x1, fma(x2, x2, -__dmul_rn(x1, x2)));
                }
                if (!ok) num[k] = 0.0;
                base[k] = ok ? es - exv[k >> 1] - eyv[k & 1] : 1e30;   // padding: 0 / 1e30
            }
            if (!FROM_CACHE && citem && (MODE != 3 || blockIdx.z == 0)) {
#pragma unroll
                for (int k = 0; k < 4; ++k) citem[k * kThreads] = num[k];
            }
        }
        if constexpr (MODE != 3) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int e = 0; e < NS; ++e) {
                    const double rc = recip(Ee[e] + base[k]);
                    sv[e] = fma(num[k], rc, sv[e]);
                    dv[e] = fma(-__dmul_rn(num[k], rc), rc, dv[e]);
                }
        } else {
            const int bo = second ? a.tm[0].nb : 0;
            const float mA = s_rng[2 * (bo + A)], MA = s_rng[2 * (bo + A) + 1];
            const float mB = s_rng[2 * (bo + B)], MB = s_rng[2 * (bo + B) + 1];
            const float f0 = (float)E0 + (float)es;
            const float cl = f0 - MA - MB, ch = f0 - mA - mB;
            const float slack = 1e-6f * (fabsf(f0) + fabsf(MA) + fabsf(MB) + fabsf(mA) + fabsf(mB));
            const float z = ((cl > 0.f ? cl : ch < 0.f ? -ch : 0.f) - slack) / fh;
            // the same in the whole block; infinite or NaN energies, h = 0: evaluate
            const int K = fabsf(cl) < 1e30f && fabsf(ch) < 1e30f && z < 1e30f ? terms_for(z) : 0;
            if (K) {
                double p[4], v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const double c = (E0 + base[k]) * hinv;
                    const double ac = fabs(c);
                    const double s2 = fma(ac, ac, -1.0);
                    const double rs = rsqrt(s2);
                    double u = fma(-s2, rs, ac);                  // |c| - sqrt(c^2 - 1)
                    u = fma(fma(u, fma(-2.0, ac, u), 1.0), 0.5 * rs, u);   // u^2 - 2 |c| u + 1 = 0
                    v[k] = c > 0.0 ? -u : u;
                    const double wn = num[k] * rs;
                    p[k] = c > 0.0 ? wn : -wn;
                }
                if (base[0] == 1e30) p[0] = v[0] = 0.0;           // padding may overflow above
                if (base[1] == 1e30) p[1] = v[1] = 0.0;
                if (base[2] == 1e30) p[2] = v[2] = 0.0;
                if (base[3] == 1e30) p[3] = v[3] = 0.0;
#pragma unroll
                for (int k0 = 0; k0 < kMom; k0 += 2) {
                    if (k0 < K) {
#pragma unroll
                        for (int k = k0; k < k0 + 2; ++k) {
                            mom[k] += (p[0] + p[1]) + (p[2] + p[3]);
#pragma unroll
                            for (int j = 0; j < 4; ++j) p[j] *= v[j];
                        }
                    }
                }
            } else {
                for (int e = 0; e < ne; e += 4) {
                    double q8[8];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const double Ej = Et[min(e + j, ne - 1)];
                        double sj = 0.0, dj = 0.0;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const double rc = recip(Ej + base[k]);
                            sj = fma(num[k], rc, sj);
                            dj = fma(-__dmul_rn(num[k], rc), rc, dj);
                        }
                        q8[2 * j] = sj;
                        q8[2 * j + 1] = dj;
                    }
                    const double tot = warp_sums<8>(q8);
                    const int vi = lane >> 2;
                    if ((lane & 3) == 0 && e + (vi >> 1) < ne) s_sum[w][2 * e + vi] += tot;
                }
            }
        }
    }

    // the block's sums, warps added in order
    if constexpr (MODE == 3) {
        double* out = a.part + (((int64_t)t * gridDim.z + blockIdx.z) * gridDim.x + blockIdx.x) * kPartC;
        const double m = warp_sums<kMom>(mom);
        s_red[w][lane] = m;                      // value index of a lane: the lane itself
        __syncthreads();
        if (tid < kMom) {
            double v = 0.0;
#pragma unroll
            for (int j = 0; j < 8; ++j) v += s_red[j][tid];
            out[tid] = a.add ? out[tid] + v : v;
        }
        for (int i = tid; i < 2 * ne; i += kThreads) {
            double v = 0.0;
#pragma unroll
            for (int j = 0; j < 8; ++j) v += s_sum[j][i];
            out[kMom + i] = a.add ? out[kMom + i] + v : v;
        }
    } else {
        double* out = a.part + ((int64_t)t * gridDim.x + blockIdx.x) * (2 * NS);
#pragma unroll
        for (int e = 0; e < NS; ++e) {
            double q2[2] = {sv[e], dv[e]};
            const double tot = warp_sums<2>(q2);
            if ((lane & 15) == 0) s_red[w][2 * e + (lane >> 4)] = tot;
        }
        __syncthreads();
        if (tid < 2 * ne) {
            double v = 0.0;
#pragma unroll
            for (int j = 0; j < 8; ++j) v += s_red[j][tid];
            out[tid] = a.add ? out[tid] + v : v;
        }
    }
}

// (s, c) += x: s the rounded sum, c the rounding errors (two-sum).
__device__ __forceinline__ void add_comp(double& s, double& c, double x) {
    const double t = s + x;
    const double v = t - s;
    c += (s - (t - v)) + (x - v);
    s = t;
}

// sigma / dsigma of one orbital (blockIdx.x) and energy zone (blockIdx.y) from
// the blocks' partials, added in order; NaN if a device-side wait gave up.
__global__ void __launch_bounds__(kThreads)
k_sigma_x_final(const double* __restrict__ part, int32_t nblk, int32_t nE,
                const double* __restrict__ E, const int32_t* __restrict__ active, bool moments,
                const int32_t* __restrict__ err, double* __restrict__ sigma,
                double* __restrict__ dsigma) {
    const int t = blockIdx.x, tid = threadIdx.x;
    if (active && !active[t]) return;
    const bool bad = err && *err;
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    __shared__ double s_acc[8][kPartC], s_low[8][kMom];
    const int stride = moments ? kPartC : nE == 1 ? 2 : kPartD;
    const int e_first = moments ? blockIdx.y * kZone : 0;
    const int ne = moments ? min(kZone, nE - e_first) : nE;
    const int nval = moments ? kMom + 2 * ne : 2 * ne;
    const double* p = part + ((int64_t)t * gridDim.y + blockIdx.y) * nblk * stride;
    // eight runs of blocks, each summed in order, then the runs in order
    const int run = tid >> 5, lane = tid & 31;
    const int b0 = (int)((int64_t)nblk * run / 8), b1 = (int)((int64_t)nblk * (run + 1) / 8);
    for (int i = lane; i < nval; i += 32) {
        double v = 0.0, c = 0.0;
        for (int b = b0; b < b1; ++b) add_comp(v, c, p[(int64_t)b * stride + i]);
        s_acc[run][i] = v;
        if (i < kMom) s_low[run][i] = c;
    }
    __syncthreads();
    for (int i = tid; i < nval; i += kThreads) {
        double v = 0.0, c = 0.0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            add_comp(v, c, s_acc[j][i]);
            if (i < kMom) c += s_low[j][i];
        }
        s_acc[0][i] = v;
        if (i < kMom) s_low[0][i] = c;
    }
    __syncthreads();
    const double* Et = E + (int64_t)t * nE + e_first;
    for (int e = tid; e < ne; e += kThreads) {
        double s, d;
        if (moments) {
            double lo = Et[0], hi = Et[0];
            for (int j = 1; j < ne; ++j) {
                const double v = Et[j];
                lo = v < lo ? v : lo;
                hi = v > hi ? v : hi;
            }
            const double hinv = 1.0 / (0.5 * (hi - lo));
            const double x = (Et[e] - 0.5 * (lo + hi)) * hinv;
            // sum A_k T_k and sum k A_k U_(k-1) (T_k' = k U_(k-1)) by Clenshaw's
            // recurrence, smallest terms first; the leading terms with their low
            // parts, so the result is rounded about once (as a direct sum's)
            double f1 = 0.0, f2 = 0.0, g1 = 0.0, g2 = 0.0;
            for (int k = kMom - 1; k >= 1; --k) {
                const double A = s_acc[0][k];
                const double fn = fma(2.0 * x, f1, -f2) + A;
                const double gl = fma(2.0 * x, g1, -g2);
                const double gn = k == 1 ? A + (s_low[0][1] + gl) : fma(A, (double)k, gl);
                f2 = f1; f1 = fn;
                g2 = g1; g1 = gn;
            }
            const double f = 2.0 * fma(x, f1, -f2);
            double top = s_acc[0][0], low = s_low[0][0];
            add_comp(top, low, f);
            s = fma(top, hinv, low * hinv);
            const double h2 = hinv * hinv, h2l = fma(hinv, hinv, -h2);
            d = 2.0 * fma(g1, h2, g1 * h2l);
            if (!(hinv > 0.0 && hinv < INFINITY)) s = d = 0.0;   // no moments were made
            s += s_acc[0][kMom + 2 * e];
            d += s_acc[0][kMom + 2 * e + 1];
        } else {
            s = s_acc[0][2 * e];
            d = s_acc[0][2 * e + 1];
        }
        sigma[(int64_t)t * nE + e_first + e] = bad ? nan : s;
        if (dsigma) dsigma[(int64_t)t * nE + e_first + e] = bad ? nan : d;
    }
}

static void set_term(XTerm& q, int32_t nx, int32_t ns, int32_t xoff, int64_t cs, int64_t cy,
                     const double* eps_s, const double* eps_x) {
    q.nx = nx;
    q.ns = ns;
    q.nb = nblocks_of(nx, TB);
    q.npb = (int32_t)npairs_of(q.nb);
    q.per = q.cper = nx > 0 && ns > 0 ? (int64_t)ns * q.npb : 0;
    q.xoff = xoff;
    q.cs = cs;
    q.cy = cy;
    q.eps_s = eps_s;
    q.eps_x = eps_x;
}

// Both sums of Eq. SE over X^t[x][(j, b)] (x over all orbitals, nv columns per j).
static void sigma_terms(XArgs& a, int32_t nmo, int32_t nocc, int32_t np, const double* eps) {
    const int32_t nv = nmo - nocc;
    set_term(a.tm[0], nocc, nv, 0, 1, nv, eps ? eps + nocc : nullptr, eps);
    set_term(a.tm[1], nv, nocc, nocc, nv, 1, eps, eps ? eps + nocc : nullptr);
    a.tm[0].item0 = 0;
    a.tm[1].item0 = (int64_t)np * a.tm[0].per;
}

// Orbitals whose integrals are held at once, and blocks per orbital.
static int32_t group_of(int64_t per_orbital, int32_t np) {
    return (int32_t)std::max<int64_t>(1, std::min<int64_t>(np, kScratch / (per_orbital * 8)));
}
static int32_t blocks_of(int64_t items, int32_t group) {
    return (int32_t)std::max<int64_t>(1, std::min<int64_t>(items, (kBlocks + group - 1) / group));
}

static int eval(const XArgs& a, int32_t norb, int32_t nblk, bool from_cache, cudaStream_t stream) {
    const bool moments = a.nE > kDirect;
    const unsigned nz = moments ? (unsigned)((a.nE + kZone - 1) / kZone) : 1u;
    const dim3 grid((unsigned)nblk, (unsigned)norb, nz);
    const size_t sm = moments ? (size_t)(a.tm[0].nb + a.tm[1].nb) * 2 * sizeof(float) : 0;
    if (from_cache)
        k_sigma_x<1, true><<<grid, kThreads, 0, stream>>>(a);
    else if (a.nE == 1)
        k_sigma_x<1, false><<<grid, kThreads, 0, stream>>>(a);
    else if (!moments)
        k_sigma_x<2, false><<<grid, kThreads, 0, stream>>>(a);
    else
        k_sigma_x<3, false><<<grid, kThreads, sm, stream>>>(a);
    CDS_LAUNCH_CHECK();
    return CDS_OK;
}

static int final_sum(const XArgs& a, int32_t np, int32_t nblk, const int32_t* err, double* sigma,
                     double* dsigma, cudaStream_t stream) {
    const bool moments = a.nE > kDirect;
    const unsigned nz = moments ? (unsigned)((a.nE + kZone - 1) / kZone) : 1u;
    k_sigma_x_final<<<dim3((unsigned)np, nz), kThreads, 0, stream>>>(
        a.part, nblk, a.nE, a.E, a.active, moments, err, sigma, dsigma);
    CDS_LAUNCH_CHECK();
    return CDS_OK;
}

struct Layout {
    dx::Operand ov, p;
    double *X, *part;
    int32_t* err;            // error word
    int32_t group, nblk;
    // in panels (width[1] > 0): spectators of either sum held at once, their operand and X
    int32_t width[2];
    dx::Operand pan[2];
    double* pX[2];
    size_t bytes;
};

// Everything at once.  rows: rows of one orbital's block of X (all orbitals, or the virtual
// ones for MP2).
static Layout layout(void* ws, int32_t nmo, int32_t nocc, int32_t M, int32_t np, int32_t nE,
                     int32_t rows, int64_t items) {
    const int64_t ov = (int64_t)nocc * (nmo - nocc);
    // bulk copies want 16-byte addresses whatever the caller's workspace starts at
    Carver c(ws ? (void*)align_up((size_t)ws) : nullptr);
    Layout l{};
    l.ov = dx::carve(c, 1, ov, M, dx::kRowsA);
    l.p = dx::carve(c, np, rows, M, dx::kRowsB);
    l.group = group_of(rows * ov, np);
    l.nblk = blocks_of(items, l.group);
    l.X = c.take<double>((size_t)l.group * rows * ov);
    const size_t nz = nE > kDirect ? (size_t)(nE + kZone - 1) / kZone : 1;
    l.part = c.take<double>((size_t)np * nz * l.nblk * part_stride(nE));
    l.err = c.take<int32_t>(1);
    l.bytes = c.off + 256;
    return l;
}

// One orbital and a panel of spectators at a time, panels of equal width and as wide as
// `bytes` allow; .bytes = 0 where a panel of kPanelRows rows does not fit (narrower ones
// leave the tensor cores idle, the fused kernel then serves).
static Layout panel_layout(void* ws, size_t bytes, int32_t nmo, int32_t nocc, int32_t M, int32_t np,
                           int32_t nE, bool mp2, int64_t items) {
    constexpr int64_t kPanelRows = 1024;
    const int32_t nv = nmo - nocc;
    Carver c(ws ? (void*)align_up((size_t)ws) : nullptr);
    Layout l{};
    l.p = dx::carve(c, 1, mp2 ? nv : std::max(nocc, nv), M, dx::kRowsB);
    l.group = 1;
    l.nblk = blocks_of(items, 1);
    const size_t nz = nE > kDirect ? (size_t)(nE + kZone - 1) / kZone : 1;
    l.part = c.take<double>((size_t)np * nz * l.nblk * part_stride(nE));
    l.err = c.take<int32_t>(1);
    size_t most = 0;
    for (int k = mp2 ? 1 : 0; k < 2; ++k) {
        const int32_t total = k ? nocc : nv, nx = k ? nv : nocc;
        auto take = [&](int32_t w) {         // both sums use the same memory in turn
            Carver q = c;
            l.pan[k] = dx::carve(q, 1, (int64_t)w * nx, M, dx::kRowsA);
            l.pX[k] = q.take<double>((size_t)w * nx * nx);
            return q.off + 256;
        };
        int32_t lo = 0, hi = total;          // the widest that fits
        while (lo < hi) {
            const int32_t mid = lo + (hi - lo + 1) / 2;
            if (take(mid) <= bytes) lo = mid; else hi = mid - 1;
        }
        if (lo == 0 || (lo < total && (int64_t)lo * nx < kPanelRows)) return Layout{};
        const int32_t n = (total + lo - 1) / lo;
        l.width[k] = (total + n - 1) / n;
        most = std::max(most, take(l.width[k]));
    }
    l.bytes = most;
    return l;
}

// The layout for a workspace of `bytes` bytes; .bytes = 0: too small for either.
static Layout layout_in(void* ws, size_t bytes, int32_t nmo, int32_t nocc, int32_t M, int32_t np,
                        int32_t nE, bool mp2, int64_t items) {
    const Layout l = layout(ws, nmo, nocc, M, np, nE, mp2 ? nmo - nocc : nmo, items);
    return l.bytes <= bytes ? l : panel_layout(ws, bytes, nmo, nocc, M, np, nE, mp2, items);
}

// X of orbitals [t0, t0 + n).
static int integrals(const Layout& l, int64_t ov, int32_t rows, int32_t M, const double* Lov,
                     const double* Q, int32_t t0, int32_t n, const int32_t* active,
                     cudaStream_t stream) {
    return dx::gemm(l.ov, dx::RowMajor{Lov, 0, M}, l.p, dx::RowMajor{Q, rows, M}, M, t0, t0 + n,
                    dx::Out{l.X, INT64_MAX, 0, 1, (int64_t)rows * ov, ov}, active, l.err, stream);
}

}  // namespace sx

using namespace sx;

bool sigma_x_serves(int32_t nmo, int32_t nocc, int32_t np) {
    const int64_t nv = nmo - nocc, ov = nocc * nv;
    // 32-bit item indices per orbital; orbitals in grid.y
    return nmo >= 64 && nocc > 0 && nv > 0 && np > 0 && np <= 65535 && ov < (1 << 22) && nmo <= (1 << 14) &&
           tc::device_ok();
}

static int64_t sigma_items(int32_t nmo, int32_t nocc, int32_t np) {
    XArgs a{};
    sigma_terms(a, nmo, nocc, np, nullptr);
    return a.tm[0].per + a.tm[1].per;
}

size_t sigma_x_bytes(int32_t nmo, int32_t nocc, int32_t M, int32_t np, int32_t nE) {
    return layout_in(nullptr, kWorkspace, nmo, nocc, M, np, nE, false, sigma_items(nmo, nocc, np)).bytes;
}

bool sigma_x_fits(int32_t nmo, int32_t nocc, int32_t M, int32_t np, int32_t nE, size_t ws_bytes) {
    return layout_in(nullptr, ws_bytes, nmo, nocc, M, np, nE, false, sigma_items(nmo, nocc, np)).bytes > 0;
}

// One sum's panel: spectators [s0, s0 + ns) of term k, whose columns of X are panel columns.
static void set_panel(XArgs& a, const XArgs& all, int k, int32_t s0, int32_t ns) {
    XTerm& q = a.tm[k];
    a.tm[0].per = a.tm[1].per = 0;
    a.tm[0].nb = a.tm[1].nb = 0;
    q = all.tm[k];
    q.ns = ns;
    q.per = (int64_t)ns * q.npb;
    q.item0 += (int64_t)s0 * q.npb;
    q.eps_s += s0;
    q.xoff = 0;
    if (k == 0) q.cy = ns;           // columns (j, a)
}

// Orbitals [0, np) over the panels: q(t): the rows of orbital t's operand that a sum takes.
template <typename Rows>
static int panels(XArgs a, const Layout& l, int32_t nocc, int32_t nv, int32_t M, const double* Lov, int32_t np,
                  Rows q, cudaStream_t stream) {
    const XArgs all = a;
    int st = CDS_OK;
    bool first = true;
    for (int k = l.width[0] > 0 ? 0 : 1; k < 2; ++k) {
        const int32_t total = k ? nocc : nv, nx = k ? nv : nocc;
        a.X = l.pX[k];
        for (int32_t s0 = 0; s0 < total; s0 += l.width[k], first = false) {
            const int32_t ns = std::min(l.width[k], total - s0);
            const int64_t cols = (int64_t)ns * nx;
            const dx::Operand A = dx::sized(l.pan[k], cols, dx::kRowsA);
            const dx::PanelRows occ{Lov + (int64_t)s0 * M, nv, M, ns};
            const dx::RowMajor vir{Lov + (int64_t)s0 * nv * M, 0, M};
            st = k ? dx::slice(vir, A, dx::kRowsA, M, stream) : dx::slice(occ, A, dx::kRowsA, M, stream);
            if (st) return st;
            set_panel(a, all, k, s0, ns);
            a.ncols = cols;
            a.add = first ? 0 : 1;
            for (int32_t t = 0; t < np; ++t) {
                const dx::RowMajor b{q(t, k), 0, M};
                const dx::Operand B = dx::sized(l.p, nx, dx::kRowsB);
                const dx::Out out{l.pX[k], INT64_MAX, 0, 1, 0, cols};
                const int32_t* on = a.active ? a.active + t : nullptr;
                if ((st = dx::slice(b, B, dx::kRowsB, M, stream))) return st;
                st = k ? dx::gemm(A, vir, B, b, M, 0, 1, out, on, l.err, stream)
                       : dx::gemm(A, occ, B, b, M, 0, 1, out, on, l.err, stream);
                if (st) return st;
                a.t0 = t;
                if ((st = eval(a, 1, l.nblk, false, stream))) return st;
            }
        }
    }
    return CDS_OK;
}

int sigma2_x(int32_t nmo, int32_t nocc, int32_t M, const double* Lov, const double* Lp, int32_t np,
             const double* eps, const double* E, int32_t nE, const int32_t* active, double* sigma,
             double* dsigma, void* ws, size_t ws_bytes, cudaStream_t stream, bool resplit, double* cache) {
    const int64_t ov = (int64_t)nocc * (nmo - nocc);
    XArgs a{};
    sigma_terms(a, nmo, nocc, np, eps);
    const Layout l = layout_in(ws, ws_bytes, nmo, nocc, M, np, nE, false, a.tm[0].per + a.tm[1].per);
    if (!l.bytes) return CDS_ERR_WORKSPACE;
    a.X = l.X;
    a.tstride = (int64_t)nmo * ov;
    a.ncols = ov;
    a.E = E;
    a.nE = nE;
    a.active = active;
    a.cache = cache;
    a.part = l.part;
    int st = CDS_OK;
    if (resplit || l.width[1] > 0) CDS_CUDA_TRY(cudaMemsetAsync(l.err, 0, sizeof(int32_t), stream));
    if (l.width[1] > 0) {
        st = panels(a, l, nocc, nmo - nocc, M, Lov, np,
                    [&](int32_t t, int k) { return Lp + ((int64_t)t * nmo + (k ? nocc : 0)) * M; }, stream);
        return st ? st : final_sum(a, np, l.nblk, l.err, sigma, dsigma, stream);
    }
    if (resplit) {
        if ((st = dx::slice(dx::RowMajor{Lov, 0, M}, l.ov, dx::kRowsA, M, stream))) return st;
        if ((st = dx::slice(dx::RowMajor{Lp, nmo, M}, l.p, dx::kRowsB, M, stream))) return st;
    }
    for (int32_t t0 = 0; t0 < np; t0 += l.group) {
        const int32_t n = std::min(l.group, np - t0);
        if (resplit || l.group < np)
            if ((st = integrals(l, ov, nmo, M, Lov, Lp, t0, n, active, stream))) return st;
        a.t0 = t0;
        if ((st = eval(a, n, l.nblk, false, stream))) return st;
    }
    return final_sum(a, np, l.nblk, l.err, sigma, dsigma, stream);
}

int sigma2_x_cached(int32_t nmo, int32_t nocc, int32_t np, const double* eps, const double* E,
                    const int32_t* active, const double* cache, double* sigma, double* dsigma,
                    double* part, cudaStream_t stream) {
    XArgs a{};
    sigma_terms(a, nmo, nocc, np, eps);
    const int64_t ov = (int64_t)nocc * (nmo - nocc);
    const int32_t nblk = blocks_of(a.tm[0].per + a.tm[1].per, group_of(nmo * ov, np));
    a.E = E;
    a.nE = 1;
    a.active = active;
    a.cache = const_cast<double*>(cache);
    a.part = part;
    const int st = eval(a, np, nblk, true, stream);
    if (st) return st;
    return final_sum(a, np, nblk, nullptr, sigma, dsigma, stream);
}

// MP2: the second sum with q := i, spectator j, E := e_i; both operands are rows of Lov.
static void mp2_terms(XArgs& a, int32_t nmo, int32_t nocc, const double* eps) {
    const int32_t nv = nmo - nocc;
    set_term(a.tm[0], 0, 0, 0, 0, 0, eps, eps);
    set_term(a.tm[1], nv, nocc, 0, nv, 1, eps, eps ? eps + nocc : nullptr);
}

static int64_t mp2_items(int32_t nmo, int32_t nocc) {
    XArgs a{};
    mp2_terms(a, nmo, nocc, nullptr);
    return a.tm[1].per;
}

size_t mp2_x_bytes(int32_t nmo, int32_t nocc, int32_t M) {
    return layout_in(nullptr, kWorkspace, nmo, nocc, M, nocc, 1, true, mp2_items(nmo, nocc)).bytes;
}

bool mp2_x_fits(int32_t nmo, int32_t nocc, int32_t M, size_t ws_bytes) {
    return layout_in(nullptr, ws_bytes, nmo, nocc, M, nocc, 1, true, mp2_items(nmo, nocc)).bytes > 0;
}

int mp2_x(int32_t nmo, int32_t nocc, int32_t M, const double* Lov, const double* eps,
          double* e_pair, void* ws, size_t ws_bytes, cudaStream_t stream) {
    const int32_t nv = nmo - nocc;
    const int64_t ov = (int64_t)nocc * nv;
    XArgs a{};
    mp2_terms(a, nmo, nocc, eps);
    const Layout l = layout_in(ws, ws_bytes, nmo, nocc, M, nocc, 1, true, a.tm[1].per);
    if (!l.bytes) return CDS_ERR_WORKSPACE;
    CDS_CUDA_TRY(cudaMemsetAsync(l.err, 0, sizeof(int32_t), stream));
    a.X = l.X;
    a.tstride = (int64_t)nv * ov;
    a.ncols = ov;
    a.E = eps;
    a.nE = 1;
    a.part = l.part;
    int st = CDS_OK;
    if (l.width[1] > 0) {
        st = panels(a, l, nocc, nv, M, Lov, nocc,
                    [&](int32_t t, int) { return Lov + (int64_t)t * nv * M; }, stream);
        return st ? st : final_sum(a, nocc, l.nblk, l.err, e_pair, nullptr, stream);
    }
    st = dx::slice(dx::RowMajor{Lov, 0, M}, l.ov, dx::kRowsA, M, stream);
    if (st) return st;
    if ((st = dx::slice(dx::RowMajor{Lov, nv, M}, l.p, dx::kRowsB, M, stream)))
        return st;
    for (int32_t t0 = 0; t0 < nocc; t0 += l.group) {
        const int32_t n = std::min(l.group, nocc - t0);
        if ((st = integrals(l, ov, nv, M, Lov, Lov, t0, n, nullptr, stream))) return st;
        a.t0 = t0;
        if ((st = eval(a, n, l.nblk, false, stream))) return st;
    }
    return final_sum(a, nocc, l.nblk, l.err, e_pair, nullptr, stream);
}

}  // namespace cds
