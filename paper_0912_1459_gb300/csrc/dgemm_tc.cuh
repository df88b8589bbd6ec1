// FP64 matrix products on the tensor cores by exact slices (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, 2012): D[n][m] = sum_k A[m][k]
// B[n][k] from operands stored as eight signed base-256 digits per element.
//
// A row is scaled by 2^ex > max|x| of the row, q = round(x 2^(62-ex)) (exact
// for every entry within 2^-9 of the row's largest, to 2^-63 of the scale
// otherwise), and q is cut into eight digits d_0 (most significant, |d_0| <= 64)
// .. d_7 in [-128, 127], each exact in BF16.  The 36 digit products with s + t <= 7
// are kept.  In units of both rows' scales the result of K columns is off by at most
// K 2^-58.9: 7 x 2^14 x 2^-76 a column from the dropped products with s + t = 8, 2^-62
// from the rounding of q, 2^-61 from FP32 sums beyond 2^24 (weights 6 and 7 of columns
// whose low digits agree).  Digits of unrelated numbers leave sqrt(K) 2^-62.
//
// That is a bound on the rows' scales, where a sum of FP64 products is good to K 2^-53
// S, S = sum_k |a_k||b_k|, however small S is beside them.  So a second pass forms S,
// from the magnitudes of the operands in BF16 (rounded down), and takes the results
// with S < 2^-5 of the scales again, each as an FP64 sum over the rows themselves:
// every result is good to K 2^-53 S.  Rows that are not finite, or beyond 2^+-400, have
// magnitudes of zero and are all taken so.
#pragma once

#include "common.cuh"

namespace cds {
namespace dx {

constexpr int kRowsA = 128;   // rows per tile of an A operand (MMA M)
constexpr int kRowsB = 64;    // rows per tile of a B operand
constexpr int kStepK = 16;    // columns per k-step (one MMA k)
constexpr int kDigits = 8;

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

// round(x 2^(62 - ex)), halves away from zero, for |x| < 2^ex.
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

// BF16 bits of |x| 2^-ex, |x| < 2^ex, rounded down (0 below 2^-126).
__device__ __forceinline__ uint32_t magnitude(double x, int ex) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ffull) - 896 - ex;
    return e > 0 ? ((uint32_t)e << 7) | ((uint32_t)(b >> 45) & 0x7fu) : 0u;
}

// One sliced operand: tiles of R rows, each [k-step][digit][R rows x 32
// bytes], already in the order and 32-byte swizzle the MMA reads, so a k-step
// of a tile is one contiguous bulk copy; mag the same with |x| / 2^ex in place of
// the digits.  Rows come in groups of `per` that start on a tile boundary (per =
// all rows for a plain matrix).
struct Operand {
    uint8_t *img, *mag;
    int32_t* ex;       // scale exponent per padded row
    int64_t groups, per, per_pad;
    int32_t ksteps;
};
inline int32_t ksteps_of(int32_t kdim) { return (kdim + kStepK - 1) / kStepK; }
inline int64_t padded_rows(int64_t per, int R) { return (per + R - 1) / R * R; }
inline Operand carve(Carver& c, int64_t groups, int64_t per, int32_t kdim, int R) {
    Operand o;
    o.groups = groups;
    o.per = per;
    o.per_pad = padded_rows(per, R);
    o.ksteps = ksteps_of(kdim);
    const size_t rows = (size_t)(groups * o.per_pad);
    o.img = c.take<uint8_t>(rows * o.ksteps * kDigits * kStepK * 2);
    o.mag = c.take<uint8_t>(rows * o.ksteps * kStepK * 2);
    o.ex = c.take<int32_t>(rows);
    return o;
}

// The same memory for another number of rows (at most those it was carved for).
inline Operand sized(Operand o, int64_t rows, int R) {
    o.per = rows;
    o.per_pad = padded_rows(rows, R);
    return o;
}

// Row sources: row(g, r)[k] is element k of row r of group g.  kAcross: neighbouring
// rows, not neighbouring k, lie side by side in memory.
struct RowMajor {         // x[(g gs + r) ld + k]
    static constexpr bool kAcross = false;
    const double* x;
    int64_t gs, ld;
    struct Row {
        const double* x;
        __device__ __forceinline__ double operator[](int k) const { return x[k]; }
    };
    __device__ __forceinline__ Row row(int64_t g, int64_t r) const { return {x + (g * gs + r) * ld}; }
};
struct PanelRows {        // row (j, a), a < an: x[(j nv + a) ld + k]
    static constexpr bool kAcross = false;
    const double* x;
    int64_t nv, ld;
    int32_t an;
    __device__ __forceinline__ RowMajor::Row row(int64_t, int64_t r) const {
        return {x + ((r / an) * nv + r % an) * ld};
    }
};
struct PackedRows {       // rows (K, nu): A^K[nu][k] of the packed symmetric vectors
    static constexpr bool kAcross = false;
    const double* L;
    int64_t npair;
    int32_t K0, N;
    struct Row {
        const double* L;
        int nu;
        __device__ __forceinline__ double operator[](int k) const {
            const int hi = max(k, nu), lo = min(k, nu);
            return L[(int64_t)hi * (hi + 1) / 2 + lo];
        }
    };
    __device__ __forceinline__ Row row(int64_t, int64_t r) const {
        return {L + (int64_t)(K0 + (int)(r / N)) * npair, (int)(r % N)};
    }
};
struct Columns {          // row j: C[k][col(j)], col(j) = j < nocc ? j : orb[j - nocc]
    static constexpr bool kAcross = true;
    const double* C;
    const int32_t* orb;
    int32_t nmo, nocc, first;
    struct Row {
        const double* C;      // null: no such orbital, NaN
        int64_t ld;
        __device__ __forceinline__ double operator[](int k) const {
            return C ? C[k * ld] : __longlong_as_double(0x7ff8000000000000LL);
        }
    };
    __device__ __forceinline__ Row row(int64_t, int64_t r) const {
        int q = (int)r + first;
        if (orb && q >= nocc) q = orb[q - nocc];
        return {q >= 0 && q < nmo ? C + q : nullptr, nmo};
    }
};

// Slice an operand (R = kRowsA or kRowsB).
int slice(const RowMajor& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream);
int slice(const PanelRows& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream);
int slice(const PackedRows& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream);
int slice(const Columns& src, const Operand& o, int R, int32_t kdim, cudaStream_t stream);

// out[(m / kdiv) m_hi + (m % kdiv) m_lo + (g - g0) g_s + n n_s] for the rows m of
// A (one group) and the rows n < B.per of B's groups [g0, g1).  Groups whose
// active[g] is 0 are skipped.  a, b: the sources that A and B were sliced from.
struct Out {
    double* p;
    int64_t kdiv, m_hi, m_lo, g_s, n_s;
};
int gemm(const Operand& A, const RowMajor& a, const Operand& B, const RowMajor& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream);
int gemm(const Operand& A, const PanelRows& a, const Operand& B, const RowMajor& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream);
int gemm(const Operand& A, const PackedRows& a, const Operand& B, const Columns& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream);
int gemm(const Operand& A, const RowMajor& a, const Operand& B, const Columns& b, int32_t kdim, int64_t g0,
         int64_t g1, const Out& out, const int32_t* active, int32_t* err, cudaStream_t stream);

// p[0..n) = NaN when *err is set (a device-side wait gave up).
int nan_on_error(const int32_t* err, double* p, int64_t n, cudaStream_t stream);

}  // namespace dx
}  // namespace cds
