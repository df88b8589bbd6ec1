// FP64 matrix products on the tensor cores by exact slices (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, 2012): D[n][m] = sum_k A[m][k]
// B[n][k] from operands stored as eight signed base-256 digits per element.
//
// A row is scaled by 2^ex > max|x| of the row, q = round(x 2^(62-ex)) (exact
// for every entry within 2^-9 of the row's largest, 2^-63 of it otherwise),
// and q is cut into eight digits d_0 (most significant, |d_0| <= 64) .. d_7
// in [-128, 127], each exact in BF16.  The 36 digit products with s + t <= 7
// are kept; the dropped ones are below 2^-60 of both rows' scales.
#pragma once

#include "common.cuh"

namespace cds {
namespace dx {

constexpr int kRowsA = 128;   // rows per tile of an A operand (MMA M)
constexpr int kRowsB = 64;    // rows per tile of a B operand
constexpr int kStepK = 16;    // columns per k-step (one MMA k)
constexpr int kDigits = 8;

// One sliced operand: tiles of R rows, each [k-step][digit][R rows x 32
// bytes], already in the order and 32-byte swizzle the MMA reads, so a k-step
// of a tile is one contiguous bulk copy.  Rows come in groups of `per` that
// start on a tile boundary (per = all rows for a plain matrix).
struct Operand {
    uint8_t* img;
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
    o.ex = c.take<int32_t>(rows);
    return o;
}

// Row sources: element k of row r of group g.
struct RowMajor {         // x[(g gs + r) ld + k]
    const double* x;
    int64_t gs, ld;
    __device__ __forceinline__ double get(int64_t g, int64_t r, int k) const {
        return x[(g * gs + r) * ld + k];
    }
};
struct PackedRows {       // rows (K, nu): A^K[nu][k] of the packed symmetric vectors
    const double* L;
    int64_t npair;
    int32_t K0, N;
    __device__ __forceinline__ double get(int64_t, int64_t r, int k) const {
        const int K = (int)(r / N), nu = (int)(r % N);
        const int hi = max(k, nu), lo = min(k, nu);
        return L[(int64_t)(K0 + K) * npair + (int64_t)hi * (hi + 1) / 2 + lo];
    }
};
struct Columns {          // row j: C[k][col(j)], col(j) = j < nocc ? j : orb[j - nocc]
    const double* C;
    const int32_t* orb;
    int32_t nmo, nocc, first;
    __device__ __forceinline__ double get(int64_t, int64_t r, int k) const {
        int q = (int)r + first;
        if (orb && q >= nocc) q = orb[q - nocc];
        if (q < 0 || q >= nmo) return __longlong_as_double(0x7ff8000000000000LL);
        return C[(int64_t)k * nmo + q];
    }
};

// Slice an operand (R = kRowsA or kRowsB).  *flag is set (never cleared) when
// a row holds a non-finite entry or a magnitude outside 2^+-400: the products
// of such a call are then left to the plain FP64 kernel (run_gemm's fallback).
int slice_rows(const RowMajor& src, const Operand& o, int R, int32_t kdim, int32_t* flag,
               cudaStream_t stream);
int slice_packed(const PackedRows& src, const Operand& o, int R, int32_t kdim, int32_t* flag,
                 cudaStream_t stream);
int slice_columns(const Columns& src, const Operand& o, int R, int32_t kdim, int32_t* flag,
                  cudaStream_t stream);

// out[(m / kdiv) m_hi + (m % kdiv) m_lo + (g - g0) g_s + n n_s] for the rows m of
// A (one group) and the rows n < B.per of B's groups [g0, g1).  Groups whose
// active[g] is 0 are skipped.  Returns at once on the device when *flag is set.
struct Out {
    double* p;
    int64_t kdiv, m_hi, m_lo, g_s, n_s;
};
int gemm(const Operand& A, const Operand& B, int64_t g0, int64_t g1, const Out& out,
         const int32_t* active, const int32_t* flag, int32_t* err, cudaStream_t stream);

// p[0..n) = NaN when *err is set (a device-side wait gave up).
int nan_on_error(const int32_t* err, double* p, int64_t n, cudaStream_t stream);

}  // namespace dx
}  // namespace cds
