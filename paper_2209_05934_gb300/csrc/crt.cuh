// FP64 products through residue planes: host-side interface inside the library.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "omm_internal.cuh"

namespace omm {
namespace crt {

constexpr int kModuli = 18;
constexpr int kPlanes = kModuli + 1;   // residues and magnitudes
constexpr int kRowSlices = 32;   // partial row norms per operand row (pack_rows)

// C_z = alpha A_z B_z + beta Cin_z from packed operands (see crt.cu); column-major.
struct Args {
    int M, N, K;
    int a_row0, b_row0, a_row_step, b_row_step;
    double alpha, beta;
    const double *Cin;
    int64_t ldcin;
    double *C;
    int64_t ldc, c_step;
    const int *eA, *eB;          // exponents of the operand rows
    int64_t eA_step, eB_step;
    // the operands themselves, for the products that the planes cannot hold as accurately as
    // FP64: A_z(i, k) = A[z A_step + i A_row + k A_col], B_z(k, j) = B[z B_step + k + j ldb]
    const double *A, *B;
    int64_t A_row, A_col, A_step, ldb, B_step;
    uint32_t *words;             // planes of the product: words_of(M, N) * nbatch words
    const DevState *state;
    int *err;
};

inline int64_t words_of(int64_t M, int64_t N) { return (int64_t)kPlanes * ((N + 3) / 4) * ((M + 3) / 4 * 4); }

// A power of two (its exponent on the device) taken into the elements k >= split of an
// operand's rows, times sign: +1 in one operand of a product and -1 in the other.
struct Balance {
    const int *p = nullptr;
    int64_t split = 0;
    int sign = 0;
};

// Operand row r = column r of the column-major K x R matrix X: planes
// dst[i * plane + r * ldk + k] and exponents e[r].  inverse: the residues carry the
// reconstruction factors (exactly one operand of a product does).
int pack_cols(int64_t K, int64_t R, const double *X, int64_t ld, int *e, __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
              bool inverse, Balance bal, const DevState *state, cudaStream_t st);
// Operand row r = row r of the column-major R x K matrix X; part: kRowSlices * R float2
int pack_rows(int64_t R, int64_t K, const double *X, int64_t ld, int *e, float2 *part, __nv_bfloat16 *dst, int64_t ldk,
              int64_t plane, bool inverse, Balance bal, const DevState *state, cudaStream_t st);
// p = the mean exponent of the m packed rows of H' less that of S's (eS = nullptr: S = I)
int balance(int64_t m, const int *eH, const int *eS, int *p, cudaStream_t st);
int gemm(const CUtensorMap &mapA, const CUtensorMap &mapB, const Args &a, int nbatch, cudaStream_t st);

}  // namespace crt
}  // namespace omm
