// Cholesky-reduced variant of the dense form (section "Overview of OMM
// approaches": the generalised problem H C = S C Lambda is reduced to the
// standard one through the Cholesky factorisation of S).
//
//   S = L L^T,   Y = L^-1,   H~ = Y H' Y^T,   W~ = L^T W,   W = Y^T W~.
//
// FP64-accurate throughout; the O(m^3) work runs on the tensor cores through
// the exact-digit GEMM (row-scaled base-128 digits, exact integer-valued FP32
// partial sums, FP64 combination), because the FP64 CUDA-core rate of this part
// is a small fraction of the tensor rate.
//
// L and Y come from one recursive factor-and-invert on halves: with
// S = [A11 A21^T; A21 A22],
//   L11, Y11 <- recursion on A11;  L21 = A21 Y11^T;  A22 -= L21 L21^T;
//   L22, Y22 <- recursion on A22;  Y21 = -Y22 (L21 Y11),
// so every GEMM at the top has K = m/2.  The 64 x 64 leaves are factored and
// inverted by one CTA in shared memory.  Inverting the diagonal blocks adds an
// error of order cond(L) eps, immaterial for the well-conditioned overlaps of
// localised basis sets.  The triangular products skip the zero triangle by
// chunking K.  A non-positive pivot sets state->status = OMM_ERR_NOT_SPD.
#include <math.h>

#include "chol.cuh"
#include "fp_convert.cuh"
#include "omm_internal.cuh"
#include "pdl.cuh"
#include "smem_optin.cuh"

namespace omm {
namespace chol {
namespace {

constexpr int kLeaf = 64;       // leaf size of the recursion
constexpr int kLeafWarps = 16;  // warps that own rows; two more compute the columns of L and the rows of Y
constexpr int kLeafThreads = 32 * (kLeafWarps + 2);
constexpr int kLeafRows = kLeaf / kLeafWarps;
constexpr int kRowBlock = 512;  // row / column blocks of the triangular products
constexpr int kLeafSmem = (kLeaf * kLeaf + kLeaf * (kLeaf + 1)) * (int)sizeof(double);

// Cholesky factor and inverse of the s x s diagonal block at (n0, n0), s <= 64:
// lower triangles of A and Y get L_kk and L_kk^-1, their strict upper triangles
// inside the block are zeroed.
//
// One CTA and a chain of 64 pivots; 88,000 multiply-adds at the FP64 rate of one SM
// are 26 us.  Factor and inverse run in one sweep, both in their outer-product form:
// with column q of L and row q of Y known, every element (i, j), i > q, takes one
// multiply-add, a(i, j) -= l(i, q) l(j, q) where j > q and sum(i, j) += l(i, q) y(q, j)
// where j <= q, so a row stays at work on all its columns until q = i.  Sixteen
// warps own rows w, w + 16, ... in registers, lanes along the columns (four warps
// a scheduler: what follows a multiply-add waits 64 cycles and more for it).  One warp is a
// column ahead: it takes column q + 1 as the owners left it before step q, adds
// step q, and has the next pivot's root, reciprocal and scaled column ready when the
// owners are done with step q.  One warp finishes row q of Y meanwhile, so the sums
// of Y run one step behind.  One barrier a step.  The roots in integers: in FP64
// they are 20 dependent instructions that queue with the owners' for the FP64 unit.
// The sum of y(i, j) is held in four interleaved slices (q - j) mod 4, added in
// order at the end; the register of a slice is the one of q mod 4, which the unrolled
// loop knows (slice g of column j is in register (g + j) mod 4).
// 140 us when factor and inverse were two sweeps over shared memory with three
// and two barriers a step; 94 us with eight owner warps that also finished the rows of
// Y; 71 us now, the FP64 unit busy for 68 % of it.  The same results to the last bit.
__global__ void __launch_bounds__(kLeafThreads, 1) chol_leaf_kernel(double *A, double *Y, int64_t m, int64_t n0, int s,
                                                                 DevState *state) {
    pdl_wait();
    extern __shared__ double sm[];
    double(*lc)[kLeaf] = (double(*)[kLeaf])sm;                              // lc[q]: column q of L
    double(*yr)[kLeaf + 1] = (double(*)[kLeaf + 1])(sm + kLeaf * kLeaf);    // yr[q]: row q of Y
    __shared__ double col[2][kLeaf];   // column q + 2 after step q
    __shared__ double rdiag[kLeaf];    // 1 / l(q, q)
    __shared__ double slice[2][4][kLeaf];   // sums of row q + 1 of Y after step q - 1
    const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) - 2;
    const double *Ab = A + n0 + n0 * m;
    auto load = [&](int r, int c) {    // beyond the block: the identity
        return (r < s && c < s) ? (c <= r ? Ab[r + c * m] : 0.0) : (r == c ? 1.0 : 0.0);
    };
    bool bad = false;
    double l[2];                   // the newest column of L (rows lane and lane + 32), of its warp
    auto pivot = [&](int q, const double (&b)[2]) {   // column q of L from its final values b
        double d = __shfl_sync(0xffffffffu, q < 32 ? b[0] : b[1], q & 31);
        if (!(d > 0.0)) {
            bad = bad || q < s;
            d = 1.0;
        }
        double root, r;
        sw_sqrt_rcp(d, root, r);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = lane + 32 * h;
            l[h] = row > q ? b[h] * r : (row == q ? root : 0.0);
            lc[q][row] = l[h];
        }
        if (lane == 0) rdiag[q] = r;
    };
    double acc[kLeafRows][2][4];   // a(i, j) in slot 3 until column j is done, then the slices
    double y[2] = {0.0, 0.0};      // the newest row of Y, of its warp
    if (warp == -2) {
        const double b0[2] = {load(lane, 0), load(lane + 32, 0)};
        pivot(0, b0);
    } else if (warp >= 0) {
#pragma unroll
        for (int k = 0; k < kLeafRows; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = warp + kLeafWarps * k;
#pragma unroll
                for (int u = 0; u < 3; ++u) acc[k][h][u] = 0.0;
                acc[k][h][3] = load(i, lane + 32 * h);
                if (h == 0 && lane == 1) col[1][i] = acc[k][h][3];
            }
    }
    __syncthreads();
#pragma unroll 1
    for (int q0 = 0; q0 < s; q0 += 4) {   // steps past s work on the identity's columns
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + u;
            constexpr int kSlot[4] = {3, 0, 1, 2};   // (q - 1) mod 4
            if (warp == -2) {
                if (q + 1 < kLeaf) {
                    const double piv = __shfl_sync(0xffffffffu, q + 1 < 32 ? l[0] : l[1], (q + 1) & 31);
                    const double b1[2] = {fma(-l[0], piv, col[(q + 1) & 1][lane]),
                                          fma(-l[1], piv, col[(q + 1) & 1][lane + 32])};
                    pivot(q + 1, b1);
                }
            } else if (warp == -1) {   // row q of Y: its last step, the sum of its slices
                const double r = rdiag[q];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = lane + 32 * h;
                    double v[4];   // slice g is in register (g + j) mod 4
#pragma unroll
                    for (int p = 0; p < 4; ++p) v[p] = j < q ? slice[q & 1][p][j] : 0.0;
                    if (j < q) v[kSlot[u]] = fma(lc[q > 0 ? q - 1 : 0][q], y[h], v[kSlot[u]]);
                    const bool r1 = (j & 1) != 0, r2 = (j & 2) != 0;
                    const double t0 = r1 ? v[1] : v[0], t1 = r1 ? v[2] : v[1], t2 = r1 ? v[3] : v[2],
                                 t3 = r1 ? v[0] : v[3];
                    const double tot = (r2 ? t2 : t0) + (r2 ? t3 : t1) + (r2 ? t0 : t2) + (r2 ? t1 : t3);
                    y[h] = j < q ? -tot * r : (j == q ? r : 0.0);
                    yr[q][j] = y[h];
                }
            } else {
                // a lane beyond column q takes step q of the factor, one before it step q - 1 of the inverse
                double v[2], sc[kLeafRows][2];
                bool fac[2], inv[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = lane + 32 * h;
                    fac[h] = j > q;
                    inv[h] = j < q;
                    v[h] = fac[h] ? -lc[q][j] : (inv[h] ? yr[q - 1][j] : 0.0);
                    const double *src = (inv[h] ? lc[q - 1] : lc[q]) + warp;
#pragma unroll
                    for (int k = 0; k < kLeafRows; ++k) sc[k][h] = src[kLeafWarps * k];
                }
#pragma unroll
                for (int k = 0; k < kLeafRows; ++k) {
                    const int i = warp + kLeafWarps * k;
                    if (i <= q) continue;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && kLeafWarps * k < 32) continue;   // rows 0 .. 31 end before column 32
                        double &a = acc[k][h][3], &sum = acc[k][h][kSlot[u]];
                        double t = fac[h] ? a : sum;
                        asm volatile("" : "+d"(t));   // one multiply-add, not one for each case
                        t = fma(sc[k][h], v[h], t);
                        if (lane + 32 * h == q + 2) col[q & 1][i] = t;
                        if (inv[h]) sum = t;
                        if (fac[h]) a = t;
                        if (lane + 32 * h == q) a = 0.0;
                        // settle the selects here: carried on unresolved over the unrolled steps they spill
                        asm volatile("" : "+d"(acc[k][h][3]), "+d"(acc[k][h][kSlot[u] % 3]));
                    }
                    if (i == q + 1) {
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int p = 0; p < 4; ++p)
                                if (h == 0 || kLeafWarps * k >= 32) slice[i & 1][p][lane + 32 * h] = acc[k][h][p];
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int e = threadIdx.x; e < s * kLeaf; e += kLeafThreads) {
        const int r = e % kLeaf, c = e / kLeaf;
        if (r >= s) continue;
        A[(n0 + r) + (n0 + c) * m] = lc[c][r];
        Y[(n0 + r) + (n0 + c) * m] = yr[r][c];
    }
    if (bad && lane == 0) state->status = OMM_ERR_NOT_SPD;
}

// Zero the strict upper triangle (the factor is read as a lower triangle).
__global__ void zero_upper_kernel(double *A, int64_t lda, int64_t m) {
    for (int64_t j = blockIdx.y; j < m; j += gridDim.y)
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < j; i += (int64_t)gridDim.x * blockDim.x)
            A[i + j * lda] = 0.0;
}

// a <- (a + a^T) / 2 in place; the CTA for tile pair (bx, by), bx >= by,
// rewrites both tiles
__global__ void symmetrize_kernel(double *a, int64_t m) {
    if (blockIdx.x < blockIdx.y) return;
    __shared__ double t1[32][33], t2[32][33];
    const int64_t i0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;
    const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
    for (int r = ly; r < 32; r += 8) {
        t1[r][lx] = (i0 + lx < m && j0 + r < m) ? a[(i0 + lx) + (j0 + r) * m] : 0.0;   // (i0 + lx, j0 + r)
        t2[r][lx] = (j0 + lx < m && i0 + r < m) ? a[(j0 + lx) + (i0 + r) * m] : 0.0;   // (j0 + lx, i0 + r)
    }
    __syncthreads();
    for (int r = ly; r < 32; r += 8) {
        if (i0 + lx < m && j0 + r < m) a[(i0 + lx) + (j0 + r) * m] = 0.5 * (t1[r][lx] + t2[lx][r]);
        if (j0 + lx < m && i0 + r < m) a[(j0 + lx) + (i0 + r) * m] = 0.5 * (t2[r][lx] + t1[lx][r]);
    }
}

__global__ void identity_kernel(double *a, int64_t m) {
    for (int64_t j = blockIdx.y; j < m; j += gridDim.y)
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
            a[i + j * m] = (i == j) ? 1.0 : 0.0;
}

// M = S + T / tau, elementwise (the division as written, not a reciprocal product)
__global__ void spd_sum_kernel(const double *__restrict__ S, const double *__restrict__ T, double tau, double *M,
                               int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        M[i] = S[i] + T[i] / tau;
}

int blocks(int64_t n, int per) {
    int64_t b = ceil_div(n, per);
    if (b > 152 * 8) b = 152 * 8;
    return (int)(b < 1 ? 1 : b);
}

int xmm(bool tA, bool tB, int64_t M, int64_t N, int64_t K, double alpha, const double *A, int64_t lda,
        const double *B, int64_t ldb, double beta, double *C, int64_t ldc, const Work &w, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return OMM_OK;
    return omm_op_exact_gemm(tA, tB, M, N, K, w.s, alpha, A, lda, B, ldb, beta, beta != 0.0 ? C : nullptr, ldc, C,
                             ldc, w.ws, w.bytes, st);
}

int64_t xbytes(int64_t M, int64_t N, int64_t K, int s) { return omm_op_exact_gemm_workspace_bytes(M, N, K, s); }

// split of a node of size s: the first half rounded up to a multiple of the leaf
int64_t split(int64_t s) { return ceil_div(ceil_div(s, 2), kLeaf) * kLeaf; }

int chol_inv(double *A, double *Y, int64_t m, int64_t n0, int64_t s, const Work &w, DevState *state,
             cudaStream_t st) {
    if (s <= kLeaf) {
        OMM_CUDA_TRY(launch_pdl(chol_leaf_kernel, dim3(1), dim3(kLeafThreads), kLeafSmem, st, A, Y, m, n0, (int)s,
                                state));
        count_launch();
        OMM_CUDA_TRY(cudaGetLastError());
        return OMM_OK;
    }
    const int64_t h = split(s), r = s - h;
    int rc = chol_inv(A, Y, m, n0, h, w, state, st);
    if (rc != OMM_OK) return rc;
    double *A21 = A + (n0 + h) + n0 * m;
    double *A22 = A + (n0 + h) + (n0 + h) * m;
    const double *Y11 = Y + n0 + n0 * m;
    double *Y21 = Y + (n0 + h) + n0 * m;
    const double *Y22 = Y + (n0 + h) + (n0 + h) * m;
    // L21 = A21 Y11^T (in place: operands are packed before the GEMM runs)
    if ((rc = xmm(false, true, r, h, h, 1.0, A21, m, Y11, m, 0.0, A21, m, w, st))) return rc;
    // A22 -= L21 L21^T
    if ((rc = xmm(false, true, r, r, h, -1.0, A21, m, A21, m, 1.0, A22, m, w, st))) return rc;
    if ((rc = chol_inv(A, Y, m, n0 + h, r, w, state, st))) return rc;
    // Y21 = -Y22 (L21 Y11), the inner product parked in Y21
    if ((rc = xmm(false, false, r, h, h, 1.0, A21, m, Y11, m, 0.0, Y21, m, w, st))) return rc;
    return xmm(false, false, r, h, r, -1.0, Y22, m, Y21, m, 0.0, Y21, m, w, st);
}

}  // namespace

int64_t work_bytes(int64_t m, int64_t n, int s) {
    int64_t b = xbytes(kRowBlock < m ? kRowBlock : m, m, m, s);               // triangular products
    const int64_t h = split(m), r = m - h;
    if (m > kLeaf) {
        // top node of the recursion (the largest): (r, h, h), (r, r, h), (r, h, r)
        const int64_t t0 = xbytes(r, h, h, s), t1 = xbytes(r, r, h, s), t2 = xbytes(r, h, r, s);
        b = b > t0 ? b : t0;
        b = b > t1 ? b : t1;
        b = b > t2 ? b : t2;
    }
    const int64_t t3 = xbytes(m, n, kChunkK < m ? kChunkK : m, s);             // W transforms
    return b > t3 ? b : t3;
}

int64_t linv_elems(int64_t m) { return m * m; }

int cholesky(double *A, int64_t m, const Work &w, DevState *state, cudaStream_t st) {
    static SmemOptIn opt_in;
    OMM_CUDA_TRY(opt_in(chol_leaf_kernel));
    OMM_CUDA_TRY(cudaMemsetAsync(w.Linv, 0, (size_t)(m * m) * sizeof(double), st));
    int rc = chol_inv(A, w.Linv, m, 0, m, w, state, st);
    if (rc != OMM_OK) return rc;
    dim3 g((unsigned)blocks(m, 256), (unsigned)(m < 4096 ? m : 4096));
    zero_upper_kernel<<<g, 256, 0, st>>>(A, m, m);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

// Wt = T^T W for a lower-triangular T (L, or Y), in K chunks of rows of T, last
// chunk first: rows [kc, kc+kw) of T touch output rows [0, kc+kw) only, and the
// first chunk taken (the last rows) covers every output row.
int lt_times(const double *T, int64_t m, const double *W, double *Wt, int64_t n, const Work &w, cudaStream_t st) {
    const int64_t nchunk = ceil_div(m, kChunkK);
    for (int64_t c = nchunk - 1; c >= 0; --c) {
        const int64_t kc = c * kChunkK;
        const int64_t kw = m - kc < kChunkK ? m - kc : kChunkK;
        const int rc = xmm(true, false, kc + kw, n, kw, 1.0, T + kc, m, W + kc, m, c == nchunk - 1 ? 0.0 : 1.0, Wt, m,
                           w, st);
        if (rc != OMM_OK) return rc;
    }
    return OMM_OK;
}

int factor(const double *S, double *L, int64_t m, const Work &w, DevState *state, cudaStream_t st) {
    OMM_CUDA_TRY(cudaMemcpyAsync(L, S, m * m * sizeof(double), cudaMemcpyDeviceToDevice, st));
    return cholesky(L, m, w, state, st);
}

int transform(double *Hs, double *T, int64_t m, const Work &w, cudaStream_t st) {
    const double *Y = w.Linv;
    int rc;
    // T = Y H': rows [r0, r0 + rr) of Y have nonzeros in columns < r0 + rr only
    for (int64_t r0 = 0; r0 < m; r0 += kRowBlock) {
        const int64_t rr = m - r0 < kRowBlock ? m - r0 : kRowBlock;
        if ((rc = xmm(false, false, rr, m, r0 + rr, 1.0, Y + r0, m, Hs, m, 0.0, T + r0, m, w, st))) return rc;
    }
    // H~ = T Y^T: columns [c0, c0 + cc) of Y^T have nonzeros in rows < c0 + cc only
    for (int64_t c0 = 0; c0 < m; c0 += kRowBlock) {
        const int64_t cc = m - c0 < kRowBlock ? m - c0 : kRowBlock;
        if ((rc = xmm(false, true, m, cc, c0 + cc, 1.0, T, m, Y + c0, m, 0.0, Hs + c0 * m, m, w, st))) return rc;
    }
    dim3 g((unsigned)ceil_div(m, 32), (unsigned)ceil_div(m, 32));
    symmetrize_kernel<<<g, 256, 0, st>>>(Hs, m);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    dim3 gi((unsigned)blocks(m, 256), (unsigned)(m < 4096 ? m : 4096));
    identity_kernel<<<gi, 256, 0, st>>>(T, m);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

int precon(const double *S, const double *T, double tau, double *P, int64_t m, const Work &w, DevState *state,
           cudaStream_t st) {
    spd_sum_kernel<<<blocks(m * m, 256), 256, 0, st>>>(S, T, tau, P, m * m);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    int rc = cholesky(P, m, w, state, st);
    if (rc != OMM_OK) return rc;
    // P = Y^T Y by row blocks: rows [r0, r0 + rr) of P take columns [r0, r0 + rr)
    // of Y, which are zero above row r0, so the K range is [r0, m)
    const double *Y = w.Linv;
    for (int64_t r0 = 0; r0 < m; r0 += kRowBlock) {
        const int64_t rr = m - r0 < kRowBlock ? m - r0 : kRowBlock;
        if ((rc = xmm(true, false, rr, m, m - r0, 1.0, Y + r0 + r0 * m, m, Y + r0, m, 0.0, P + r0, m, w, st)))
            return rc;
    }
    dim3 g((unsigned)ceil_div(m, 32), (unsigned)ceil_div(m, 32));
    symmetrize_kernel<<<g, 256, 0, st>>>(P, m);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

}  // namespace chol
}  // namespace omm
