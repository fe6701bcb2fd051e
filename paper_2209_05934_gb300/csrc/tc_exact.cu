// Exact-digit BF16 tensor-core GEMM: near-FP64 products on tcgen05 (sm_103a).
//
// Error-free splitting in the manner of Ozaki, Ogita, Oishi & Rump (2012),
// applied to BF16 tensor cores as in Mukunoki et al. (2020): every K-major
// row r of an operand is scaled by 2^-e_r so its entries lie in (-1, 1), then
// cut into s fixed-point digits: the integer F = round(a 2^(6 + 7(s-1))) is
// written in balanced base 128, so a = sum_t d_t 2^-(7t-1) + O(2^-(7s)) with
// each |d_t| <= 64 (exact in BF16).
// A product of two digits is at most 2^12 in magnitude, so a sum of up to
// 4096 of them is an integer below 2^24: the tensor cores accumulate every
// digit pair (t, u) over a K chunk of <= 4096 exactly in FP32.  Pairs with
// t + u <= s + 1 are kept; pairs of one level L = t + u share the weight
// 2^-(7L-2).
//
// The GEMM (tc_units.cu) leaves one int32 plane per level; the fold below combines
// the levels of an element as an integer, converts it once and writes
// C = alpha * A B + beta * Cin.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include "fp_convert.cuh"
#include "omm_internal.cuh"
#include "pdl.cuh"
#include "tc_exact.cuh"
#include "tc_gemm.cuh"
#include "tc_units.cuh"

namespace omm {
namespace tc {
namespace {

constexpr int kChunkMax = 4096;             // 4096 * 64 * 64 = 2^24: exact FP32 integer sums
constexpr int64_t kPlaneCap = 48ll << 20;   // words of level planes one launch may fill (192 MB)

// ------------------------------------------------------------------ level fold
struct FoldArgs {
    int M, N, nlev;
    const uint32_t *planes;       // group g (level nlev + 1 - g) at g * plane, batch z at z * z_step
    int64_t plane, z_step;
    int shift[kExactMaxDigits];   // per level from the top: < 0: R <- 128 R + acc, else R += acc >> shift
    int lvl_r;                    // level whose units R counts in at the end
    double alpha, beta;
    const double *Cin;
    int64_t ldcin, cin_step;
    double *C;
    float *C32;
    int64_t ldc, c_step;
    const int *eA, *eB;
    int64_t eA_step, eB_step;
    const DevState *state;
};

// R = sum_L acc_L 2^(7 (Lr - L)) over the levels from the top, counted in units of
// level Lr: R <- 128 R + acc_L (Lr <- L) while a bound on |R| stays below 2^62; past
// that Lr stays and a later level adds acc_L 2^-7(L - Lr) rounded to an integer.
// With 7 digits and K up to 32768 every level is exact; otherwise the rounding is
// below 2^-47 of the scaled operands' unit, far inside an FP64 GEMM's error bound.
//
// Bound by the plane traffic (4 bytes per level and element, mostly from L2): a
// thread takes one row of four columns and issues its 4 NLEV loads together, which
// takes the level count at compile time (6 and 7, the solver's; NLEV = 0 takes any):
// 1024 x 1000 outputs of 7 levels from 31 to 14 us.
template <int NLEV>
__global__ void __launch_bounds__(256) level_fold_kernel(const __grid_constant__ FoldArgs a) {
    pdl_wait();
    if (a.state != nullptr && *((volatile const int *)&a.state->done)) return;
    const int row = blockIdx.x * 32 + threadIdx.x;
    const int col0 = (blockIdx.y * 8 + threadIdx.y) * 4;
    const int z = blockIdx.z;
    if (row >= a.M || col0 >= a.N) return;
    const int nc = a.N - col0 < 4 ? a.N - col0 : 4;
    const uint32_t *w = a.planes + (int64_t)z * a.z_step + (int64_t)col0 * a.M + row;
    int64_t R[4] = {0, 0, 0, 0};
    auto step = [](int64_t r, uint32_t word, int sh) {   // sh is uniform: one branch for the warp
        const int64_t acc = (int64_t)(int32_t)word;
        return sh < 0 ? r * 128 + acc : r + ((acc + ((int64_t)1 << (sh - 1))) >> sh);
    };
    if (NLEV > 0) {
        uint32_t acc[NLEV > 0 ? NLEV : 1][4];
#pragma unroll
        for (int l = 0; l < NLEV; ++l)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                acc[l][j] = j < nc ? __ldg(w + (int64_t)(NLEV - 1 - l) * a.plane + (int64_t)j * a.M) : 0u;
#pragma unroll
        for (int l = 0; l < NLEV; ++l)
#pragma unroll
            for (int j = 0; j < 4; ++j) R[j] = step(R[j], acc[l][j], a.shift[l]);
    } else {
        for (int l = 0; l < a.nlev; ++l) {
            const uint32_t *p = w + (int64_t)(a.nlev - 1 - l) * a.plane;
#pragma unroll
            for (int j = 0; j < 4; ++j) R[j] = step(R[j], j < nc ? __ldg(p + (int64_t)j * a.M) : 0u, a.shift[l]);
        }
    }
    const double *Cin = a.Cin != nullptr ? a.Cin + (int64_t)z * a.cin_step + row + (int64_t)col0 * a.ldcin : nullptr;
    double cin[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) cin[j] = (Cin != nullptr && j < nc) ? Cin[j * a.ldcin] : 0.0;
    const int e_row = a.eA[(int64_t)z * a.eA_step + row] - (7 * a.lvl_r - 2);
    const int *eB = a.eB + (int64_t)z * a.eB_step + col0;
    const int64_t o = (int64_t)z * a.c_step + row + (int64_t)col0 * a.ldc;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (j >= nc) break;
        const int e = e_row + eB[j];
        // normal-range results by integer ops; anything else (never for operands
        // within 2^+-900) through ldexp
        double out = (e > -960 && e < 900)
                         ? sw_u64_scaled(R[j] < 0 ? 0ull - (uint64_t)R[j] : (uint64_t)R[j], R[j] < 0, e)
                         : ldexp((double)R[j], e);
        if (a.alpha != 1.0) out *= a.alpha;
        if (Cin != nullptr) out = fma(a.beta, cin[j], out);
        if (a.C32 != nullptr) a.C32[o + j * a.ldc] = sw_d2f(out);
        else a.C[o + j * a.ldc] = out;
    }
}

// ------------------------------------------------------------------ digit packing
// All integer arithmetic: the FP64 unit of GB300 is far too narrow for
// per-element digit splitting.
//
// A row's exponent e makes the scaled row lie in (-1, 1): 2^e > max |a|.
// Magnitudes of non-negative doubles order like their bit patterns, so the
// row maximum is an integer max over the bits with the sign cleared.
__device__ __forceinline__ int exponent_from_maxbits(uint64_t mb) {
    const int be = (int)(mb >> 52);                 // biased exponent of max |a|
    if (be == 0) return 0;                           // zero (or subnormal) row
    int e = be - 1023 + 1;                           // 2^e > max |a| >= 2^(e-1)
    return e < -1000 ? -1000 : (e > 1000 ? 1000 : e);
}

// Digits of a = v 2^-e: F = round(v 2^(B-e)) with B = 6 + 7(s-1), then balanced
// base-128 digits from the bottom: F = sum_t d_t 128^(s-t), d_t in [-64, 64].
// d_t then carries the weight 2^-(7t-1) of the fixed-point splitting.
__device__ __forceinline__ void put_digits(double v, int e, int s, __nv_bfloat16 *dst, int64_t o, int64_t plane) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int be = (int)((b >> 52) & 0x7FF);
    int64_t F = 0;
    if (be != 0) {
        const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);   // v = mant 2^(be - 1075)
        const int shift = be - 1075 + (6 + 7 * (s - 1)) - e;
        if (shift >= 0) {
            F = (int64_t)(mant << shift);             // |F| < 2^(6 + 7(s-1)) <= 2^55
        } else if (shift > -64) {
            F = (int64_t)((mant + (1ull << (-shift - 1))) >> (-shift));
        }
        if (b >> 63) F = -F;
    }
    for (int t = s - 1; t >= 1; --t) {
        const int64_t r = ((F + 64) & 127) - 64;      // in [-64, 63]
        dst[t * plane + o] = __float2bfloat16_rn((float)(int)r);   // small integers: exact, 32-bit convert
        F = (F - r) >> 7;
    }
    dst[o] = __float2bfloat16_rn((float)(int)F);      // |F| <= 64
}

// K along the source's rows: operand row r is source column r (warp per column).
__global__ void exp_cm_kernel(int64_t K, int64_t R, const double *__restrict__ X, int64_t ld, int *e,
                              const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t *Xb = (const uint64_t *)X;
    for (int64_t r = w; r < R; r += nw) {
        // four independent maxima: four loads of each lane in flight (with one warp
        // per column the grid holds few warps, so each must keep several loads going)
        unsigned long long m4[4] = {0, 0, 0, 0};
        int64_t k = lane;
        for (; k + 96 < K; k += 128)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned long long a = Xb[k + 32 * u + r * ld] & 0x7FFFFFFFFFFFFFFFull;
                m4[u] = a > m4[u] ? a : m4[u];
            }
        for (; k < K; k += 32) {
            const unsigned long long a = Xb[k + r * ld] & 0x7FFFFFFFFFFFFFFFull;
            m4[0] = a > m4[0] ? a : m4[0];
        }
        unsigned long long mx = m4[0] > m4[1] ? m4[0] : m4[1];
        const unsigned long long m23 = m4[2] > m4[3] ? m4[2] : m4[3];
        mx = m23 > mx ? m23 : mx;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
            mx = o > mx ? o : mx;
        }
        if (lane == 0) e[r] = exponent_from_maxbits(mx);
    }
}

// Row exponents when K runs along the source's columns, split over K: each warp
// takes 32 rows (one per lane, coalesced) and a slice of the columns, and folds
// the biased exponent of its largest magnitude into be[r] with an integer
// atomic max (be zeroed first); exp_finish_kernel turns be into exponents.
__global__ void exp_t_split_kernel(int64_t R, int64_t K, const double *__restrict__ X, int64_t ld, int *be,
                                   int64_t kslice, const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
    const int64_t r = (int64_t)blockIdx.x * 32 + lx;
    const int64_t k0 = (int64_t)blockIdx.y * kslice, k1 = k0 + kslice < K ? k0 + kslice : K;
    const uint64_t *Xb = (const uint64_t *)X;
    unsigned long long mx = 0;
    if (r < R)
        for (int64_t k = k0 + ly; k < k1; k += 8) {
            const unsigned long long a = Xb[r + k * ld] & 0x7FFFFFFFFFFFFFFFull;
            mx = a > mx ? a : mx;
        }
    if (r < R && mx != 0) atomicMax(&be[r], (int)(mx >> 52));
}

__global__ void exp_finish_kernel(int64_t R, int *e, const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < R; r += (int64_t)gridDim.x * blockDim.x)
        e[r] = exponent_from_maxbits((uint64_t)e[r] << 52);
}

__global__ void digits_cm_kernel(int64_t K, int64_t R, const double *__restrict__ X, int64_t ld,
                                 const int *__restrict__ e, __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
                                 int s, const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    for (int64_t r = blockIdx.y; r < R; r += gridDim.y) {
        const int er = e[r];
        for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < K; k += (int64_t)gridDim.x * blockDim.x)
            put_digits(X[k + r * ld], er, s, dst, r * ldk + k, plane);
    }
}

__global__ void digits_t_kernel(int64_t R, int64_t K, const double *__restrict__ X, int64_t ld,
                                const int *__restrict__ e, __nv_bfloat16 *dst, int64_t ldk, int64_t plane, int s,
                                const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    __shared__ double tile[32][33];
    const int64_t tr = (int64_t)blockIdx.x * 32, tk = (int64_t)blockIdx.y * 32;
    const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
    for (int i = ly; i < 32; i += 8) {
        const int64_t r = tr + lx, k = tk + i;
        tile[i][lx] = (r < R && k < K) ? X[r + k * ld] : 0.0;
    }
    __syncthreads();
    for (int i = ly; i < 32; i += 8) {
        const int64_t r = tr + i, k = tk + lx;
        if (r < R && k < K) put_digits(tile[lx][i], e[r], s, dst, r * ldk + k, plane);
    }
}

int grid_for(int64_t work, int per_block) {
    int64_t nb = ceil_div(work, per_block);
    if (nb > 152 * 16) nb = 152 * 16;
    return (int)(nb < 1 ? 1 : nb);
}

}  // namespace

// (never decreasing in any argument and the same for (M, N) and (N, M), so that the
// workspace of a caller's largest product serves its others)
int64_t exact_plane_words(int64_t M, int64_t N, int64_t nbatch, int s) {
    const int64_t all = (int64_t)s * nbatch * M * N;
    const int64_t least = (int64_t)s * nbatch * (M > N ? M : N) * 256;   // one tile of columns
    const int64_t most = least > kPlaneCap ? least : kPlaneCap;
    return all < most ? all : most;
}

int exact_pack(bool k_along_rows, int64_t rows, int64_t cols, const double *X, int64_t ld, int *e,
               __nv_bfloat16 *dst, int64_t ldk, int64_t plane, int s, const DevState *state, cudaStream_t st) {
    if (rows <= 0 || cols <= 0) return OMM_OK;
    if (s < 1 || s > kExactMaxDigits) return OMM_ERR_ARG;
    if (k_along_rows) {   // K = rows, operand rows = cols
        OMM_CUDA_TRY(launch_pdl(exp_cm_kernel, dim3(grid_for(cols * 32, 256)), dim3(256), 0, st, rows, cols, X, ld,
                                e, state));
        count_launch();
        OMM_CUDA_TRY(cudaGetLastError());
        dim3 grid((unsigned)ceil_div(rows, 256 * 2), (unsigned)(cols < 8192 ? cols : 8192));
        OMM_CUDA_TRY(launch_pdl(digits_cm_kernel, grid, dim3(256), 0, st, rows, cols, X, ld, e, dst, ldk, plane, s,
                                state));
        count_launch();
        OMM_CUDA_TRY(cudaGetLastError());
    } else {              // K = cols, operand rows = rows
        // biased exponents by an atomic max over K slices of 256 columns, then exponents
        OMM_CUDA_TRY(cudaMemsetAsync(e, 0, (size_t)rows * sizeof(int), st));
        const int64_t kslice = 256;
        dim3 eg((unsigned)ceil_div(rows, 32), (unsigned)ceil_div(cols, kslice));
        OMM_CUDA_TRY(launch_pdl(exp_t_split_kernel, eg, dim3(256), 0, st, rows, cols, X, ld, e, kslice, state));
        count_launch();
        OMM_CUDA_TRY(cudaGetLastError());
        OMM_CUDA_TRY(launch_pdl(exp_finish_kernel, dim3(grid_for(rows, 256)), dim3(256), 0, st, rows, e, state));
        count_launch();
        OMM_CUDA_TRY(cudaGetLastError());
        dim3 grid((unsigned)ceil_div(rows, 32), (unsigned)ceil_div(cols, 32));
        OMM_CUDA_TRY(launch_pdl(digits_t_kernel, grid, dim3(256), 0, st, rows, cols, X, ld, e, dst, ldk, plane, s,
                                state));
        count_launch();
        OMM_CUDA_TRY(cudaGetLastError());
    }
    return OMM_OK;
}

int exact_gemm(const CUtensorMap &mapA, const CUtensorMap &mapB, const ExactArgs &a, int nbatch, cudaStream_t st) {
    const int s = a.s;
    if (a.M <= 0 || a.N <= 0 || a.K <= 0 || s < 1 || s > kExactMaxDigits || nbatch < 1 || a.planes == nullptr)
        return OMM_ERR_ARG;
    // groups: the level with the most pairs first
    UnitArgs u{};
    u.M = a.M;
    u.K = a.K;
    u.nbatch = nbatch;
    u.ngroups = s;
    int np = 0;
    for (int lvl = s + 1; lvl >= 2; --lvl) {
        const int g = s + 1 - lvl;
        u.first[g] = (uint8_t)np;
        u.cnt[g] = (uint8_t)(lvl - 1);
        for (int t = 1; t < lvl; ++t, ++np) {
            u.pa[np] = (uint8_t)(t - 1);
            u.pb[np] = (uint8_t)(lvl - t - 1);
        }
    }
    u.a_row0 = a.a_row0;
    u.a_row_step = a.a_row_step;
    u.b_row_step = a.b_row_step;
    u.ldp = a.M;
    u.out = a.planes;
    u.state = a.state;
    u.err = a.err;
    FoldArgs f{};
    f.M = a.M;
    f.nlev = s;
    f.planes = a.planes;
    const double nchunks = (double)ceil_div(ceil_div(a.K, 64), kChunkMax / 64);
    double bound = 0.0;   // on |R|
    for (int l = 0; l < s; ++l) {
        const int lvl = l + 2;
        const double add = (double)(lvl - 1) * nchunks * 16777216.0;   // |acc| < pairs * chunks * 2^24
        const bool grow = l == 0 || (f.shift[l - 1] < 0 && bound * 128.0 + add < 4.6e18);
        if (grow) {
            f.shift[l] = -1;
            bound = l == 0 ? add : bound * 128.0 + add;
            f.lvl_r = lvl;
        } else {
            f.shift[l] = 7 * (lvl - f.lvl_r);
            bound += add / ldexp(1.0, f.shift[l]) + 1.0;
        }
    }
    f.alpha = a.alpha;
    f.beta = a.beta;
    f.Cin = a.Cin;
    f.ldcin = a.ldcin;
    f.cin_step = a.cin_step;
    f.C = a.C;
    f.C32 = a.C32;
    f.ldc = a.ldc;
    f.c_step = a.c_step;
    f.eA = a.eA;
    f.eB = a.eB;
    f.eA_step = a.eA_step;
    f.eB_step = a.eB_step;
    f.state = a.state;
    int64_t slab = exact_plane_words(a.M, a.N, nbatch, s) / ((int64_t)s * nbatch * a.M);
    if (slab < a.N) slab = slab / 256 * 256;
    for (int64_t c0 = 0; c0 < a.N; c0 += slab) {
        const int nc = (int)(a.N - c0 < slab ? a.N - c0 : slab);
        u.N = f.N = nc;
        u.b_row0 = a.b_row0 + (int)c0;
        u.plane = f.plane = (int64_t)a.M * nc;
        u.z_step = f.z_step = u.plane * s;
        const int rc = unit_gemm(mapA, mapB, u, false, kChunkMax, st);
        if (rc != OMM_OK) return rc;
        dim3 grid((unsigned)ceil_div(a.M, 32), (unsigned)ceil_div(nc, 32), (unsigned)nbatch);
        auto fold = s == 6 ? level_fold_kernel<6> : s == 7 ? level_fold_kernel<7> : level_fold_kernel<0>;
        OMM_CUDA_TRY(launch_pdl(fold, grid, dim3(32, 8), 0, st, f));
        count_launch();
        OMM_CUDA_TRY(cudaGetLastError());
        if (f.Cin != nullptr) f.Cin += slab * a.ldcin;
        if (f.C32 != nullptr) f.C32 += slab * a.ldc;
        else f.C += slab * a.ldc;
        f.eB += slab;
    }
    return OMM_OK;
}

}  // namespace tc
}  // namespace omm

// ---------------------------------------------------------------- op-level entry
extern "C" int64_t omm_op_exact_gemm_workspace_bytes(int64_t M, int64_t N, int64_t K, int32_t ndigits) {
    if (M < 0 || N < 0 || K < 0 || ndigits < 1 || ndigits > omm::tc::kExactMaxDigits) return -1;
    const int64_t ldk = (K + 7) / 8 * 8;
    return (int64_t)ndigits * (M + N) * ldk * 2 + (M + N) * 4 + 2048 +
           4 * omm::tc::exact_plane_words(M, N, 1, ndigits);
}

extern "C" int omm_op_exact_gemm(int32_t transA, int32_t transB, int64_t M, int64_t N, int64_t K,
                                 int32_t ndigits, double alpha, const double *A, int64_t lda,
                                 const double *B, int64_t ldb, double beta, const double *Cin,
                                 int64_t ldcin, double *C, int64_t ldc, void *workspace,
                                 int64_t workspace_bytes, void *stream) {
    using namespace omm;
    if (M <= 0 || N <= 0 || K <= 0 || ndigits < 1 || ndigits > tc::kExactMaxDigits) return OMM_ERR_ARG;
    if (M > (1 << 30) || N > (1 << 30) || K > (1 << 30)) return OMM_ERR_ARG;
    if (A == nullptr || B == nullptr || C == nullptr || workspace == nullptr) return OMM_ERR_ARG;
    if (lda < (transA ? K : M) || ldb < (transB ? N : K) || ldc < M) return OMM_ERR_ARG;
    if (beta != 0.0 && (Cin == nullptr || ldcin < M)) return OMM_ERR_ARG;
    if (workspace_bytes < omm_op_exact_gemm_workspace_bytes(M, N, K, ndigits)) return OMM_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t ldk = (K + 7) / 8 * 8;
    uintptr_t base = ((uintptr_t)workspace + 255) & ~(uintptr_t)255;
    __nv_bfloat16 *Ad = (__nv_bfloat16 *)base;
    __nv_bfloat16 *Bd = Ad + (int64_t)ndigits * M * ldk;
    int *eA = (int *)(Bd + (int64_t)ndigits * N * ldk);
    int *eB = eA + M;
    int rc;
    // op(A) M x K: rows of op(A) are K-major operand rows
    if ((rc = tc::exact_pack(transA != 0, transA ? K : M, transA ? M : K, A, lda, eA, Ad, ldk, M * ldk, ndigits,
                             nullptr, st)))
        return rc;
    // op(B) K x N: columns of op(B) are K-major operand rows
    if ((rc = tc::exact_pack(transB == 0, transB ? N : K, transB ? K : N, B, ldb, eB, Bd, ldk, N * ldk, ndigits,
                             nullptr, st)))
        return rc;
    CUtensorMap ma, mb;
    if ((rc = tc::make_digit_map(&ma, Ad, K, M, ldk, M * ldk, ndigits, 128))) return rc;
    if ((rc = tc::make_digit_map(&mb, Bd, K, N, ldk, N * ldk, ndigits, 128))) return rc;
    tc::ExactArgs a{};
    a.s = ndigits;
    a.planes = (uint32_t *)(((uintptr_t)(eB + N) + 255) & ~(uintptr_t)255);
    a.M = (int)M;
    a.N = (int)N;
    a.K = (int)K;
    a.alpha = alpha;
    a.beta = beta;
    a.Cin = beta != 0.0 ? Cin : nullptr;
    a.ldcin = ldcin;
    a.C = C;
    a.ldc = ldc;
    a.eA = eA;
    a.eB = eB;
    return tc::exact_gemm(ma, mb, a, 1, st);
}
