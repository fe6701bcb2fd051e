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
constexpr int64_t kSlabCols = 65280ll * 32;  // columns of one fold launch: 32 per block of a grid's y (at most 65535)

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

// Digits of NV values a = v 2^-e, stored side by side: F = round(v 2^(B-e)) with
// B = 6 + 7(s-1), then balanced base-128 digits F = sum_t d_t 128^(s-t), d_t in
// [-64, 64] (all but the leading one in [-64, 63]: adding 64 to each turns them into
// plain base-128 digits).  d_t then carries the weight 2^-(7t-1) of the fixed-point
// splitting.  A small integer has its BF16 form in the upper half of its float.
template <int NV>
__device__ __forceinline__ void put_digits(const double (&v)[NV], int e, int s, __nv_bfloat16 *dst, int64_t plane, int nv) {
    int64_t G[NV];
    int64_t bias = 0;
    for (int i = 0; i < s - 1; ++i) bias = bias * 128 + 64;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const uint64_t b = (uint64_t)__double_as_longlong(v[j]);
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
        G[j] = F + bias;
    }
    for (int t = s - 1; t >= 0; --t) {
        uint32_t w[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            const int d = t > 0 ? (int)((uint32_t)G[j] & 127u) - 64 : (int)G[j];
            w[j] = __float_as_uint(__uint_as_float((uint32_t)(0x4B400000 + d)) - 12582912.f);
            G[j] >>= 7;
        }
        __nv_bfloat16 *o = dst + t * plane;
        if (NV == 4 && nv == 4)
            *reinterpret_cast<uint2 *>(o) = make_uint2(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[NV - 1], 0x7632));
        else if (NV == 2 && nv == 2)
            *reinterpret_cast<uint32_t *>(o) = __byte_perm(w[0], w[1], 0x7632);
        else
#pragma unroll
            for (int j = 0; j < NV; ++j)
                if (j < nv) reinterpret_cast<uint16_t *>(o)[j] = (uint16_t)(w[j] >> 16);
    }
}

// One operand of a launch, with its share of the blocks of both kernels.
struct PackBlocks {
    PackJob j;
    int64_t R, K;            // operand rows and their length
    int nslice, tiles;       // columns in nslice slices; 32-row tiles (rows of the source)
    int64_t slice;
    int blocks_max, blocks;  // blocks of the maxima kernel, of the digits kernel
};
struct PackArgs {
    PackBlocks p[2];
    int s;
    const DevState *state;
};

// Largest biased exponent of every operand row over a slice of its columns, for
// operands whose K runs along the source's columns: a thread per row, coalesced.
__global__ void __launch_bounds__(128) row_max_kernel(const __grid_constant__ PackArgs a) {
    pdl_wait();
    if (a.state != nullptr && *((volatile const int *)&a.state->done)) return;
    const int second = (int)blockIdx.x >= a.p[0].blocks_max ? 1 : 0;
    const PackBlocks &p = a.p[second];
    const int b = (int)blockIdx.x - (second ? a.p[0].blocks_max : 0);
    const int sl = b % p.nslice;
    const int64_t r = (int64_t)(b / p.nslice) * 128 + threadIdx.x;
    if (r >= p.R) return;
    const int64_t k0 = sl * p.slice, k1 = k0 + p.slice < p.K ? k0 + p.slice : p.K;
    const uint64_t *x = reinterpret_cast<const uint64_t *>(p.j.X) + r;
    uint64_t mx = 0;
    for (int64_t k = k0; k < k1; k += 8) {
        uint64_t v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = k + u < k1 ? x[(k + u) * p.j.ld] & 0x7FFFFFFFFFFFFFFFull : 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = v[u] > mx ? v[u] : mx;
    }
    p.j.part[(int64_t)sl * p.R + r] = (int)(mx >> 52);
}

// Digits and exponents of one or two operands.  K along the source's rows: a warp per
// operand row (K <= kWarpK) or a CTA, which finds the maximum and then the digits, the
// second read from L1; else 32-row tiles of 64 columns turned through shared memory,
// with the exponents from row_max_kernel's slices.  Writes are 4 to 8 bytes a thread
// and whole lines a warp.  One launch (two with row maxima) for both operands of a
// product where there were up to eight: the recursion of the Cholesky factor runs 150
// products a solve, most of them small.
constexpr int64_t kWarpK = 1024;
__global__ void __launch_bounds__(256) digit_pack_kernel(const __grid_constant__ PackArgs a) {
    pdl_wait();
    if (a.state != nullptr && *((volatile const int *)&a.state->done)) return;
    const int second = (int)blockIdx.x >= a.p[0].blocks ? 1 : 0;
    const PackBlocks &p = a.p[second];
    const PackJob &j = p.j;
    const int64_t b = (int64_t)blockIdx.x - (second ? a.p[0].blocks : 0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ double tile[2][32][33];
    __shared__ unsigned long long smax[8];
    __shared__ int part[8][32], es[32];
    if (j.k_along_rows) {
        const bool by_warp = p.K <= kWarpK;
        const int64_t r = by_warp ? b * 8 + warp : b;
        const int at = by_warp ? lane : tid, step = by_warp ? 32 : 256;
        const double *x = j.X + r * j.ld;
        unsigned long long mx = 0;
        if (r < p.R)
            for (int64_t k = at; k < p.K; k += step) {
                const unsigned long long v = reinterpret_cast<const uint64_t *>(x)[k] & 0x7FFFFFFFFFFFFFFFull;
                mx = v > mx ? v : mx;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = v > mx ? v : mx;
        }
        if (!by_warp) {
            if (lane == 0) smax[warp] = mx;
            __syncthreads();
            for (int w = 0; w < 8; ++w) mx = smax[w] > mx ? smax[w] : mx;
        }
        if (r >= p.R) return;
        const int e = exponent_from_maxbits(mx);
        if (at == 0) j.e[r] = e;
        for (int64_t k = 4 * at; k < p.K; k += 4 * step) {
            const int nv = p.K - k < 4 ? (int)(p.K - k) : 4;
            double v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = u < nv ? x[k + u] : 0.0;
            put_digits(v, e, a.s, j.dst + r * j.ldk + k, j.plane, nv);
        }
        return;
    }
    const int64_t r0 = (b % p.tiles) * 32, k0 = (b / p.tiles) * 64;
    for (int i = warp; i < 64; i += 8) {
        const int64_t r = r0 + lane, k = k0 + i;
        tile[i & 1][i >> 1][lane] = (r < p.R && k < p.K) ? j.X[r + k * j.ld] : 0.0;
    }
    int be = 0;
    for (int sl = warp; sl < p.nslice; sl += 8) {
        const int v = r0 + lane < p.R ? j.part[(int64_t)sl * p.R + r0 + lane] : 0;
        be = v > be ? v : be;
    }
    part[warp][lane] = be;
    __syncthreads();
    if (warp == 0) {
        for (int w = 1; w < 8; ++w) be = part[w][lane] > be ? part[w][lane] : be;
        es[lane] = exponent_from_maxbits((uint64_t)be << 52);
        if (k0 == 0 && r0 + lane < p.R) j.e[r0 + lane] = es[lane];
    }
    __syncthreads();
    const int64_t k = k0 + 2 * lane;
    const int nv = p.K - k < 2 ? (int)(p.K - k) : 2;
    for (int i = warp; i < 32; i += 8) {
        if (r0 + i >= p.R || nv <= 0) break;
        const double v[2] = {tile[0][lane][i], tile[1][lane][i]};
        put_digits(v, es[i], a.s, j.dst + (r0 + i) * j.ldk + k, j.plane, nv);
    }
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

int exact_pack(const PackJob &A, const PackJob *B, int s, const DevState *state, cudaStream_t st) {
    if (s < 1 || s > kExactMaxDigits) return OMM_ERR_ARG;
    PackArgs a{};
    a.s = s;
    a.state = state;
    int64_t bmax = 0, bdig = 0;
    const PackJob *jobs[2] = {&A, B};
    for (int i = 0; i < 2; ++i) {
        if (jobs[i] == nullptr) continue;
        PackBlocks &p = a.p[i];
        p.j = *jobs[i];
        p.R = p.j.k_along_rows ? p.j.cols : p.j.rows;
        p.K = p.j.k_along_rows ? p.j.rows : p.j.cols;
        if (p.R <= 0 || p.K <= 0) continue;
        int64_t nb, nm = 0;
        if (p.j.k_along_rows) {
            nb = p.K <= kWarpK ? ceil_div(p.R, 8) : p.R;
        } else {
            p.slice = ceil_div(ceil_div(p.K, kDigitSlices), 8) * 8;
            p.nslice = (int)ceil_div(p.K, p.slice);
            nm = ceil_div(p.R, 128) * p.nslice;
            p.tiles = (int)ceil_div(p.R, 32);
            nb = p.tiles * ceil_div(p.K, 64);
        }
        bmax += nm;
        bdig += nb;
        if (bdig > 2147483647) return OMM_ERR_ARG;
        p.blocks_max = (int)nm;
        p.blocks = (int)nb;
    }
    if (bdig == 0) return OMM_OK;
    if (bmax > 0) {
        OMM_CUDA_TRY(launch_pdl(row_max_kernel, dim3((unsigned)bmax), dim3(128), 0, st, a));
        count_launch();
    }
    OMM_CUDA_TRY(launch_pdl(digit_pack_kernel, dim3((unsigned)bdig), dim3(256), 0, st, a));
    count_launch();
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
    if (slab > kSlabCols) slab = kSlabCols;
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
    return (int64_t)ndigits * (M + N) * ldk * 2 + (1 + omm::tc::kDigitSlices) * (M + N) * 4 + 2048 +
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
    int *part = eB + N;   // row maxima of an operand whose K runs along its columns
    int rc;
    // op(A) M x K: rows of op(A) are K-major operand rows; op(B) K x N: columns of op(B)
    const tc::PackJob pa{transA != 0, transA ? K : M, transA ? M : K, A, lda, eA, Ad, ldk, M * ldk, part};
    const tc::PackJob pb{transB == 0, transB ? N : K, transB ? K : N, B, ldb, eB, Bd, ldk, N * ldk,
                         part + tc::kDigitSlices * M};
    if ((rc = tc::exact_pack(pa, &pb, ndigits, nullptr, st))) return rc;
    CUtensorMap ma, mb;
    if ((rc = tc::make_digit_map(&ma, Ad, K, M, ldk, M * ldk, ndigits, 128))) return rc;
    if ((rc = tc::make_digit_map(&mb, Bd, K, N, ldk, N * ldk, ndigits, 128))) return rc;
    tc::ExactArgs a{};
    a.s = ndigits;
    a.planes = (uint32_t *)(((uintptr_t)(part + tc::kDigitSlices * (M + N)) + 255) & ~(uintptr_t)255);
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
