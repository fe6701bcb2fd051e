// FP64 products on the BF16 tensor cores through residues (sm_103a).
//
// The Chinese remainder form of an error-free matrix product (Ozaki, Uchino &
// Imamura 2025, "Ozaki scheme II"): every K-major operand row is scaled by a power
// of two to a vector of integers F with ||F||_2 <= 2^62, so each exact inner
// product of two such rows is an integer below 2^124 in magnitude (Cauchy-Schwarz).
// It is found from its residues modulo 16 pairwise coprime numbers below 257, whose
// product P exceeds 2^125.3: one product of BF16 integers |r| <= 128 per modulus on
// the tensor cores (tc_units.cu), exact in FP32 over 1024-long pieces of K, each
// piece reduced modulo p on readout.
//
// Only the rounding of the operands to F and of the result to FP64 remain: about
// 2^-62 of ||a|| ||b|| in all, where an FP64 multiply-add chain over K leaves
// 2^-57 .. 2^-54 on the operands of the solver.  16 products at the BF16 rate
// against one at the FP64 rate (1/1500 of it) is why this is the FP64 form's
// product: digits of a fixed-point split (tc_exact.cu) would take 45 pairs for it.
// With the step's other kernels as they are, a converged FP64 solve went from 18.9 to
// 4.0 ms at m = 144, 69 to 5.5 ms at m = 512 and 758 to 21.0 ms at m = 1996; S W and W^T H'W against quad precision went from
// 3e-16 .. 1e-15 to 4e-17 .. 7e-17 (m = 141 .. 1597, H alone and with a kinetic part).
//
// Reconstruction.  With q_i = (P / p_i)^-1 mod p_i folded into one operand's
// residues, x / P = frac(sum_i y_i / p_i), y_i the residues of the product.  Two
// moduli at a time, y_i / p_i + y_j / p_j = (y_i p_j + y_j p_i) / (p_i p_j): a sum of
// 17-bit integers times 90-bit fractions in three 30-bit limbs (24 wide multiply-adds
// in place of 48), taken modulo 1 by letting the 64-bit integers wrap, times P,
// rounded once.
//
// A row with a NaN or an infinity gets the exponent kNonFinite, and every output of
// that row is a NaN.
#include <math.h>

#include "crt.cuh"
#include "fixed.cuh"
#include "fp_convert.cuh"
#include "pdl.cuh"
#include "tc_units.cuh"

namespace omm {
namespace crt {
namespace {

constexpr int kNormBits = 62;         // ||F||_2 <= 2^62
constexpr int kKmax = 1024;           // 1024 * 128 * 128 = 2^24
constexpr float kMagic = 12582912.f;  // 1.5 * 2^23

// 2^8 and odd numbers up to 253: (p + 1) / 2 <= 127 fits a signed byte even where
// the nearest-multiple rounding of the reduction lands one step off (255 would not)
struct Tables {
    int p[kModuli];
    float pf[kModuli], inv[kModuli];
    float c[2][kModuli][4];        // 2^(16 j) mod p (centred); [1]: times q_i
    int f2[kModuli / 2], f1[kModuli / 2], f0[kModuli / 2];   // floor(2^90 / (p_2i p_2i+1)) in 30-bit limbs
    unsigned long long pm;         // P / 2^62
};

constexpr int centred(int r, int p) { return 2 * r > p ? r - p : r; }

constexpr Tables make_tables() {
    Tables t{};
    const int p[kModuli] = {256, 253, 251, 247, 245, 241, 239, 233, 229, 227, 223, 219, 211, 199, 197, 193};
    unsigned __int128 P = 1;
    for (int i = 0; i < kModuli; ++i) P *= (unsigned __int128)p[i];
    t.pm = (unsigned long long)((P + ((unsigned __int128)1 << 61)) >> 62);
    for (int i = 0; i < kModuli; ++i) {
        t.p[i] = p[i];
        t.pf[i] = (float)p[i];
        t.inv[i] = 1.f / (float)p[i];
        int rest = 1;   // (P / p_i) mod p_i
        for (int j = 0; j < kModuli; ++j)
            if (j != i) rest = rest * (p[j] % p[i]) % p[i];
        int q = 1;
        while (q * rest % p[i] != 1) ++q;
        int pw = 1;
        for (int j = 0; j < 4; ++j) {
            t.c[0][i][j] = (float)centred(pw, p[i]);
            t.c[1][i][j] = (float)centred(pw * q % p[i], p[i]);
            pw = pw * (65536 % p[i]) % p[i];
        }
    }
    for (int i = 0; i < kModuli / 2; ++i) {
        // 2^90 / (p_2i p_2i+1) by long division, 30 bits at a time
        const unsigned long long pp = (unsigned long long)p[2 * i] * p[2 * i + 1];
        unsigned long long rem = 1ull << 30;
        t.f2[i] = (int)(rem / pp);
        rem = (rem % pp) << 30;
        t.f1[i] = (int)(rem / pp);
        rem = (rem % pp) << 30;
        t.f0[i] = (int)(rem / pp);
    }
    return t;
}
constexpr Tables kTables = make_tables();
__constant__ constexpr Tables kT = make_tables();

// Residues of NV values, written as BF16 to dst[i * plane + 0..NV).  F in four
// balanced 16-bit pieces f_j: sum_j f_j (2^(16 j) mod p) <= 4 * 2^15 * 2^7 = 2^24 is
// exact in FP32, and one multiply-add each finds and removes the multiple of p.
// An integer of at most 8 bits has its BF16 form in the upper half of its float.
template <bool INV, int NV>
__device__ __forceinline__ void put_residues(const int64_t (&F)[NV], __nv_bfloat16 *dst, int64_t plane, int nv) {
    float f[NV][4];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const uint64_t G = (uint64_t)F[v] + 0x8000800080008000ull;   // every piece biased by 2^15
#pragma unroll
        for (int j = 0; j < 4; ++j)
            f[v][j] = __uint_as_float(0x4B000000u | (uint32_t)((G >> (16 * j)) & 0xFFFFu)) - 8421376.f;
    }
#pragma unroll
    for (int i = 0; i < kModuli; ++i) {
        constexpr int s = INV ? 1 : 0;
        const float p = kT.pf[i], inv = kT.inv[i];
        uint32_t w[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            float t = f[v][0] * kT.c[s][i][0];
            t = fmaf(f[v][1], kT.c[s][i][1], t);
            t = fmaf(f[v][2], kT.c[s][i][2], t);
            t = fmaf(f[v][3], kT.c[s][i][3], t);
            const float qf = fmaf(t, inv, kMagic) - kMagic;
            w[v] = __float_as_uint(fmaf(-p, qf, t));
        }
        __nv_bfloat16 *d = dst + (int64_t)i * plane;
        if (NV == 4 && nv == 4) {
            uint2 o;
            o.x = __byte_perm(w[0], w[1], 0x7632);
            o.y = __byte_perm(w[2], w[NV - 1], 0x7632);
            *reinterpret_cast<uint2 *>(d) = o;
        } else if (NV == 2 && nv == 2) {
            *reinterpret_cast<uint32_t *>(d) = __byte_perm(w[0], w[1], 0x7632);
        } else {
#pragma unroll
            for (int v = 0; v < NV; ++v)
                if (v < nv) reinterpret_cast<uint16_t *>(d)[v] = (uint16_t)(w[v] >> 16);
        }
    }
}

// ------------------------------------------------------------------ packing, K along the columns' rows
// One CTA per column: largest magnitude, sum of squares, residues.  The column (at
// most 64 KB at m = 8192) is read from memory once and stays in L1 for the other
// two passes; the 16 planes written are what bounds it.
template <bool INV>
__global__ void __launch_bounds__(256) pack_cols_kernel(int64_t K, int64_t R, const double *__restrict__ X, int64_t ld,
                                                        int *e, __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
                                                        const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    __shared__ unsigned long long smax[8];
    __shared__ float ssum[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    for (int64_t r = blockIdx.x; r < R; r += gridDim.x) {
        const double *x = X + r * ld;
        const uint64_t *xb = reinterpret_cast<const uint64_t *>(x);
        unsigned long long mx = 0;
        for (int64_t k = tid; k < K; k += blockDim.x) {
            const unsigned long long a = xb[k] & 0x7FFFFFFFFFFFFFFFull;
            mx = a > mx ? a : mx;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = v > mx ? v : mx;
        }
        if (lane == 0) smax[warp] = mx;
        __syncthreads();
        for (int w = 0; w < nw; ++w) mx = smax[w] > mx ? smax[w] : mx;
        const int be = (int)(mx >> 52);
        float S = 0.f;
        if (be != 0 && be != 0x7FF)
            for (int64_t k = tid; k < K; k += blockDim.x) S += fx_square(xb[k] & 0x7FFFFFFFFFFFFFFFull, be - 1022);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
        if (lane == 0) ssum[warp] = S;
        __syncthreads();
        S = 0.f;
        for (int w = 0; w < nw; ++w) S += ssum[w];
        const int er = fx_exponent(be, S, kNormBits);
        if (tid == 0) e[r] = er;
        for (int64_t k = 4 * tid; k < K; k += 4 * blockDim.x) {
            const int nv = K - k < 4 ? (int)(K - k) : 4;
            int64_t F[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) F[v] = v < nv ? fx_round(x[k + v], er) : 0;
            put_residues<INV, 4>(F, dst + r * ldk + k, plane, nv);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ packing, K along the rows' columns
// Partial (X, S) of every row over one slice of the columns, a thread per row
// (coalesced); S follows X up as larger elements come.
__global__ void __launch_bounds__(128) row_norm_kernel(int64_t R, int64_t K, const double *__restrict__ X, int64_t ld,
                                                       float2 *part, int64_t slice, const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    const int64_t k0 = (int64_t)blockIdx.y * slice, k1 = k0 + slice < K ? k0 + slice : K;
    const uint64_t *xb = reinterpret_cast<const uint64_t *>(X) + r;
    int be = 0;
    float S = 0.f;
    for (int64_t k = k0; k < k1; k += 8) {
        uint64_t a[8];
        int top = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            a[u] = k + u < k1 ? xb[(k + u) * ld] & 0x7FFFFFFFFFFFFFFFull : 0;
            const int b = (int)(a[u] >> 52);
            top = b > top ? b : top;
        }
        if (top > be) {
            const int d = 127 - 2 * (top - be);
            S = d > 0 ? S * __uint_as_float((uint32_t)d << 23) : 0.f;
            be = top;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) S += fx_square(a[u], be - 1022);
    }
    part[(int64_t)blockIdx.y * R + r] = make_float2(__int_as_float(be), S);
}

// (X, S) pairs combined in the order of their index
__device__ __forceinline__ void norm_join(int &be, float &S, int be2, float S2) {
    const int top = be > be2 ? be : be2;
    const int d1 = 127 - 2 * (top - be), d2 = 127 - 2 * (top - be2);
    S = (d1 > 0 ? S * __uint_as_float((uint32_t)d1 << 23) : 0.f) +
        (d2 > 0 ? S2 * __uint_as_float((uint32_t)d2 << 23) : 0.f);
    be = top;
}

// 32 rows x 64 columns per CTA, turned through shared memory so that both the reads
// (along rows) and the writes (along K) are whole 128-byte lines.
template <bool INV>
__global__ void __launch_bounds__(256) pack_rows_kernel(int64_t R, int64_t K, const double *__restrict__ X, int64_t ld,
                                                        const float2 *__restrict__ part, int nslice, int *e,
                                                        __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
                                                        const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    __shared__ double tile[2][32][33];   // [k & 1][k / 2][row]: conflict-free both ways
    __shared__ float2 ns[8][32];
    __shared__ int es[32];
    const int64_t r0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 64;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = warp; i < 64; i += 8) {
        const int64_t r = r0 + lane, k = k0 + i;
        tile[i & 1][i >> 1][lane] = (r < R && k < K) ? X[r + k * ld] : 0.0;
    }
    {
        // the rows' partial norms: warp w joins slices w, w + 8, ..., warp 0 the warps' results
        float2 v[kRowSlices / 8];
#pragma unroll
        for (int q = 0; q < kRowSlices / 8; ++q)
            v[q] = (warp + 8 * q < nslice && r0 + lane < R) ? part[(int64_t)(warp + 8 * q) * R + r0 + lane]
                                                            : make_float2(0.f, 0.f);
        int be = __float_as_int(v[0].x);
        float S = v[0].y;
#pragma unroll
        for (int q = 1; q < kRowSlices / 8; ++q) norm_join(be, S, __float_as_int(v[q].x), v[q].y);
        ns[warp][lane] = make_float2(__int_as_float(be), S);
    }
    __syncthreads();
    if (warp == 0) {
        int be = __float_as_int(ns[0][lane].x);
        float S = ns[0][lane].y;
#pragma unroll
        for (int w = 1; w < 8; ++w) norm_join(be, S, __float_as_int(ns[w][lane].x), ns[w][lane].y);
        es[lane] = fx_exponent(be, S, kNormBits);
        if (blockIdx.y == 0 && r0 + lane < R) e[r0 + lane] = es[lane];
    }
    __syncthreads();
    const int64_t k = k0 + 2 * lane;
    const int nv = K - k < 2 ? (int)(K - k) : 2;
    for (int i = warp; i < 32; i += 8) {
        if (r0 + i >= R || nv <= 0) break;
        const int64_t F[2] = {fx_round(tile[0][lane][i], es[i]), fx_round(tile[1][lane][i], es[i])};
        put_residues<INV, 2>(F, dst + (r0 + i) * ldk + k, plane, nv);
    }
}

// ------------------------------------------------------------------ reconstruction
struct FoldArgs {
    int M, N, ldp;
    const uint32_t *words;
    int64_t plane, z_step;
    double alpha, beta;
    const double *Cin;
    int64_t ldcin;
    double *C;
    int64_t ldc, c_step;
    const int *eA, *eB;
    int64_t eA_step, eB_step;
    const DevState *state;
};

// A thread takes one row of four columns: 16 words of four residues, four outputs.
__global__ void __launch_bounds__(256) fold_kernel(const __grid_constant__ FoldArgs a) {
    pdl_wait();
    if (a.state != nullptr && *((volatile const int *)&a.state->done)) return;
    const int row = blockIdx.x * 32 + threadIdx.x;
    const int c4 = blockIdx.y * 8 + threadIdx.y;
    const int z = blockIdx.z;
    if (row >= a.M || 4 * c4 >= a.N) return;
    const uint32_t *w = a.words + (int64_t)z * a.z_step + (int64_t)c4 * a.ldp + row;
    uint32_t y[kModuli];
#pragma unroll
    for (int i = 0; i < kModuli; ++i) y[i] = __ldg(w + (int64_t)i * a.plane);
    const int nc = a.N - 4 * c4 < 4 ? a.N - 4 * c4 : 4;
    const double *Cin = a.Cin != nullptr ? a.Cin + row + (int64_t)(4 * c4) * a.ldcin : nullptr;
    double *C = a.C + (int64_t)z * a.c_step + row + (int64_t)(4 * c4) * a.ldc;
    double cin[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) cin[j] = (Cin != nullptr && j < nc) ? Cin[j * a.ldcin] : 0.0;
    const int ea = a.eA[(int64_t)z * a.eA_step + row];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (j >= nc) break;
        const int eb = a.eB[(int64_t)z * a.eB_step + 4 * c4 + j];
        int64_t s2 = 0, s1 = 0, s0 = 0;
        const int lsh = 24 - 8 * j;   // byte j to the top, and back with its sign
#pragma unroll
        for (int i = 0; i < kModuli / 2; ++i) {
            const int v = ((int)(y[2 * i] << lsh) >> 24) * kT.p[2 * i + 1] +
                          ((int)(y[2 * i + 1] << lsh) >> 24) * kT.p[2 * i];
            s2 += (int64_t)v * kT.f2[i];
            s1 += (int64_t)v * kT.f1[i];
            s0 += (int64_t)v * kT.f0[i];
        }
        // x / P as a signed 64-bit fraction: whole multiples of P wrap away
        const int64_t V = (int64_t)(((uint64_t)s2 << 34) + ((uint64_t)s1 << 4) + (uint64_t)(s0 >> 26));
        const uint64_t A = V < 0 ? 0ull - (uint64_t)V : (uint64_t)V;
        const uint64_t hi = __umul64hi(A, kT.pm), lo = A * kT.pm;
        const uint64_t u = ((hi << 1) | (lo >> 63)) + ((lo >> 62) & 1ull);   // |x| / 2^61
        double out;
        if (ea == kNonFinite || eb == kNonFinite) {
            out = __longlong_as_double(0x7FF8000000000000ll);
        } else {
            const int ex = ea + eb + 61;
            // normal results by integer operations; anything else through ldexp
            out = (ex > -960 && ex < 900) ? sw_u64_scaled(u, V < 0, ex) : ldexp(V < 0 ? -(double)u : (double)u, ex);
        }
        if (a.alpha != 1.0) out *= a.alpha;
        if (Cin != nullptr) out = fma(a.beta, cin[j], out);
        C[j * a.ldc] = out;
    }
}

}  // namespace

int pack_cols(int64_t K, int64_t R, const double *X, int64_t ld, int *e, __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
              bool inverse, const DevState *state, cudaStream_t st) {
    if (K <= 0 || R <= 0) return OMM_OK;
    const unsigned grid = (unsigned)(R < 65536 ? R : 65536);
    const int threads = K <= 256 ? 64 : (K <= 512 ? 128 : 256);
    if (inverse) OMM_CUDA_TRY(launch_pdl(pack_cols_kernel<true>, grid, dim3(threads), 0, st, K, R, X, ld, e, dst,
                                         ldk, plane, state));
    else OMM_CUDA_TRY(launch_pdl(pack_cols_kernel<false>, grid, dim3(threads), 0, st, K, R, X, ld, e, dst, ldk,
                                 plane, state));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

int pack_rows(int64_t R, int64_t K, const double *X, int64_t ld, int *e, float2 *part, __nv_bfloat16 *dst, int64_t ldk,
              int64_t plane, bool inverse, const DevState *state, cudaStream_t st) {
    if (K <= 0 || R <= 0) return OMM_OK;
    int64_t slice = ceil_div(ceil_div(K, kRowSlices), 8) * 8;
    const int nslice = (int)ceil_div(K, slice);
    dim3 ng((unsigned)ceil_div(R, 128), (unsigned)nslice);
    OMM_CUDA_TRY(launch_pdl(row_norm_kernel, ng, dim3(128), 0, st, R, K, X, ld, part, slice, state));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    dim3 grid((unsigned)ceil_div(R, 32), (unsigned)ceil_div(K, 64));
    if (inverse) OMM_CUDA_TRY(launch_pdl(pack_rows_kernel<true>, grid, dim3(256), 0, st, R, K, X, ld, part, nslice,
                                         e, dst, ldk, plane, state));
    else OMM_CUDA_TRY(launch_pdl(pack_rows_kernel<false>, grid, dim3(256), 0, st, R, K, X, ld, part, nslice, e, dst,
                                 ldk, plane, state));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

int gemm(const CUtensorMap &mapA, const CUtensorMap &mapB, const Args &a, int nbatch, cudaStream_t st) {
    tc::UnitArgs u{};
    u.M = a.M;
    u.N = a.N;
    u.K = a.K;
    u.nbatch = nbatch;
    u.ngroups = kModuli;
    for (int i = 0; i < kModuli; ++i) {
        u.pa[i] = u.pb[i] = u.first[i] = (uint8_t)i;
        u.cnt[i] = 1;
        u.mod[i] = kTables.pf[i];
        u.inv_mod[i] = kTables.inv[i];
    }
    u.a_row0 = a.a_row0;
    u.b_row0 = a.b_row0;
    u.a_row_step = a.a_row_step;
    u.b_row_step = a.b_row_step;
    u.out = a.words;
    u.ldp = (a.M + 3) / 4 * 4;
    u.plane = (int64_t)u.ldp * ((a.N + 3) / 4);
    u.z_step = u.plane * kModuli;
    u.state = a.state;
    u.err = a.err;
    const int rc = tc::unit_gemm(mapA, mapB, u, true, kKmax, st);
    if (rc != OMM_OK) return rc;
    FoldArgs f{};
    f.M = a.M;
    f.N = a.N;
    f.ldp = u.ldp;
    f.words = a.words;
    f.plane = u.plane;
    f.z_step = u.z_step;
    f.alpha = a.alpha;
    f.beta = a.beta;
    f.Cin = a.beta != 0.0 ? a.Cin : nullptr;
    f.ldcin = a.ldcin;
    f.C = a.C;
    f.ldc = a.ldc;
    f.c_step = a.c_step;
    f.eA = a.eA;
    f.eB = a.eB;
    f.eA_step = a.eA_step;
    f.eB_step = a.eB_step;
    f.state = a.state;
    dim3 grid((unsigned)ceil_div(a.M, 32), (unsigned)ceil_div(ceil_div(a.N, 4), 8), (unsigned)nbatch);
    OMM_CUDA_TRY(launch_pdl(fold_kernel, grid, dim3(32, 8), 0, st, f));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

}  // namespace crt
}  // namespace omm
