// FP64 products on the BF16 tensor cores through residues (sm_103a).
//
// The Chinese remainder form of an error-free matrix product (Ozaki, Uchino &
// Imamura 2025, "Ozaki scheme II"): every K-major operand row is scaled by a power
// of two to a vector of integers F with ||F||_2 <= 2^69, so each exact inner
// product of two such rows is an integer below 2^138 in magnitude (Cauchy-Schwarz).
// It is found from its residues modulo 18 pairwise coprime numbers below 257, whose
// product P exceeds 2^140: one product of BF16 integers |r| <= 128 per modulus on
// the tensor cores (tc_units.cu), exact in FP32 over 1024-long pieces of K, each
// piece reduced modulo p on readout.
//
// Only the rounding of the operands to F and of the result to FP64 remain.  In units of
// the integer product (||F|| between 2^68 and 2^69) the operands' rounding is 2^67.7 rms at
// most, sqrt(K) 2^69 at worst, the reconstruction below 2^64.  That is relative to the norms,
// where an FP64 multiply-add chain is relative to sum |a_k| |b_k|: u = 2^-53 of it from a
// single rounding, K u at worst.  The two are compared for every element.  A plane of its
// own holds the magnitudes |F| 2^-69 cut to BF16, whose product bounds sum |F_a| |F_b| 2^-138
// from below.  Where that is under 2^-16 (but not zero, for want of a common index), u sum
// |F_a| |F_b| may be below 2^69 and the fold finds the element from the FP64 operands
// themselves, as it does for rows without a fixed-point form.  Elsewhere the rms error is at
// most half of that single rounding, and the worst case below the chain's.  (Without this a
// vector of one element 1e9 and many of 1 came out against its reciprocals with 2e-11 of
// relative error, and the gradient of energies in units of 1e-18 with no digit.)
// 16 moduli (62 bits) would have it at 2^-9, which 1 to 20% of the elements of S D fall below
// at m = 2000 (22 -> 114 ms a solve); at 2^-16 none do up to m ~ 10^5 of dense columns.
//
// [SW | H'W] [H_W ; S_W] stacks two products, one with a unit of energy on its left factor
// and one on its right.  A power of two, from the exponents of H' and S, goes from one half
// of K to the other, so that the unit drops out of both rows' norms.
//
// 19 products at the BF16 rate against one at the FP64 rate (1/1500 of it) is why this is
// the FP64 form's product: digits of a fixed-point split (tc_exact.cu) would take 55 pairs
// for it.  A converged FP64 solve takes 4.4 ms at m = 144, 6.0 at m = 512 and 26.5 at m =
// 1996, where CUDA-core products took 18, 70 and 763 (16 moduli without the comparison: 10 to
// 14% less); W's error against 64 bits is the same.  Where every product is recomputed (W0 decaying
// by a factor of 20 per Angstrom at m = 2016) 17 steps take 144 ms, the CUDA-core form 252.
//
// Reconstruction.  With q_i = (P / p_i)^-1 mod p_i folded into one operand's
// residues, x / P = frac(sum_i y_i / p_i), y_i the residues of the product.  Two
// moduli at a time, y_i / p_i + y_j / p_j = (y_i p_j + y_j p_i) / (p_i p_j): a sum of
// 17-bit integers times 93-bit fractions in three 31-bit limbs (27 wide multiply-adds
// in place of 54), taken modulo 1 by letting the integers wrap, times P, rounded once.
#include <math.h>

#include "crt.cuh"
#include "fixed.cuh"
#include "fp_convert.cuh"
#include "pdl.cuh"
#include "tc_units.cuh"

namespace omm {
namespace crt {
namespace {

constexpr int kNormBits = 69;         // ||F||_2 <= 2^69
constexpr int kKmax = 1024;           // 1024 * 128 * 128 = 2^24
constexpr float kMagic = 12582912.f;  // 1.5 * 2^23

// 2^8 and odd numbers up to 253: (p + 1) / 2 <= 127 fits a signed byte even where
// the nearest-multiple rounding of the reduction lands one step off (255 would not)
constexpr int kPieces = 5;            // F in 16-bit pieces, the last of at most 2^5
struct Tables {
    int p[kModuli];
    float pf[kModuli], inv[kModuli];
    float c[2][kModuli][kPieces];  // 2^(16 j) mod p (centred); [1]: times q_i
    int f2[kModuli / 2], f1[kModuli / 2], f0[kModuli / 2];   // 2^93 / (p_2i p_2i+1), rounded, in 31-bit limbs
    unsigned long long pm;         // P / 2^77
};

constexpr int centred(int r, int p) { return 2 * r > p ? r - p : r; }

constexpr Tables make_tables() {
    Tables t{};
    const int p[kModuli] = {256, 253, 251, 247, 245, 241, 239, 233, 229, 227, 223, 219, 211, 199, 197, 193, 191, 181};
    unsigned __int128 P = 1;       // of the first 16; the last two beyond 128 bits
    for (int i = 0; i < 16; ++i) P *= (unsigned __int128)p[i];
    const unsigned __int128 last = (unsigned __int128)p[16] * p[17];
    const unsigned __int128 hi = (P >> 64) * last + (((P & 0xFFFFFFFFFFFFFFFFull) * last) >> 64);   // P / 2^64
    t.pm = (unsigned long long)((hi + ((unsigned __int128)1 << 12)) >> 13);
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
        for (int j = 0; j < kPieces; ++j) {
            t.c[0][i][j] = (float)centred(pw, p[i]);
            t.c[1][i][j] = (float)centred(pw * q % p[i], p[i]);
            pw = pw * (65536 % p[i]) % p[i];
        }
    }
    for (int i = 0; i < kModuli / 2; ++i) {
        // (2^93 + pp / 2) / pp by long division, 31 bits at a time
        const unsigned long long pp = (unsigned long long)p[2 * i] * p[2 * i + 1];
        unsigned long long rem = 1ull << 31;
        t.f2[i] = (int)(rem / pp);
        rem = (rem % pp) << 31;
        t.f1[i] = (int)(rem / pp);
        rem = ((rem % pp) << 31) + pp / 2;   // the quotient stays below 2^31: pp < 2^16, odd or not a power of two
        t.f0[i] = (int)(rem / pp);
    }
    return t;
}
constexpr Tables kTables = make_tables();
__constant__ constexpr Tables kT = make_tables();

// Residues of NV values and their magnitudes, written as BF16 to dst[i * plane + 0..NV).  F in
// balanced 16-bit pieces f_j: |sum_j f_j (2^(16 j) mod p)| <= 4 * 2^15 * 126 + 2^5 * 126 < 2^24
// (p = 256: its first piece alone counts) is exact in FP32, and one multiply-add each finds
// and removes the multiple of p.
// An integer of at most 8 bits has its BF16 form in the upper half of its float.
template <int NV>
__device__ __forceinline__ void put_plane(const uint32_t (&w)[NV], __nv_bfloat16 *d, int nv) {   // upper halves of w
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

template <bool INV, int NV>
__device__ __forceinline__ void put_planes(const Fixed (&F)[NV], const uint32_t (&mag)[NV], __nv_bfloat16 *dst,
                                           int64_t plane, int nv) {
    float f[NV][kPieces];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const uint64_t G = F[v].lo + 0x8000800080008000ull;   // every piece biased by 2^15
#pragma unroll
        for (int j = 0; j < 4; ++j)
            f[v][j] = __uint_as_float(0x4B000000u | (uint32_t)((G >> (16 * j)) & 0xFFFFu)) - 8421376.f;
        const int top = F[v].hi + (G < F[v].lo ? 1 : 0);
        f[v][4] = __uint_as_float((uint32_t)(0x4B400000 + top)) - kMagic;
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
            t = fmaf(f[v][4], kT.c[s][i][4], t);
            const float qf = fmaf(t, inv, kMagic) - kMagic;
            w[v] = __float_as_uint(fmaf(-p, qf, t));
        }
        put_plane<NV>(w, dst + (int64_t)i * plane, nv);
    }
    uint32_t w[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = mag[v] << 16;
    put_plane<NV>(w, dst + (int64_t)kModuli * plane, nv);
}

// An operand's shift of element k, and the largest of its shifts
struct Shift {
    int64_t split;
    int s, smax;
    __device__ __forceinline__ explicit Shift(const Balance &b)
        : split(b.split), s(b.p != nullptr ? b.sign * *b.p : 0), smax(s > 0 ? s : 0) {}
    __device__ __forceinline__ int at(int64_t k) const { return k >= split ? s : 0; }
};

// ------------------------------------------------------------------ packing, K along the columns' rows
// One CTA per column: largest exponent, sum of squares, planes.  The column (at
// most 64 KB at m = 8192) is read from memory once and stays in L1 for the other
// two passes; the 19 planes written are what bounds it.
template <bool INV>
__global__ void __launch_bounds__(256) pack_cols_kernel(int64_t K, int64_t R, const double *__restrict__ X, int64_t ld,
                                                        int *e, __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
                                                        const Balance bal, const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    __shared__ int smax[8];
    __shared__ float ssum[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const Shift sh(bal);
    for (int64_t r = blockIdx.x; r < R; r += gridDim.x) {
        const double *x = X + r * ld;
        const uint64_t *xb = reinterpret_cast<const uint64_t *>(x);
        int code = 0;
        for (int64_t k = tid; k < K; k += blockDim.x) code = max(code, fx_code(xb[k] & 0x7FFFFFFFFFFFFFFFull, sh.at(k)));
        code = __reduce_max_sync(0xffffffffu, code);
        if (lane == 0) smax[warp] = code;
        __syncthreads();
        for (int w = 0; w < nw; ++w) code = max(code, smax[w]);
        float S = 0.f;
        for (int64_t k = tid; k < K; k += blockDim.x) S += fx_square(xb[k] & 0x7FFFFFFFFFFFFFFFull, sh.at(k), code);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
        if (lane == 0) ssum[warp] = S;
        __syncthreads();
        S = 0.f;
        for (int w = 0; w < nw; ++w) S += ssum[w];
        const int er = fx_exponent(code, S, kNormBits, sh.smax);
        if (tid == 0) e[r] = er;
        for (int64_t k = 4 * tid; k < K; k += 4 * blockDim.x) {
            const int nv = K - k < 4 ? (int)(K - k) : 4;
            Fixed F[4];
            uint32_t mag[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const double a = v < nv ? x[k + v] : 0.0;
                F[v] = fx_round(a, sh.at(k + v), er);
                mag[v] = fx_magnitude(a, sh.at(k + v), er, kNormBits);
            }
            put_planes<INV, 4>(F, mag, dst + r * ldk + k, plane, nv);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ packing, K along the rows' columns
// S of one code in units of another
__device__ __forceinline__ float rescaled(float S, int from, int to) {
    const int d = 127 - 2 * (to - from);
    return d > 0 ? S * __uint_as_float((uint32_t)d << 23) : 0.f;
}

// (code, S) pairs combined in the order of their index
__device__ __forceinline__ void norm_join(int &code, float &S, int code2, float S2) {
    const int top = max(code, code2);
    S = rescaled(S, code, top) + rescaled(S2, code2, top);
    code = top;
}

// Partial (code, S) of every row over one slice of the columns, a thread per row
// (coalesced); S follows the code up as larger elements come.  The columns on either side
// of the balance's split are summed without a shift, which then goes to the code (with a
// shift looked up for every element the kernel took 20 us at m = 1996 in place of 10).
__global__ void __launch_bounds__(128) row_norm_kernel(int64_t R, int64_t K, const double *__restrict__ X, int64_t ld,
                                                       float2 *part, int64_t slice, const Balance bal,
                                                       const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    const Shift sh(bal);
    const int64_t k0 = (int64_t)blockIdx.y * slice, k1 = k0 + slice < K ? k0 + slice : K;
    const uint64_t *xb = reinterpret_cast<const uint64_t *>(X) + r;
    int code = 0;
    float S = 0.f;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        const int64_t ka = half == 0 ? k0 : max(k0, sh.split), kb = half == 0 ? min(k1, sh.split) : k1;
        int be = 0;
        uint64_t any = 0;
        float s = 0.f;
        for (int64_t k = ka; k < kb; k += 8) {
            uint64_t a[8];
            int top = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                a[u] = k + u < kb ? xb[(k + u) * ld] & 0x7FFFFFFFFFFFFFFFull : 0;
                any |= a[u];
                top = max(top, (int)(a[u] >> 52));
            }
            if (top > be) {
                s = rescaled(s, be, top);
                be = top;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) s += fx_square(a[u], 0, be + kCodeBias);
        }
        const int c = be == 0x7FF ? kCodeInf : (be != 0 ? be + kCodeBias + (half != 0 ? sh.s : 0) : (any != 0 ? 1 : 0));
        norm_join(code, S, c, s);
    }
    part[(int64_t)blockIdx.y * R + r] = make_float2(__int_as_float(code), S);
}

// 32 rows x 64 columns per CTA, turned through shared memory so that both the reads
// (along rows) and the writes (along K) are whole 128-byte lines.
template <bool INV>
__global__ void __launch_bounds__(256) pack_rows_kernel(int64_t R, int64_t K, const double *__restrict__ X, int64_t ld,
                                                        const float2 *__restrict__ part, int nslice, int *e,
                                                        __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
                                                        const Balance bal, const DevState *state) {
    pdl_wait();
    if (state != nullptr && *((volatile const int *)&state->done)) return;
    const Shift sh(bal);
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
        int code = __float_as_int(v[0].x);
        float S = v[0].y;
#pragma unroll
        for (int q = 1; q < kRowSlices / 8; ++q) norm_join(code, S, __float_as_int(v[q].x), v[q].y);
        ns[warp][lane] = make_float2(__int_as_float(code), S);
    }
    __syncthreads();
    if (warp == 0) {
        int code = __float_as_int(ns[0][lane].x);
        float S = ns[0][lane].y;
#pragma unroll
        for (int w = 1; w < 8; ++w) norm_join(code, S, __float_as_int(ns[w][lane].x), ns[w][lane].y);
        es[lane] = fx_exponent(code, S, kNormBits, sh.smax);
        if (blockIdx.y == 0 && r0 + lane < R) e[r0 + lane] = es[lane];
    }
    __syncthreads();
    const int64_t k = k0 + 2 * lane;
    const int nv = K - k < 2 ? (int)(K - k) : 2;
    for (int i = warp; i < 32; i += 8) {
        if (r0 + i >= R || nv <= 0) break;
        const double a = tile[0][lane][i], b = tile[1][lane][i];
        const int e0 = es[i], sa = sh.at(k), sb = sh.at(k + 1);
        const Fixed F[2] = {fx_round(a, sa, e0), fx_round(b, sb, e0)};
        const uint32_t mag[2] = {fx_magnitude(a, sa, e0, kNormBits), fx_magnitude(b, sb, e0, kNormBits)};
        put_planes<INV, 2>(F, mag, dst + (r0 + i) * ldk + k, plane, nv);
    }
}

// One CTA: mean exponents over the rows that have one
__global__ void __launch_bounds__(256) balance_kernel(int64_t m, const int *__restrict__ eH, const int *__restrict__ eS,
                                                      int *p) {
    __shared__ long long sum[8];
    __shared__ int cnt[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto mean = [&](const int *e) {
        long long s = 0;
        int c = 0;
        for (int64_t i = threadIdx.x; i < m; i += 256)
            if (e[i] != kUnscaled) {
                s += e[i];
                ++c;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        __syncthreads();
        if (lane == 0) {
            sum[warp] = s;
            cnt[warp] = c;
        }
        __syncthreads();
        s = 0;
        c = 0;
        for (int w = 0; w < 8; ++w) {
            s += sum[w];
            c += cnt[w];
        }
        return c > 0 ? (int)(s / c) : 0;
    };
    const int one = 1 - kNormBits;   // exponent of a vector of norm 1
    const int d = mean(eH) - (eS != nullptr ? mean(eS) : one);
    if (threadIdx.x == 0) *p = d < -kShiftMax ? -kShiftMax : (d > kShiftMax ? kShiftMax : d);
}

// ------------------------------------------------------------------ reconstruction
struct FoldArgs {
    int M, N, K, ldp;
    const uint32_t *words;
    int64_t plane, z_step;
    double alpha, beta;
    const double *Cin;
    int64_t ldcin;
    double *C;
    int64_t ldc, c_step;
    const int *eA, *eB;
    int64_t eA_step, eB_step;
    const double *A, *B;
    int64_t A_row, A_col, A_step, ldb, B_step;
    const DevState *state;
};

// The elements marked in `bad` (bit j: column col0 + j of the lane's row) from the FP64
// operands, all lanes of a warp together: 32 rows of four columns.  Few of them: one
// after the other, the lanes along K.  Many: a lane per row and all columns that have one
// together, so that a row's elements of A serve all four.  Both are bound by the FP64 unit (1.8
// multiply-adds per clock and SM), like the CUDA-core product.
static __device__ __noinline__ void fold_fp64(const FoldArgs &a, unsigned bad, int row, int col0, int z) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x, row0 = row - lane;
    const double *A = a.A + (int64_t)z * a.A_step, *B = a.B + (int64_t)z * a.B_step + (int64_t)col0 * a.ldb;
    const double *Cin = a.Cin != nullptr ? a.Cin + (int64_t)col0 * a.ldcin : nullptr;
    double *C = a.C + (int64_t)z * a.c_step + (int64_t)col0 * a.ldc;
    auto put = [&](int64_t r, int j, double out) {
        if (a.alpha != 1.0) out *= a.alpha;
        if (Cin != nullptr) out = fma(a.beta, Cin[r + j * a.ldcin], out);
        C[r + j * a.ldc] = out;
    };
    unsigned mask[4];
    int count = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        mask[j] = __ballot_sync(full, (bad >> j) & 1u);
        count += __popc(mask[j]);
    }
    if (count <= 32) {
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
            const double *b = B + (int64_t)j * a.ldb;
            unsigned rest = j == 0 ? mask[0] : j == 1 ? mask[1] : j == 2 ? mask[2] : mask[3];
            while (rest != 0) {
                const int r = row0 + __ffs(rest) - 1;
                rest &= rest - 1;
                const double *x = A + (int64_t)r * a.A_row;
                double s = 0.0;
#pragma unroll 4
                for (int k = lane; k < a.K; k += 32) s = fma(x[(int64_t)k * a.A_col], b[k], s);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
                if (lane == 0) put(r, j, s);
            }
        }
        return;
    }
    if (bad == 0) return;
    const double *x = A + (int64_t)row * a.A_row;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t b1 = mask[1] ? a.ldb : 0, b2 = mask[2] ? 2 * a.ldb : 0, b3 = mask[3] ? 3 * a.ldb : 0;
#pragma unroll 4
    for (int k = 0; k < a.K; ++k) {
        const double v = x[(int64_t)k * a.A_col];
        if (mask[0]) s[0] = fma(v, B[k], s[0]);
        if (mask[1]) s[1] = fma(v, B[b1 + k], s[1]);
        if (mask[2]) s[2] = fma(v, B[b2 + k], s[2]);
        if (mask[3]) s[3] = fma(v, B[b3 + k], s[3]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if ((bad >> j) & 1u) put(row, j, s[j]);
}

// A thread takes one row of four columns: 19 words of four bytes, four outputs.
__global__ void __launch_bounds__(256) fold_kernel(const __grid_constant__ FoldArgs a) {
    pdl_wait();
    if (a.state != nullptr && *((volatile const int *)&a.state->done)) return;
    const int row = blockIdx.x * 32 + threadIdx.x;
    const int c4 = blockIdx.y * 8 + threadIdx.y;
    const int z = blockIdx.z;
    if (4 * c4 >= a.N) return;   // whole warps
    unsigned bad = 0;
    if (row < a.M) {
        const uint32_t *w = a.words + (int64_t)z * a.z_step + (int64_t)c4 * a.ldp + row;
        uint32_t y[kPlanes];
#pragma unroll
        for (int i = 0; i < kPlanes; ++i) y[i] = __ldg(w + (int64_t)i * a.plane);
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
            if (((y[kModuli] >> (8 * j)) & 1u) == 0 || ea == kUnscaled || eb == kUnscaled) {
                bad |= 1u << j;
                continue;
            }
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
            // x / P as a signed 128-bit fraction: whole multiples of P wrap away
            const __int128 V = (__int128)((((unsigned __int128)(__int128)s2 << 62) + ((unsigned __int128)(__int128)s1 << 31) +
                                           (unsigned __int128)(__int128)s0) << 35);
            const unsigned __int128 A = V < 0 ? 0 - (unsigned __int128)V : (unsigned __int128)V;
            // |x| = t 2^13, then its leading 64 bits and a sticky one
            const unsigned __int128 t = (unsigned __int128)(uint64_t)(A >> 64) * kT.pm + __umul64hi((uint64_t)A, kT.pm);
            const uint64_t th = (uint64_t)(t >> 64), tl = (uint64_t)t;
            const int lz = th != 0 ? __clzll((long long)th) : 64;
            uint64_t u = lz == 64 ? tl : (lz != 0 ? th << lz | tl >> (64 - lz) : th);
            if (lz != 64 && (tl << lz) != 0) u |= 1;
            const int ex = ea + eb + 13 + 64 - lz;
            // normal results by integer operations; anything else through ldexp
            double out = (ex > -960 && ex < 900) ? sw_u64_scaled(u, V < 0, ex) : ldexp(V < 0 ? -(double)u : (double)u, ex);
            if (a.alpha != 1.0) out *= a.alpha;
            if (Cin != nullptr) out = fma(a.beta, cin[j], out);
            C[j * a.ldc] = out;
        }
    }
    if (__any_sync(0xffffffffu, bad != 0)) fold_fp64(a, bad, row, 4 * c4, z);
}

}  // namespace

int pack_cols(int64_t K, int64_t R, const double *X, int64_t ld, int *e, __nv_bfloat16 *dst, int64_t ldk, int64_t plane,
              bool inverse, Balance bal, const DevState *state, cudaStream_t st) {
    if (K <= 0 || R <= 0) return OMM_OK;
    const unsigned grid = (unsigned)(R < 65536 ? R : 65536);
    const int threads = K <= 256 ? 64 : (K <= 512 ? 128 : 256);
    if (inverse) OMM_CUDA_TRY(launch_pdl(pack_cols_kernel<true>, grid, dim3(threads), 0, st, K, R, X, ld, e, dst,
                                         ldk, plane, bal, state));
    else OMM_CUDA_TRY(launch_pdl(pack_cols_kernel<false>, grid, dim3(threads), 0, st, K, R, X, ld, e, dst, ldk,
                                 plane, bal, state));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

int pack_rows(int64_t R, int64_t K, const double *X, int64_t ld, int *e, float2 *part, __nv_bfloat16 *dst, int64_t ldk,
              int64_t plane, bool inverse, Balance bal, const DevState *state, cudaStream_t st) {
    if (K <= 0 || R <= 0) return OMM_OK;
    int64_t slice = ceil_div(ceil_div(K, kRowSlices), 8) * 8;
    const int nslice = (int)ceil_div(K, slice);
    dim3 ng((unsigned)ceil_div(R, 128), (unsigned)nslice);
    OMM_CUDA_TRY(launch_pdl(row_norm_kernel, ng, dim3(128), 0, st, R, K, X, ld, part, slice, bal, state));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    dim3 grid((unsigned)ceil_div(R, 32), (unsigned)ceil_div(K, 64));
    if (inverse) OMM_CUDA_TRY(launch_pdl(pack_rows_kernel<true>, grid, dim3(256), 0, st, R, K, X, ld, part, nslice,
                                         e, dst, ldk, plane, bal, state));
    else OMM_CUDA_TRY(launch_pdl(pack_rows_kernel<false>, grid, dim3(256), 0, st, R, K, X, ld, part, nslice, e, dst,
                                 ldk, plane, bal, state));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

int balance(int64_t m, const int *eH, const int *eS, int *p, cudaStream_t st) {
    balance_kernel<<<1, 256, 0, st>>>(m, eH, eS, p);
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
    u.ngroups = kPlanes;
    for (int i = 0; i < kPlanes; ++i) {
        u.pa[i] = u.pb[i] = u.first[i] = (uint8_t)i;
        u.cnt[i] = 1;
        u.mod[i] = i < kModuli ? kTables.pf[i] : 0.f;       // 0: the magnitudes
        u.inv_mod[i] = i < kModuli ? kTables.inv[i] : 0.f;
    }
    u.a_row0 = a.a_row0;
    u.b_row0 = a.b_row0;
    u.a_row_step = a.a_row_step;
    u.b_row_step = a.b_row_step;
    u.out = a.words;
    u.ldp = (a.M + 3) / 4 * 4;
    u.plane = (int64_t)u.ldp * ((a.N + 3) / 4);
    u.z_step = u.plane * kPlanes;
    u.state = a.state;
    u.err = a.err;
    const int rc = tc::unit_gemm(mapA, mapB, u, true, kKmax, st);
    if (rc != OMM_OK) return rc;
    FoldArgs f{};
    f.M = a.M;
    f.N = a.N;
    f.K = a.K;
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
    f.A = a.A;
    f.B = a.B;
    f.A_row = a.A_row;
    f.A_col = a.A_col;
    f.A_step = a.A_step;
    f.ldb = a.ldb;
    f.B_step = a.B_step;
    f.state = a.state;
    dim3 grid((unsigned)ceil_div(a.M, 32), (unsigned)ceil_div(ceil_div(a.N, 4), 8), (unsigned)nbatch);
    OMM_CUDA_TRY(launch_pdl(fold_kernel, grid, dim3(32, 8), 0, st, f));
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

}  // namespace crt
}  // namespace omm
