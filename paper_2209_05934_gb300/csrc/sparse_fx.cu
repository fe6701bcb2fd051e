// FP64-accurate block products of the linear-scaling form in integers (sm_103a).
//
// This part retires about 1.8 FP64 multiply-adds per clock and SM; a 32 x 32 -> 64-bit
// integer multiply-add runs at 30.  So the gathers of the FP64 form (products,
// contractions, gradient) multiply fixed-point operands: every scalar row of the left
// and column of the right operand is scaled by a power of two to integers F with
// ||F||_2 <= 2^57 and held as two limbs, F = hi 2^26 + lo (|hi| < 2^31, |lo| <= 2^25),
// and an inner product is
//     hh 2^52 + cr 2^26,  hh = sum hi hi',  cr = sum (hi lo' + lo hi'),
// three wide multiply-adds a term.  By Cauchy-Schwarz |hh| stays below 2^63 whatever the
// length, and |cr| <= 2^57 sqrt(n), so cr is folded into hh every 4096 terms.  What is
// left out, sum lo lo' (2^48 sqrt(n) for uncorrelated low parts), lies below the
// operands' own rounding, 2^56 of 2^114 in all, about 2^-57 of ||a|| ||b||; an FP64
// chain leaves 2^-56 .. 2^-54 there.
//
// With the arithmetic no longer the limit, the latency of the gathers and the L1's
// return bandwidth are: lanes compute every output that shares their loaded rows, and
// the triples of a block are dealt over several lane groups (integer sums can be taken
// in any order).
// The scales cost three short passes over an operand (largest exponent, sum of
// squares, conversion); both reductions are integer atomics, so their order does not
// matter and results repeat bit for bit.  The sum of a block element's column is
// collected in fixed point for that reason.
//
// A step of 512 atoms (R_C = 6 A): products 209 -> 97 us, contraction 509 -> 210,
// gradient 327 -> 163, and about 60 us of conversions.
//
// Screening (omm_options.screen_eps) keeps the FP64 gathers of sparse.cu, which skip
// single block products; so do the mixed form's handles, whose FP32 first phase turns a
// start that differs in the last bit into another trajectory (4e-6 in W after 24 steps
// of 1728 atoms).
#include <math.h>

#include "fixed.cuh"
#include "fp_convert.cuh"
#include "omm_internal.cuh"
#include "sparse.cuh"

namespace omm {
namespace sp {
namespace {

constexpr int NT = 256;
constexpr int kBits = 57;            // ||F||_2 <= 2^57
constexpr int kLimb = 26;
constexpr int kFold = 512;           // block triples (8 terms each) between folds of cr
constexpr float kSqUnit = 68719476736.f;   // 2^36: fixed point of the sums of squares

__device__ __forceinline__ bool fx_done(const DevState *s) { return s != nullptr && *((volatile const int *)&s->done); }

// exponent of vector g of an operand from its collected statistics
__device__ __forceinline__ int stat_exponent(const FxStat &s, int64_t g) {
    return fx_exponent(s.mx[g], (float)s.sq[g] * (1.f / kSqUnit), kBits);
}

// ------------------------------------------------------------------ operand conversion
// Largest biased exponent of every vector (PASS 0) and its sum of squares (PASS 1): a
// thread takes one row or column of one block (at most 8 values, loaded together).
template <int PASS>
__global__ void __launch_bounds__(NT) fx_stat_kernel(const __grid_constant__ FxJobs jobs, const DevState *state) {
    if (fx_done(state)) return;
    const FxJob &j = jobs.j[blockIdx.y];
    const int lg = j.by_row ? j.lrows : j.lcols, len = 1 << (j.by_row ? j.lcols : j.lrows);
    const int step = j.by_row ? 1 : 1 << j.lcols;
    const uint64_t *src = reinterpret_cast<const uint64_t *>(j.src);
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < j.nblk << lg; i += (int64_t)gridDim.x * NT) {
        const int64_t b = i >> lg;
        const int v = (int)i & ((1 << lg) - 1);
        const uint64_t *p = src + b * j.stride + (j.by_row ? v << j.lcols : v);
        uint64_t a[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = k < len ? p[k * step] & 0x7FFFFFFFFFFFFFFFull : 0;
        const int64_t g = ((int64_t)j.idx[b] << lg) + v;
        if (PASS == 0) {
            uint64_t top = a[0];
#pragma unroll
            for (int k = 1; k < 8; ++k) top = a[k] > top ? a[k] : top;
            const int be = (int)(top >> 52);
            if (be > j.stat.mx[g]) atomicMax(&j.stat.mx[g], be);
        } else {
            const int be = j.stat.mx[g];
            if (be == 0 || be == 0x7FF) continue;
            float S = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) S += fx_square(a[k], be - 1022);
            atomicAdd(&j.stat.sq[g], (unsigned long long)(S * kSqUnit));
        }
    }
}

__global__ void __launch_bounds__(NT) fx_convert_kernel(const __grid_constant__ FxJobs jobs, const DevState *state) {
    if (fx_done(state)) return;
    const FxJob &j = jobs.j[blockIdx.y];
    const int lb = j.lrows + j.lcols, lg = j.by_row ? j.lrows : j.lcols;
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < j.nblk << lb; i += (int64_t)gridDim.x * NT) {
        const int64_t b = i >> lb;
        const int e = (int)i & ((1 << lb) - 1), v = j.by_row ? e >> j.lcols : e & ((1 << j.lcols) - 1);
        const int64_t F = fx_round(j.src[b * j.stride + e], stat_exponent(j.stat, ((int64_t)j.idx[b] << lg) + v));
        const int64_t hi = (F + (1ll << (kLimb - 1))) >> kLimb;
        j.dst[b * j.stride + e] = make_int2((int)hi, (int)(F - (hi << kLimb)));
    }
}

// ------------------------------------------------------------------ arithmetic
struct Acc {
    int64_t hh, cr;
};
__device__ __forceinline__ void mad(Acc &s, int ah, int al, int bh, int bl) {
    s.hh += (int64_t)ah * bh;
    s.cr += (int64_t)ah * bl;
    s.cr += (int64_t)al * bh;
}
__device__ __forceinline__ void fold(Acc &s) {
    const int64_t q = (s.cr + (1ll << (kLimb - 1))) >> kLimb;
    s.hh += q;
    s.cr -= q << kLimb;
}
// R 2^(2 kLimb + e): the inner product whose folded high sum is R
__device__ __forceinline__ double fx_value(int64_t R, int ea, int eb) {
    if (ea == kNonFinite || eb == kNonFinite) return __longlong_as_double(0x7FF8000000000000ll);
    const int e = ea + eb + 2 * kLimb;
    return (e > -960 && e < 900) ? sw_u64_scaled(R < 0 ? 0ull - (uint64_t)R : (uint64_t)R, R < 0, e)
                                 : ldexp((double)R, e);
}
__device__ __forceinline__ int4 ldi4(const int2 *p) { return __ldg(reinterpret_cast<const int4 *>(p)); }

// sums over lanes whose numbers differ in the bits of `mask` (integers: any order)
template <int N>
__device__ __forceinline__ void lane_sum(int64_t (&R)[N], int first, int last) {
#pragma unroll
    for (int off = first; off <= last; off <<= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) R[i] += __shfl_xor_sync(0xffffffffu, R[i], off);
}

// ------------------------------------------------------------------ products
// Half a warp per output block: lane (part, r) computes row r of both H'D and SD, both
// columns, over every second block triple (part), from one row of H' and of S and the
// whole D block: 8 bytes from the L1 per multiply-add (a lane per matrix read 12).
__global__ void __launch_bounds__(NT) fx_products_kernel(int64_t nnzHW, const int64_t *__restrict__ Prp,
                                                         const int32_t *__restrict__ Ph,
                                                         const int32_t *__restrict__ Pw,
                                                         const int32_t *__restrict__ HWrow,
                                                         const int32_t *__restrict__ HWcol,
                                                         const int2 *__restrict__ HS, const int2 *__restrict__ D,
                                                         FxStat sH, FxStat sS, FxStat sD, double *HD, double *SD,
                                                         const DevState *state) {
    if (fx_done(state)) return;
    const int lane = threadIdx.x & 31, r = lane & 7, part = (lane >> 3) & 1;
    const int64_t nwarps = ((int64_t)gridDim.x * NT) >> 5;
    for (int64_t ob = (((int64_t)blockIdx.x * NT + threadIdx.x) >> 5) * 2; ob < nnzHW; ob += nwarps * 2) {
        const int64_t o = ob + (lane >> 4);
        const bool valid = o < nnzHW;
        Acc s[4] = {};
        const int64_t t1 = valid ? Prp[o + 1] : 0;
        for (int64_t tc = valid ? Prp[o] : 0; tc < t1; tc += kFold) {
            const int64_t te = tc + kFold < t1 ? tc + kFold : t1;
            for (int64_t t = tc + part; t < te; t += 2) {
                const int2 *A = HS + (int64_t)Ph[t] * 128 + r * 8;
                const int2 *B = D + (int64_t)Pw[t] * 16;
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    const int4 h = ldi4(A + k), w = ldi4(A + 64 + k), b0 = ldi4(B + 2 * k), b1 = ldi4(B + 2 * k + 2);
                    mad(s[0], h.x, h.y, b0.x, b0.y);
                    mad(s[1], h.x, h.y, b0.z, b0.w);
                    mad(s[2], w.x, w.y, b0.x, b0.y);
                    mad(s[3], w.x, w.y, b0.z, b0.w);
                    mad(s[0], h.z, h.w, b1.x, b1.y);
                    mad(s[1], h.z, h.w, b1.z, b1.w);
                    mad(s[2], w.z, w.w, b1.x, b1.y);
                    mad(s[3], w.z, w.w, b1.z, b1.w);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) fold(s[i]);
        }
        int64_t R[4] = {s[0].hh, s[1].hh, s[2].hh, s[3].hh};
        lane_sum(R, 8, 8);
        if (!valid) continue;
        // part 0 writes H'D, part 1 SD
        const int ea = stat_exponent(part ? sS : sH, (int64_t)HWrow[o] * 8 + r);
        const int64_t c = (int64_t)HWcol[o] * 2;
        *reinterpret_cast<double2 *>((part ? SD : HD) + o * 16 + r * 2) =
            make_double2(fx_value(part ? R[2] : R[0], ea, stat_exponent(sD, c)),
                         fx_value(part ? R[3] : R[1], ea, stat_exponent(sD, c + 1)));
    }
}

// ------------------------------------------------------------------ contractions
// Half a warp per P_N block: lane (side, k) holds for basis row k the eight outputs of
// its left operand (W, side 0: X and Y; D, side 1: h2 and s2).  Where only X and Y are
// wanted (lower-triangle blocks with Ntr given; XY: every block), both sides multiply W
// and take every second block triple.
template <bool XY>
__global__ void __launch_bounds__(NT, 3) fx_contract_kernel(int64_t nnzN, const int64_t *__restrict__ Crp,
                                                            const int32_t *__restrict__ Ca,
                                                            const int32_t *__restrict__ Cb,
                                                            const int32_t *__restrict__ Nrow,
                                                            const int32_t *__restrict__ Ncol,
                                                            const int2 *__restrict__ W, const int2 *__restrict__ D,
                                                            const int2 *__restrict__ HD, const int2 *__restrict__ SD,
                                                            FxStat sW, FxStat sD, FxStat sHD, FxStat sSD, double *X,
                                                            double *Y, double *h2, double *s2,
                                                            const int32_t *__restrict__ Ntr, const DevState *state) {
    if (fx_done(state)) return;
    const int lane = threadIdx.x & 31, k = lane & 7, side = (lane >> 3) & 1;
    const int64_t nwarps = ((int64_t)gridDim.x * NT) >> 5;
    for (int64_t qb = (((int64_t)blockIdx.x * NT + threadIdx.x) >> 5) * 2; qb < nnzN; qb += nwarps * 2) {
        const int64_t q = qb + (lane >> 4);
        const bool valid = q < nnzN;
        const bool both = XY || (valid && Ntr != nullptr && Ntr[q] < q);   // both sides on W
        const int2 *L = (both || side == 0 ? W : D) + 2 * k, *RH = HD + 2 * k, *RS = SD + 2 * k;
        const int64_t step = both ? 2 : 1;
        Acc s[8] = {};
        const int64_t t1 = valid ? Crp[q + 1] : 0;
        for (int64_t tc = valid ? Crp[q] : 0; tc < t1; tc += 8 * kFold) {   // one term a triple and lane
            const int64_t te = tc + 8 * kFold < t1 ? tc + 8 * kFold : t1;
#pragma unroll 2
            for (int64_t t = tc + (both ? side : 0); t < te; t += step) {
                const int64_t ib = (int64_t)Cb[t] * 16;
                const int4 w = ldi4(L + (int64_t)Ca[t] * 16), hd = ldi4(RH + ib), sd = ldi4(RS + ib);
                mad(s[0], w.x, w.y, hd.x, hd.y);
                mad(s[1], w.x, w.y, hd.z, hd.w);
                mad(s[2], w.z, w.w, hd.x, hd.y);
                mad(s[3], w.z, w.w, hd.z, hd.w);
                mad(s[4], w.x, w.y, sd.x, sd.y);
                mad(s[5], w.x, w.y, sd.z, sd.w);
                mad(s[6], w.z, w.w, sd.x, sd.y);
                mad(s[7], w.z, w.w, sd.z, sd.w);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) fold(s[i]);
        }
        // sums over the eight basis rows by halving: bit 2 of the lane keeps SD's or HD's
        // outputs, bit 1 a row of them; the two lanes of bit 0 then hold half sums each
        int64_t R[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) R[i] = s[i].hh;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int bit = 4 >> h, n = 4 >> h;
            const bool up = (k & bit) != 0;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const int64_t give = up ? R[i] : R[i + n], keep = up ? R[i + n] : R[i];
                R[i] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
            }
        }
        int64_t P[2] = {R[0], R[1]};
        lane_sum(P, 1, 1);
        // both sides worked on the same outputs: add them up
        const int64_t o0 = __shfl_xor_sync(0xffffffffu, P[0], 8), o1 = __shfl_xor_sync(0xffffffffu, P[1], 8);
        if (both) {
            P[0] += o0;
            P[1] += o1;
        }
        if (valid && (k & 1) == 0 && !(both && side)) {
            const int a = (k >> 1) & 1, sr = k >> 2;   // row, and HD (0) or SD (1)
            const int64_t J = (int64_t)Nrow[q] * 2 + a, J2 = (int64_t)Ncol[q] * 2;
            const int ea = stat_exponent(side == 0 ? sW : sD, J);
            const FxStat &sR = sr ? sSD : sHD;
            double *o = side == 0 ? (sr ? Y : X) : (sr ? s2 : h2);
            *reinterpret_cast<double2 *>(o + q * 4 + a * 2) =
                make_double2(fx_value(P[0], ea, stat_exponent(sR, J2)), fx_value(P[1], ea, stat_exponent(sR, J2 + 1)));
        }
    }
}

// ------------------------------------------------------------------ gradient
// G_o = 2 (2 H'W_o - sum (SW_(I,K) h0_(K,J) + H'W_(I,K) s0_(K,J))): a warp per block,
// lane (part, r) both columns of row r over every fourth triple; the two sums have
// scales of their own
__global__ void __launch_bounds__(NT) fx_gradient_kernel(int64_t nnzW, const int64_t *__restrict__ Grp,
                                                         const int32_t *__restrict__ Gb,
                                                         const int32_t *__restrict__ Gq,
                                                         const int32_t *__restrict__ WtoHW,
                                                         const int32_t *__restrict__ HWrow,
                                                         const int32_t *__restrict__ HWcol,
                                                         const int2 *__restrict__ HWx, const int2 *__restrict__ SWx,
                                                         const int2 *__restrict__ h0, const int2 *__restrict__ s0,
                                                         FxStat sHW, FxStat sSW, FxStat sh0, FxStat ss0,
                                                         const double *__restrict__ HW, double *G,
                                                         const DevState *state) {
    if (fx_done(state)) return;
    const int lane = threadIdx.x & 31, r = lane & 7, part = lane >> 3;
    const int64_t nwarps = ((int64_t)gridDim.x * NT) >> 5;
    for (int64_t o = ((int64_t)blockIdx.x * NT + threadIdx.x) >> 5; o < nnzW; o += nwarps) {
        Acc s[4] = {};
        const int64_t t1 = Grp[o + 1];
        for (int64_t tc = Grp[o]; tc < t1; tc += 4 * kFold) {   // two terms a triple
            const int64_t te = tc + 4 * kFold < t1 ? tc + 4 * kFold : t1;
#pragma unroll 2
            for (int64_t t = tc + part; t < te; t += 4) {
                const int64_t gb = (int64_t)Gb[t] * 16 + r * 2, gq = (int64_t)Gq[t] * 4;
                const int4 sw = ldi4(SWx + gb), hw = ldi4(HWx + gb);
                const int4 h = ldi4(h0 + gq), hn = ldi4(h0 + gq + 2), v = ldi4(s0 + gq), vn = ldi4(s0 + gq + 2);
                mad(s[0], sw.x, sw.y, h.x, h.y);
                mad(s[1], sw.x, sw.y, h.z, h.w);
                mad(s[0], sw.z, sw.w, hn.x, hn.y);
                mad(s[1], sw.z, sw.w, hn.z, hn.w);
                mad(s[2], hw.x, hw.y, v.x, v.y);
                mad(s[3], hw.x, hw.y, v.z, v.w);
                mad(s[2], hw.z, hw.w, vn.x, vn.y);
                mad(s[3], hw.z, hw.w, vn.z, vn.w);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) fold(s[i]);
        }
        int64_t R[4] = {s[0].hh, s[1].hh, s[2].hh, s[3].hh};
        lane_sum(R, 8, 16);
        if (part >= 2) continue;   // parts 0 and 1 finish one column each
        const int64_t p = WtoHW[o], row = (int64_t)HWrow[p] * 8 + r, col = (int64_t)HWcol[p] * 2 + part;
        const double g = fx_value(part ? R[1] : R[0], stat_exponent(sSW, row), stat_exponent(sh0, col)) +
                         fx_value(part ? R[3] : R[2], stat_exponent(sHW, row), stat_exponent(ss0, col));
        G[o * 16 + r * 2 + part] = 2.0 * (2.0 * HW[p * 16 + r * 2 + part] - g);
    }
}

int blocks_for(int64_t work, int per) {
    int64_t nb = ceil_div(work, per);
    if (nb > 152 * 16) nb = 152 * 16;
    return (int)(nb < 1 ? 1 : nb);
}

// statistics and conversion of the listed operands; [zero, zero + bytes) are their
// statistics
int convert(const FxJobs &jobs, void *zero, size_t bytes, const DevState *state, cudaStream_t st) {
    OMM_CUDA_TRY(cudaMemsetAsync(zero, 0, bytes, st));
    int64_t units = 0, elems = 0;
    for (int i = 0; i < jobs.n; ++i) {
        const FxJob &j = jobs.j[i];
        const int64_t u = j.nblk << (j.by_row ? j.lrows : j.lcols), e = j.nblk << (j.lrows + j.lcols);
        units = u > units ? u : units;
        elems = e > elems ? e : elems;
    }
    const dim3 gu((unsigned)blocks_for(units, NT), (unsigned)jobs.n), ge((unsigned)blocks_for(elems, NT), (unsigned)jobs.n);
    fx_stat_kernel<0><<<gu, NT, 0, st>>>(jobs, state);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    fx_stat_kernel<1><<<gu, NT, 0, st>>>(jobs, state);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    fx_convert_kernel<<<ge, NT, 0, st>>>(jobs, state);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

}  // namespace

int fx_alloc(const Host &hs, Dev &d) {
    Fx &f = d.fx;
    // row and column of every block
    std::vector<int32_t> hrow((size_t)d.nnzH), hwrow((size_t)d.nnzHW), nrow((size_t)d.nnzN);
    for (int64_t I = 0; I < d.nbr; ++I) {
        for (int64_t b = hs.Hrp[I]; b < hs.Hrp[I + 1]; ++b) hrow[b] = (int32_t)I;
        for (int64_t b = hs.HWrp[I]; b < hs.HWrp[I + 1]; ++b) hwrow[b] = (int32_t)I;
    }
    for (int64_t J = 0; J < d.nbc; ++J)
        for (int64_t b = hs.Nrp[J]; b < hs.Nrp[J + 1]; ++b) nrow[b] = (int32_t)J;
    const int64_t m = d.nbr * d.bm, n = d.nbc * d.bn, mn = m > n ? m : n;
    const int64_t bb = (int64_t)d.bm * d.bm, bw = (int64_t)d.bm * d.bn, bq = (int64_t)d.bn * d.bn;
    int64_t bytes = 0;
    auto take = [&](int64_t size) {
        const int64_t at = bytes;
        bytes += (size + 255) / 256 * 256;
        return at;
    };
    const int64_t oHrow = take(4 * d.nnzH), oWcol = take(4 * d.nnzW), oHWrow = take(4 * d.nnzHW),
                  oHWcol = take(4 * d.nnzHW), oNrow = take(4 * d.nnzN), oNcol = take(4 * d.nnzN);
    const int64_t oHS = take(8 * 2 * d.nnzH * bb), oW = take(8 * d.nnzW * bw), oD = take(8 * d.nnzW * bw),
                  oA = take(8 * d.nnzHW * bw), oB = take(8 * d.nnzHW * bw), oh = take(8 * d.nnzN * bq),
                  os = take(8 * d.nnzN * bq);
    // statistics, 12 bytes a vector: [H | S], [W | D], [A | B | h0 | s0]
    const int64_t oSt = take(12 * (2 * m + 2 * n + 2 * mn + 2 * n) + 16 * 8);
    if (cudaMalloc((void **)&f.base, (size_t)bytes) != cudaSuccess) {
        f = Fx{};
        return OMM_ERR_NOMEM;
    }
    f.Hrow = (int32_t *)(f.base + oHrow);
    f.Wcol = (int32_t *)(f.base + oWcol);
    f.HWrow = (int32_t *)(f.base + oHWrow);
    f.HWcol = (int32_t *)(f.base + oHWcol);
    f.Nrow = (int32_t *)(f.base + oNrow);
    f.Ncol = (int32_t *)(f.base + oNcol);
    f.HS = (int2 *)(f.base + oHS);
    f.W = (int2 *)(f.base + oW);
    f.D = (int2 *)(f.base + oD);
    f.A = (int2 *)(f.base + oA);
    f.B = (int2 *)(f.base + oB);
    f.h0 = (int2 *)(f.base + oh);
    f.s0 = (int2 *)(f.base + os);
    char *p = f.base + oSt;
    auto stat = [&](FxStat &s, int64_t count) {   // 8-byte sums, then 4-byte exponents (padded to 8)
        s.sq = (unsigned long long *)p;
        p += 8 * count;
        s.mx = (int *)p;
        p += (4 * count + 7) / 8 * 8;
    };
    f.z0 = p;
    stat(f.sH, m);
    stat(f.sS, m);
    f.z1 = p;
    stat(f.sW, n);
    stat(f.sD, n);
    f.z2 = p;
    stat(f.sA, mn);
    stat(f.sB, mn);
    stat(f.sh0, n);
    stat(f.ss0, n);
    f.z3 = p;
    auto up = [](int32_t *dst, const std::vector<int32_t> &v) {
        return v.empty() || cudaMemcpy(dst, v.data(), v.size() * 4, cudaMemcpyHostToDevice) == cudaSuccess;
    };
    if (!up(f.Hrow, hrow) || !up(f.Wcol, hs.Wcol) || !up(f.HWrow, hwrow) || !up(f.HWcol, hs.HWcol) ||
        !up(f.Nrow, nrow) || !up(f.Ncol, hs.Ncol))
        return OMM_ERR_CUDA;
    return OMM_OK;
}

int fx_set_HS(Dev &d, cudaStream_t st) {
    Fx &f = d.fx;
    FxJobs jobs{};
    // H' and S blocks lie side by side: a stride of two blocks
    jobs.j[jobs.n++] = FxJob{d.HS, f.HS, d.nnzH, f.Hrow, 3, 3, 1, 128, f.sH};
    jobs.j[jobs.n++] = FxJob{d.HS + 64, f.HS + 64, d.nnzH, f.Hrow, 3, 3, 1, 128, f.sS};
    return convert(jobs, f.z0, (size_t)(f.z1 - f.z0), nullptr, st);
}

int fx_products(Dev &d, const double *Din, double *HDo, double *SDo, const DevState *state, cudaStream_t st) {
    Fx &f = d.fx;
    FxJobs jobs{};
    const bool isW = Din == d.W;   // the start multiplies W; a step's D also needs W for its contraction
    jobs.j[jobs.n++] = FxJob{d.W, f.W, d.nnzW, f.Wcol, 3, 1, 0, 16, f.sW};
    if (!isW) jobs.j[jobs.n++] = FxJob{Din, f.D, d.nnzW, f.Wcol, 3, 1, 0, 16, f.sD};
    const int rc = convert(jobs, f.z1, (size_t)(f.z2 - f.z1), state, st);
    if (rc != OMM_OK) return rc;
    fx_products_kernel<<<blocks_for(d.nnzHW * 16, NT), NT, 0, st>>>(d.nnzHW, d.Prp, d.Ph, d.Pw, f.HWrow, f.HWcol, f.HS,
                                                                    isW ? f.W : f.D, f.sH, f.sS, isW ? f.sW : f.sD, HDo,
                                                                    SDo, state);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

int fx_contract(Dev &d, const double *Wl, const double *Dl, const double *HDr, const double *SDr, double *Xo, double *Yo,
                double *h2o, double *s2o, const int32_t *Ntr, const DevState *state, cudaStream_t st) {
    Fx &f = d.fx;
    FxJobs jobs{};
    jobs.j[jobs.n++] = FxJob{HDr, f.A, d.nnzHW, f.HWcol, 3, 1, 0, 16, f.sA};
    jobs.j[jobs.n++] = FxJob{SDr, f.B, d.nnzHW, f.HWcol, 3, 1, 0, 16, f.sB};
    const int rc = convert(jobs, f.z2, (size_t)(f.z3 - f.z2), state, st);
    if (rc != OMM_OK) return rc;
    const int grid = blocks_for(d.nnzN * 16, NT);
    if (Wl == Dl)   // W^T of both: X and Y are all there is
        fx_contract_kernel<true><<<grid, NT, 0, st>>>(d.nnzN, d.Crp, d.Ca, d.Cb, f.Nrow, f.Ncol, f.W, f.W, f.A, f.B, f.sW,
                                                      f.sW, f.sA, f.sB, Xo, Yo, nullptr, nullptr, nullptr, state);
    else
        fx_contract_kernel<false><<<grid, NT, 0, st>>>(d.nnzN, d.Crp, d.Ca, d.Cb, f.Nrow, f.Ncol, f.W, f.D, f.A, f.B,
                                                       f.sW, f.sD, f.sA, f.sB, Xo, Yo, h2o, s2o, Ntr, state);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

int fx_gradient(Dev &d, const DevState *state, cudaStream_t st) {
    Fx &f = d.fx;
    FxJobs jobs{};
    jobs.j[jobs.n++] = FxJob{d.HW, f.A, d.nnzHW, f.HWrow, 3, 1, 1, 16, f.sA};
    jobs.j[jobs.n++] = FxJob{d.SW, f.B, d.nnzHW, f.HWrow, 3, 1, 1, 16, f.sB};
    jobs.j[jobs.n++] = FxJob{d.h0, f.h0, d.nnzN, f.Ncol, 1, 1, 0, 4, f.sh0};
    jobs.j[jobs.n++] = FxJob{d.s0, f.s0, d.nnzN, f.Ncol, 1, 1, 0, 4, f.ss0};
    const int rc = convert(jobs, f.z2, (size_t)(f.z3 - f.z2), state, st);
    if (rc != OMM_OK) return rc;
    fx_gradient_kernel<<<blocks_for(d.nnzW * 32, NT), NT, 0, st>>>(d.nnzW, d.Grp, d.Gb, d.Gq, d.WtoHW, f.HWrow, f.HWcol,
                                                                  f.A, f.B, f.h0, f.s0, f.sA, f.sB, f.sh0, f.ss0, d.HW,
                                                                  d.G, state);
    count_launch();
    OMM_CUDA_TRY(cudaGetLastError());
    return OMM_OK;
}

}  // namespace sp
}  // namespace omm
