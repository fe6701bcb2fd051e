// Persistent tcgen05 GEMM over exact integer units (sm_103a).
//
// The FP64-accurate products of the library are sums of integer products: the
// operands are planes of small integers held in BF16 (fixed-point digits or
// residues modulo small primes), and a sum of such products over a bounded K
// range is an integer below 2^24, which the tensor cores' FP32 accumulator holds
// exactly.  This kernel computes the integer planes; a following elementwise pass
// (tc_exact.cu, crt.cu) turns them into FP64.
//
// Why this shape.  On this part a tcgen05.mma with 128 output columns takes about
// as long as one with 256, so tiles are 256 columns wide; and each unit's sum has
// to be read out of tensor memory between MMAs, so the 512 columns hold two
// 256-column accumulators and the readout of one unit runs under the MMAs of the
// next.  That leaves no tensor memory for the combination of the planes, which is
// why it is a pass of its own over planes that mostly stay in L2.  An earlier form
// combined the levels in tensor memory and had room for 128 columns only: it ran
// the tensor pipe 36% of its active cycles.  W^T (H W) of 1024 x 1000 x 4096 with 7
// digits (packing included) went from 621 to 187 us, the 6-digit gradient of a
// 4096 x 1024 system from 494 to 228 us (fold included), with the same bits.
//
// One work item is one output tile of one plane.  Planes are independent, so a
// product of few tiles still fills the chip: 19 planes of residues and magnitudes (or
// 6 to 8 digit levels) of a 512 x 128 product give 76 items.  Items are ordered heaviest plane
// first and dealt out in alternating directions, CTAs (or CTA pairs) being
// persistent; the shared-memory ring and the accumulators run on across items.
//
// Roles: warp 0 streams operand tiles by TMA, warp 1 issues the MMAs, warps 2..9
// read the units out (two warps per tensor-memory lane quarter, half of the
// columns each).  With PAIR, two CTAs of a cluster compute a 256-row tile with
// tcgen05.mma.cta_group::2, each holding half of the B tile.  Every wait is
// bounded; on timeout the kernel records the error and unwinds.
#include <cuda.h>
#include <cuda_bf16.h>

#include "omm_internal.cuh"
#include "pdl.cuh"
#include "smem_optin.cuh"
#include "tc_ptx.cuh"
#include "tc_units.cuh"

namespace omm {
namespace tc {
namespace {

using namespace ptx;

constexpr int kUnitThreads = 320;
constexpr int kBox = 128 * BK * 2;   // bytes of one 128-row operand box
constexpr int kAccCols = 256;
constexpr float kMagic = 12582912.f;   // 1.5 * 2^23: adding it rounds |x| < 2^22 to an integer in the low bits

// The t-th item of CTA group `g` of `n`: rounds of n items dealt in alternating
// directions, so the groups that got the heaviest items first get the lightest next.
__device__ __forceinline__ int item_of(int t, int g, int n) { return t * n + ((t & 1) ? n - 1 - g : g); }

struct Item {
    int g, z, mi, ni;
};
__device__ __forceinline__ Item item_at(const UnitArgs &a, int idx) {
    Item it;
    it.ni = idx % a.tiles_n;
    idx /= a.tiles_n;
    it.mi = idx % a.tiles_m;
    idx /= a.tiles_m;
    it.z = idx % a.nbatch;
    it.g = idx / a.nbatch;
    return it;
}

template <bool PAIR, bool CRT>
__global__ void __launch_bounds__(kUnitThreads, 1)
    tc_unit_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                   const __grid_constant__ UnitArgs args) {
    constexpr int STAGES = PAIR ? 6 : 4;
    constexpr int STAGE_BYTES = PAIR ? 2 * kBox : 3 * kBox;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
    const int group = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int ngroups = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    const int bn = args.bn;
    const int nkb = (args.K + BK - 1) / BK;
    const int kb_chunk = args.kchunk / BK;
    const int nchunks = (nkb + kb_chunk - 1) / kb_chunk;
    const int ppu = args.ppu;

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[STAGES];    // (leading CTA) a stage's copies landed
    __shared__ __align__(8) uint64_t empty_bar[STAGES];   // the MMAs of a stage completed
    __shared__ __align__(8) uint64_t tfull_bar[2];        // a unit is complete in accumulator b
    __shared__ __align__(8) uint64_t tempty_bar[2];       // (leading CTA) accumulator b has been read
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    const uint64_t deadline = globaltimer_ns() + kWaitNs;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull_bar[b], 1);
            mbar_init(&tempty_bar[b], PAIR ? 16 : 8);
        }
        abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        if (PAIR) tmem_alloc_pair(&tmem_base, 512);
        else tmem_alloc(&tmem_base, 512);
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync_all();   // both CTAs' barriers exist before any copy signals them
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    int issued = 0;
    pdl_wait();   // the operands and the state are the work of earlier launches
    // state->done only changes between launches: every CTA of a finished solve has no items
    const bool live = args.state == nullptr || !*((volatile const int *)&args.state->done);
    const int nitems = live ? args.ngroups * args.nbatch * args.tiles_m * args.tiles_n : 0;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer: the ring runs on across units and items
        uint32_t it = 0;
        bool ok = true;
        for (int t = 0; ok; ++t) {
            const int idx = item_of(t, group, ngroups);
            if (t * ngroups >= nitems) break;
            if (idx >= nitems) continue;
            const Item w = item_at(args, idx);
            const int a_row = args.a_row0 + w.z * args.a_row_step + w.mi * (PAIR ? 256 : 128) + 128 * (int)rank;
            const int b_row = args.b_row0 + w.z * args.b_row_step + w.ni * bn + (PAIR ? bn / 2 : 0) * (int)rank;
            const int npair = args.cnt[w.g], p0 = args.first[w.g];
            for (int c = 0; c < nchunks && ok; ++c) {
                const int kb0 = c * kb_chunk, kb1 = min(nkb, kb0 + kb_chunk);
                for (int p = 0; p < npair && ok; ++p) {
                    const int pa = args.pa[p0 + p], pb = args.pb[p0 + p];
                    for (int kb = kb0; kb < kb1; ++kb, ++it) {
                        const int s = (int)(it % STAGES);
                        const uint32_t ph = (it / STAGES) & 1u;
                        if (!mbar_wait(&empty_bar[s], ph ^ 1u, deadline, &abort_flag, args.err)) { ok = false; break; }
                        uint8_t *st = smem + s * STAGE_BYTES;
                        if (PAIR) {
                            if (rank == 0) {
                                mbar_arrive_expect_tx(&full_bar[s], 4u * kBox);
                                tma_load_3d(st, &mapA, kb * BK, a_row, pa, &full_bar[s]);
                                tma_load_3d(st + kBox, &mapB, kb * BK, b_row, pb, &full_bar[s]);
                            } else {
                                const uint32_t fb = mapa_shared(smem_u32(&full_bar[s]), 0u);
                                tma_load_3d_pair(st, &mapA, kb * BK, a_row, pa, fb);
                                tma_load_3d_pair(st + kBox, &mapB, kb * BK, b_row, pb, fb);
                            }
                        } else {
                            mbar_arrive_expect_tx(&full_bar[s], (bn > 128 ? 3u : 2u) * kBox);
                            tma_load_3d(st, &mapA, kb * BK, a_row, pa, &full_bar[s]);
                            tma_load_3d(st + kBox, &mapB, kb * BK, b_row, pb, &full_bar[s]);
                            if (bn > 128) tma_load_3d(st + 2 * kBox, &mapB, kb * BK, b_row + 128, pb, &full_bar[s]);
                        }
                        issued = (int)it + 1;
                    }
                }
            }
        }
    } else if (warp == 1 && lane == 0 && rank == 0) {
        // ---------------- MMA issuer: units alternate between the two accumulators
        const uint32_t idesc = idesc_bf16(PAIR ? 256 : 128, bn);
        uint32_t it = 0, u = 0;
        bool ok = true;
        for (int t = 0; ok; ++t) {
            const int idx = item_of(t, group, ngroups);
            if (t * ngroups >= nitems) break;
            if (idx >= nitems) continue;
            const int npair = args.cnt[item_at(args, idx).g];
            for (int c = 0; c < nchunks && ok; ++c) {
                const int kb0 = c * kb_chunk, kb1 = min(nkb, kb0 + kb_chunk);
                for (int p = 0; p < npair && ok; p += ppu, ++u) {
                    const uint32_t b = u & 1u;
                    if (!mbar_wait_cluster(&tempty_bar[b], ((u >> 1) & 1u) ^ 1u, deadline, &abort_flag, args.err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t tacc = tmem + b * kAccCols;
                    const int nk = (kb1 - kb0) * min(ppu, npair - p);
                    for (int k = 0; k < nk; ++k, ++it) {
                        const int s = (int)(it % STAGES);
                        const uint32_t ph = (it / STAGES) & 1u;
                        if (!mbar_wait_cluster(&full_bar[s], ph, deadline, &abort_flag, args.err)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t st = smem_u32(smem + s * STAGE_BYTES);
                        const uint64_t da = sdesc_sw128(st), db = sdesc_sw128(st + kBox);
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            const uint32_t acc = (k != 0 || kk != 0) ? 1u : 0u;
                            if (PAIR) umma_bf16_pair(tacc, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, acc);
                            else umma_bf16(tacc, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, acc);
                        }
                        if (PAIR) umma_commit_pair_mc(&empty_bar[s], (uint16_t)0x3);
                        else umma_commit(&empty_bar[s]);
                    }
                    if (PAIR) umma_commit_pair_mc(&tfull_bar[b], (uint16_t)0x3);
                    else umma_commit(&tfull_bar[b]);
                }
            }
        }
    } else if (warp >= 2) {
        // ---------------- readout: this warp's 32 rows x half of the tile's columns
        const int q = warp & 3;
        const int half = bn >> 1;                       // a multiple of 16
        const int c_lo = (warp - 2) < 4 ? 0 : half;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c_lo;
        const uint32_t te_local = smem_u32(tempty_bar);
        const uint32_t te = PAIR ? mapa_shared(te_local, 0u) : te_local;
        // units of at most 2^22 convert by one FADD and one IADD per element (the
        // F2I conversion runs at an eighth of that rate)
        const bool small = args.small != 0;
        uint32_t acc[128];
        uint32_t u = 0;
        bool ok = true;
        for (int t = 0; ok; ++t) {
            const int idx = item_of(t, group, ngroups);
            if (t * ngroups >= nitems) break;
            if (idx >= nitems) continue;
            const Item w = item_at(args, idx);
            const int npair = args.cnt[w.g];
            const float mod = CRT ? args.mod[w.g] : 0.f, inv = CRT ? args.inv_mod[w.g] : 0.f;
            const int nunits = nchunks * ((npair + ppu - 1) / ppu);
            for (int k = 0; k < nunits; ++k, ++u) {
                const uint32_t b = u & 1u;
                const bool got = mbar_wait(&tfull_bar[b], (u >> 1) & 1u, deadline, &abort_flag, args.err);
                ok = __all_sync(0xffffffffu, got);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < 128; c0 += 16) {
                    if (c0 < half) {
                        uint32_t r0[16];
                        tmem_ld16_async(lane_base + b * kAccCols + (uint32_t)c0, r0);
                        tmem_wait_ld(r0);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float x = __uint_as_float(r0[j]);
                            if (CRT) {
                                // x - mod * rint(x / mod): exact, in [-mod/2 - 1, mod/2 + 1]
                                // (mod = inv = 0: x)
                                const float qf = fmaf(x, inv, kMagic) - kMagic;
                                float r = fmaf(-mod, qf, x);
                                if (k != 0) r += __uint_as_float(acc[c0 + j]);
                                acc[c0 + j] = __float_as_uint(r);
                            } else {
                                const uint32_t v = small ? __float_as_uint(x + kMagic) - __float_as_uint(kMagic)
                                                         : (uint32_t)__float2int_rn(x);
                                acc[c0 + j] = k != 0 ? acc[c0 + j] + v : v;
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (PAIR) mbar_arrive_remote(te + b * 8u);
                    else mbar_arrive(&tempty_bar[b]);
                }
            }
            if (!ok) break;
            const int row = w.mi * (PAIR ? 256 : 128) + 128 * (int)rank + 32 * q + lane;
            const int col0 = w.ni * bn + c_lo;
            uint32_t *o = args.out + (int64_t)w.g * args.plane + (int64_t)w.z * args.z_step + row;
            if (row < args.M) {
                if (CRT) {
#pragma unroll
                    for (int c = 0; c < 128; c += 4) {
                        if (c < half && col0 + c < args.N) {
                            uint32_t y[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float r = __uint_as_float(acc[c + j]);
                                if (mod == 0.f) r = (r >= kMagnitudeFloor || r == 0.f) ? 1.f : 0.f;
                                if (nunits > 1) r = fmaf(-mod, fmaf(r, inv, kMagic) - kMagic, r);
                                y[j] = __float_as_uint(r + kMagic);   // low byte: r mod 256
                            }
                            o[(int64_t)((col0 + c) >> 2) * args.ldp] =
                                __byte_perm(__byte_perm(y[0], y[1], 0x0040), __byte_perm(y[2], y[3], 0x0040), 0x5410);
                        }
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 128; ++c)
                        if (c < half && col0 + c < args.N) o[(int64_t)(col0 + c) * args.ldp] = acc[c];
                }
            }
        }
    }
    if (warp == 0 && lane == 0 && abort_flag) {
        // an aborted pipeline: let the issued copies land before the CTA can exit
        const uint64_t now = globaltimer_ns();
        if (rank == 0) {
            const uint64_t until = now + 200000000ull;
            for (int g = issued - STAGES < 0 ? 0 : issued - STAGES; g < issued; ++g) {
                const uint32_t addr = smem_u32(&full_bar[g % STAGES]);
                const uint32_t ph = (uint32_t)((g / STAGES) & 1);
                while (!mbar_try_wait_cluster(addr, ph) && globaltimer_ns() < until) {
                }
            }
        } else {
            while (globaltimer_ns() < now + 1000000ull) {
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync_all();   // neither CTA leaves while the pair's MMAs or copies may touch it
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(tmem, 512);
        else tmem_dealloc(tmem, 512);
    }
}

template <bool PAIR, bool CRT>
int launch_unit(const CUtensorMap &ma, const CUtensorMap &mb, const UnitArgs &a, int groups, cudaStream_t st) {
    const int smem = (PAIR ? 6 * 2 : 4 * 3) * kBox + 1024;
    static SmemOptIn opt_in;
    OMM_CUDA_TRY(opt_in(tc_unit_kernel<PAIR, CRT>));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(PAIR ? 2 * groups : groups), 1, 1);
    cfg.blockDim = dim3(kUnitThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = PAIR ? 2 : 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    OMM_CUDA_TRY(cudaLaunchKernelEx(&cfg, tc_unit_kernel<PAIR, CRT>, ma, mb, a));
    count_launch();
    return OMM_OK;
}

}  // namespace

int unit_gemm(const CUtensorMap &mapA, const CUtensorMap &mapB, const UnitArgs &args, bool crt, int kmax,
              cudaStream_t st) {
    if (args.M <= 0 || args.N <= 0 || args.K <= 0 || args.nbatch < 1 || args.ngroups < 1 ||
        args.ngroups > kUnitMaxGroups || kmax < BK)
        return OMM_ERR_ARG;
    UnitArgs a = args;
    // columns: as few tiles as 256 allows, of equal width (a multiple of 32: half a
    // tile is a multiple of the 16 columns of one tensor-memory load)
    a.tiles_n = (int)ceil_div(a.N, 256);
    a.bn = (int)ceil_div(ceil_div(a.N, a.tiles_n), 32) * 32;
    // K in chunks whose sums stay exact; where one chunk holds all of K, several
    // pairs of a group share one accumulator run (short K: within 2^22, which the
    // readout converts fastest)
    a.kchunk = kmax;
    a.ppu = 1;
    a.small = 0;
    if (a.K <= kmax) {
        const int kpad = (int)ceil_div(a.K, BK) * BK;
        a.kchunk = kpad;
        a.small = 4 * a.K <= kmax;
        a.ppu = (a.small ? kmax / 4 : kmax) / a.K;
    }
    int weight = 0, wmax = 0;
    for (int g = 0; g < a.ngroups; ++g) {
        weight += a.cnt[g];
        wmax = wmax > a.cnt[g] ? wmax : a.cnt[g];
    }
    // CTA pairs halve the operand traffic per SM; single CTAs have twice as many,
    // half as tall tiles.  The pair form is taken when it fills the chip as evenly.
    const int64_t tn = (int64_t)a.tiles_n * a.nbatch;
    const int64_t tm1 = ceil_div(a.M, 128), tm2 = ceil_div(a.M, 256);
    auto span = [&](int64_t tiles, int groups) {   // units in the longest group, roughly
        const int64_t s = ceil_div(tiles * weight, groups);
        return (double)(s > wmax ? s : wmax);
    };
    const bool pair = span(tm2 * tn, 76) <= 1.08 * span(tm1 * tn, 152);
    a.tiles_m = (int)(pair ? tm2 : tm1);
    const int64_t items = (int64_t)a.ngroups * a.tiles_m * tn;
    if (items > 2147483647) return OMM_ERR_ARG;
    const int cap = pair ? 76 : 152;
    const int groups = items < cap ? (int)items : cap;
    if (pair) return crt ? launch_unit<true, true>(mapA, mapB, a, groups, st) : launch_unit<true, false>(mapA, mapB, a, groups, st);
    return crt ? launch_unit<false, true>(mapA, mapB, a, groups, st) : launch_unit<false, false>(mapA, mapB, a, groups, st);
}

}  // namespace tc
}  // namespace omm
