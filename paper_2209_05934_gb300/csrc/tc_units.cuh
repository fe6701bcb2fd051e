// Persistent tcgen05 GEMM over exact integer units: host-side interface inside the library.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "omm_internal.cuh"

namespace omm {
namespace tc {

constexpr int kUnitMaxGroups = 19;   // planes of one launch
constexpr int kUnitMaxPairs = 36;

// One launch computes `ngroups` integer planes of an M x N product (z-batched).
// Plane g is the exact integer sum, over the operand plane pairs
// first[g] .. first[g] + cnt[g] - 1, of A_pa B_pb^T.
//   digits (crt = 0): the sum as int32, plane g at out + g * plane words,
//     element (i, j) of batch z at z * z_step + j * ldp + i;
//   residues (crt = 1, one pair per group): the sum reduced modulo mod[g], a
//     signed byte; four columns share a word: word (j / 4) * ldp + i.  A group with
//     mod[g] = 0 multiplies magnitudes instead of integers: its byte is 1 where the sum
//     is zero or at least kMagnitudeFloor, else 0.
constexpr float kMagnitudeFloor = 1.f / 65536.f;

struct UnitArgs {
    int M, N, K;
    int nbatch;
    int ngroups;
    uint8_t pa[kUnitMaxPairs], pb[kUnitMaxPairs];
    uint8_t first[kUnitMaxGroups], cnt[kUnitMaxGroups];
    int a_row0, b_row0, a_row_step, b_row_step;
    float mod[kUnitMaxGroups], inv_mod[kUnitMaxGroups];
    uint32_t *out;
    int64_t plane, z_step;
    int ldp;
    const DevState *state;
    int *err;
    // set by the launcher
    int bn, tiles_m, tiles_n, kchunk, ppu, small;
};

// mapA, mapB: digit-plane maps with 128-row boxes and 64-wide K blocks.
// kmax: K range over which one pair's sum stays below 2^24.
int unit_gemm(const CUtensorMap &mapA, const CUtensorMap &mapB, const UnitArgs &a, bool crt, int kmax,
              cudaStream_t st);

}  // namespace tc
}  // namespace omm
