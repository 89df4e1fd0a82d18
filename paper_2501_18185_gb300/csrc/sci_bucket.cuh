// Walking the (N-2)-hole buckets: the disjointness test of two members and the window
// of buckets a CTA owns.  Shared by the sigma and density-matrix kernels, so that both
// enumerate exactly the same connections.
#pragma once

#include <cstdint>

#include "sci_internal.cuh"

namespace sci {

// Disjointness test of two members of one bucket.  A member with extra orbitals x < y
// is coded as bytes (x, y, x, y) when it is the bra (row) and (x', y', y', x') when it is
// the ket (column); the XOR of the two codes has a zero byte exactly when they share an
// orbital (x = x', y = y', x = y' or y = x').
__device__ __forceinline__ uint32_t row_code(uint32_t code)
{
    const uint32_t x = code & 0xFFu, y = (code >> 8) & 0xFFu;
    return x | (y << 8) | (x << 16) | (y << 24);
}
__device__ __forceinline__ uint32_t col_code(uint32_t code)
{
    const uint32_t x = code & 0xFFu, y = (code >> 8) & 0xFFu;
    return x | (y << 8) | (y << 16) | (x << 24);
}
__device__ __forceinline__ bool disjoint(uint32_t rc, uint32_t cc)
{
    const uint32_t v = rc ^ cc;
    return ((v - 0x01010101u) & ~v & 0x80808080u) == 0u;
}

// The doubles of a row among `n` <= 32 consecutive staged members, as a bit mask: bit u is
// set when member u shares no extra orbital with the row (rc: row_code of the row; code:
// the members' col_code words).  The row itself and its single excitations leave a 0.
__device__ __forceinline__ uint32_t doubles_mask(uint32_t rc, const uint32_t *code, int n)
{
    uint32_t m = 0;
    int u = 0;
    for (; u + 4 <= n; u += 4) {
        uint32_t g = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) g |= (uint32_t)disjoint(rc, code[u + k]) << k;
        m |= g << u;
    }
    for (; u < n; u++) m |= (uint32_t)disjoint(rc, code[u]) << u;
    return m;
}

// A CTA's stable counting sort of the rows it owns by a key below 64: each warp counts its
// rows by sort_rank() in its own histogram (zeroed before), a barrier, one warp runs
// sort_prefix(), a barrier; a row then goes to base[key] + hist[warp][key] + its rank.
//
// sort_rank(): the rank of this lane's row (key < 0: it has none) among the rows of its warp
// with the same key, in the order of calls and lanes.  Called by whole warps.
__device__ __forceinline__ int sort_rank(int key, uint16_t *hist, int lane)
{
    const unsigned act = __ballot_sync(0xffffffffu, key >= 0);
    unsigned same = 0;
    int rank = 0;
    if (key >= 0) {
        same = __match_any_sync(act, key);
        rank = hist[key] + __popc(same & ((1u << lane) - 1u));
    }
    __syncwarp();
    if (key >= 0 && (same >> lane) == 1u) hist[key] = (uint16_t)(rank + 1);   // last of its bin
    __syncwarp();
    return rank;
}
// exclusive prefix over (bin, warp), by one warp; lane l owns bins 2l and 2l + 1
template <int WARPS>
__device__ __forceinline__ void sort_prefix(uint16_t (*hist)[64], int lane, int *base, int &total)
{
    int tot[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        int run = 0;
#pragma unroll
        for (int w = 0; w < WARPS; w++) {
            const int c = hist[w][2 * lane + h];
            hist[w][2 * lane + h] = (uint16_t)run;
            run += c;
        }
        tot[h] = run;
    }
    int inc = tot[0] + tot[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    base[2 * lane] = inc - tot[0] - tot[1];
    base[2 * lane + 1] = inc - tot[1];
    if (lane == 31) total = inc;
}

// The rows of CTA b: the buckets that start in [b*CH, (b+1)*CH), i.e. from the start of
// the bucket holding row b*CH to the start of the bucket holding row (b+1)*CH.  Every
// bucket lands in exactly one window; a window has at most CH + maxb - 1 rows (it can be
// empty when one bucket spans a whole range).
__device__ __forceinline__ void window_of(const uint32_t *__restrict__ e_pos, int64_t E, int CH, int64_t b, int64_t &r0,
                                          int64_t &r1)
{
    const int64_t a0 = b * CH, a1 = a0 + CH;
    r0 = a0 - pos_off(e_pos[a0]);
    r1 = a1 < E ? a1 - pos_off(e_pos[a1]) : E;
}
__device__ __forceinline__ void window(const uint32_t *__restrict__ e_pos, int64_t E, int CH, int64_t &r0, int64_t &r1)
{
    window_of(e_pos, E, CH, blockIdx.x, r0, r1);
}

}  // namespace sci
