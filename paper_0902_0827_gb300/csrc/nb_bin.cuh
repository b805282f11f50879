// nb_bin.cuh - binning of one atom into its x-y column (section "Molecular
// dynamics on the GPU": atoms binned by their coordinates, one per thread,
// with atomic operations), shared by the binning kernel and by the MD
// half-steps, which bin the atoms they have just moved.
#pragma once

#include "nb_internal.cuh"

namespace acenb {

__device__ __forceinline__ int column_of(float x, float inv_w, int n)
{
    int c = (int)floorf(__fmul_rn(x, inv_w));
    if (c > n - 1) c = n - 1;
    if (c < 0) c = 0;
    return c;
}

// Warp-aggregated counter update: lanes with the same key (-1 = none) take
// consecutive positions from one atomic per distinct key; returns the old
// counter value plus the lane's rank among its peers.
__device__ __forceinline__ int warp_aggregated_add(int *counter_base, int key)
{
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (key >= 0 && lane == leader) base = atomicAdd(&counter_base[key], __popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    return base + __popc(peers & ((1u << lane) - 1u));
}

// The step's charges and types when they are in host memory, read by the
// binning kernel beside the positions (coalesced, in caller order, across
// the host link): the charge goes to the wrapped position's w, the
// range-checked type to atom_t, and the column sort carries both into sorted
// order.  q = null: positions only (w = 0); device-resident charges and
// types are gathered by the column sort instead (faster there).
struct AtomPack {
    const float *q;
    const int *type;
    int T;
    int *atom_t;  // [N] checked types in caller order
};

// Wrap, column, histogram and staging place of atom a (-1: none) of system s;
// every lane of the warp calls it.  A coordinate that is not finite, or too
// large for the FP32 wrap (|x| beyond about 2^24 L), is reported and taken as
// 0, so that every later index stays in range.
__device__ __forceinline__ void bin_atom(const BinArgs &B, int a, int s, float x, float y, float z, float q)
{
    int col = -1;
    if (a >= 0) {
        const SysDesc &S = B.sys[s];
        if (!(isfinite(x) && isfinite(y) && isfinite(z))) {
            atomicOr(B.status, ST_NONFINITE);
            x = 0.0f; y = 0.0f; z = 0.0f;
        }
        x = wrap_coord(x, S.L[0]);
        y = wrap_coord(y, S.L[1]);
        z = wrap_coord(z, S.L[2]);
        if (!(x >= 0.0f && x < S.L[0] && y >= 0.0f && y < S.L[1] && z >= 0.0f && z < S.L[2])) {
            atomicOr(B.status, ST_NONFINITE);
            x = 0.0f; y = 0.0f; z = 0.0f;
        }
        col = S.col_begin + column_of(y, S.inv_w[1], S.ny) * S.nx + column_of(x, S.inv_w[0], S.nx);
        B.atom_col[a] = col;
        B.wpos[a] = make_float4(x, y, z, q);
    }
    const int place = warp_aggregated_add(B.col_count, col);
    if (col >= 0 && place < B.col_cap) B.stage_fix[(long long)col * B.col_cap + place] = a;
}

}  // namespace acenb
