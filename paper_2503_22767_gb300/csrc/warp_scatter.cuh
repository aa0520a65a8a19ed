// Warp-aggregated stencil scatter of the 3D particle kernels (the P2G of the
// forward kernel, the G2P^T of the adjoint kernel).
#pragma once

#include "mpm_device.cuh"
#include "packed.cuh"

namespace mpm {

// ---------------------------------------------------------------------------
// Aggregated stencil scatter (the P2G of the forward kernel, the G2P^T of the
// adjoint kernel).
//
// The cell-sorted particles of one cell (8 per cell in 3D at the
// configurations' densities) share their base node, and so every stencil
// node; issued one per lane, their float4 atomics reach L2 as separate
// same-address updates.  Here the lanes of one base node (a group, found with
// one __match_any_sync) sum their contributions in shared memory first, slab
// by slab of kAggSlab stencil nodes: every lane writes its node values to its
// slot, then each quarter-warp takes one group and sums the group's value of
// one slab node per lane over the group's slots (in lane order), and issues
// one atomic per node.  A warp with G groups thus takes ceil(G / 4) passes
// per slab.
//
// The slots are ordered by group, so a group is a run of slots and its sum a
// walk with a fixed stride.  Cell-sorted lanes are in that order already
// (their slot is their lane); once particles have left the order, the slots
// come from a prefix sum over the group sizes.
//
// The 3D forward kernel is bound by the L1 data pipe (556 wavefronts per warp,
// 62% of peak, 40% of them here), so the split follows the wavefronts: a full
// slab is 8 lanes x 16 bytes of one slot, one conflict-free wavefront per
// group and slot.  1,000,000 particles, 100 forward substeps: 9,010 us with
// groups as lane masks walked by bit scans, 8,890 with planes of 9 nodes and
// three groups at a time (664 wavefronts: the 9-lane groups straddle the
// 8-lane phases), 9,450 with the slots cut into thirds and an atomic at every
// group's end, 8,480 with this split.
// ---------------------------------------------------------------------------
// Nodes per slab: 8, one per lane of a quarter-warp (27 = 8 + 8 + 8 + 3).  A
// lane's slots are 9 float4 apart (144 bytes, 36 banks), so the 8 lanes of a
// quarter-warp storing their values hit disjoint banks, and a quarter-warp
// summing one group reads 8 consecutive float4 of one slot.
constexpr int kAggSlab = 8;
constexpr int kAggStride = 9;
constexpr int kAggValueSlots = kAggStride * 32;  // float4 of node values per warp
// after the values, per group: first slot, size and base node (32 x int2)
constexpr int kAggTableSlots = 16;
constexpr int kAggSlots = kAggValueSlots + kAggTableSlots;  // float4 per warp

// Always in 3D (the forward kernel went from 98 to 59 us per launch on
// 600,000 particles).  In 2D, with 4 particles per cell, it pays only for
// large launches: the forward P2G of the 64-walker batch (1.5M particles) went
// from 81 to 72 us, while the single 30,000-particle walker lost 10% per
// design iteration and the 2D G2P^T lost on both.  2D P2G takes it per handle
// (Params::agg2, chosen by the autotuner); 2D G2P^T never does.
template <int D>
__host__ __device__ constexpr bool aggregate_scatter() {
    return D == 3;
}

// float4 slots of dynamic shared memory per warp of a particle kernel whose
// scatter is aggregated (AGG), none otherwise
template <int D, bool SCATTER, bool AGG = aggregate_scatter<D>()>
__host__ __device__ constexpr int warp_slots() {
    return SCATTER && AGG ? kAggSlots : 0;
}

// Offset of stencil node k (last axis fastest, k < 3^D) from the base node on
// a grid of res nodes per axis (res2 = res^2): k / 9, (k / 3) % 3 and k % 3
// by multiply and shift (exact for k < 27).
template <int D>
__device__ __forceinline__ int stencil_node_offset(int k, int res, int res2) {
    if (D == 3) {
        const int a0 = (k * 57) >> 9, r = k - 9 * a0;
        const int a1 = (r * 11) >> 5;
        return a0 * res2 + a1 * res + (r - 3 * a1);
    }
    const int a0 = (k * 11) >> 5;
    return a0 * res + (k - 3 * a0);
}

// Value of stencil node k (last axis fastest), w (base + sum_a o_a slope[a])
// at node offset o, for k = 0, 1, 2, ... in turn (k a constant of the
// unrolled loop).  Every component of a node is multiplied by the same
// rounded weight, so that the weight's error cancels in the node velocity
// (momentum over mass).
template <int D, typename V>
struct NodeValues {
    const Stencil<D>& s;
    const V& base;
    const V (&slope)[D];
    V row;     // base + slopes of all but the last axis at the current row
    float pw;  // the row's product of the other axes' weights

    __device__ __forceinline__ float4 operator()(int k) {
        constexpr int M = D - 2, L = D - 1;
        const int o0 = stencil_offset<D>(k, 0), om = stencil_offset<D>(k, M), ol = stencil_offset<D>(k, L);
        if (ol == 0) {
            row = om == 0 ? base : (om == 1 ? padd(base, slope[M]) : pfma(dup2(2.0f), slope[M], base));
            if (D == 3 && o0 > 0) row = o0 == 1 ? padd(row, slope[0]) : pfma(dup2(2.0f), slope[0], row);
            pw = D == 3 ? s.w[0][o0] * s.w[M][om] : s.w[M][om];
        }
        const V val = ol == 0 ? row : (ol == 1 ? padd(row, slope[L]) : pfma(dup2(2.0f), slope[L], row));
        return NodePack<D>::node(pmul(dup2(pw * s.w[L][ol]), val));
    }
};

// Every lane of the warp calls this; a lane without a particle passes
// active = false (its values go nowhere).  value(k) gives the float4 that
// stencil node k (last axis fastest) receives from this lane's particle; it
// is called with k = 0 .. 3^D - 1 in turn.  grid0 is instance 0's grid
// (instance i's starts nodes further on each; all grids together hold fewer
// than 2^31 nodes), nb the base node, sm this warp's kAggSlots slots.
template <int D, typename Value>
__device__ __forceinline__ void scatter_aggregated(int nb, int inst, bool active, float4* __restrict__ grid0,
                                                   long long nodes, int res, float4* sm, Value value) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // base node over all grids; negative and unlike any other without a particle
    const int base = active ? (int)((long long)inst * nodes) + nb : -1 - lane;
    const unsigned peers = __match_any_sync(full, base);
    const int leader = __ffs(peers) - 1;
    const unsigned run = peers >> leader;
    int slot = lane;
    if (!__all_sync(full, (run & (run + 1u)) == 0)) {
        // some group's lanes are not adjacent: order the slots by group
        const int size = lane == leader ? __popc(peers) : 0;
        int incl = size;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(full, incl, off);
            if (lane >= off) incl += y;
        }
        slot = __shfl_sync(full, incl - size, leader) + __popc(peers & ((1u << lane) - 1u));
    }
    const bool leads = active && lane == leader;
    const unsigned leaders = __ballot_sync(full, leads);
    const int G = __popc(leaders);
    int2* table = reinterpret_cast<int2*>(sm + kAggValueSlots);
    __syncwarp();  // the readers of an earlier call are done
    if (leads) table[__popc(leaders & ((1u << lane) - 1u))] = make_int2(slot | __popc(peers) << 8, base);
    constexpr int kNodes = D == 3 ? 27 : 9;
    const int n = lane & 7;  // this lane's node of a slab
    const int res2 = res * res;
    const float4* values = sm + n;
    float4* own = sm + slot * kAggStride;
#pragma unroll
    for (int k0 = 0; k0 < kNodes; k0 += kAggSlab) {
        const int nk = kNodes - k0 < kAggSlab ? kNodes - k0 : kAggSlab;  // nodes in this slab
        if (k0 > 0) __syncwarp();  // the slots' readers of the slab before are done
#pragma unroll
        for (int j = 0; j < kAggSlab; ++j)
            if (j < nk) own[j] = value(k0 + j);
        __syncwarp();
        if (nk < kAggSlab && n >= nk) continue;
        float4* node = grid0 + stencil_node_offset<D>(k0 + n, res, res2);
        for (int g = lane >> 3; g < G; g += 4) {
            const int2 e = table[g];
            const float4* c = values + (e.x & 255) * kAggStride;
            float4 v = c[0];
            float2 a01 = make_float2(v.x, v.y), a23 = make_float2(v.z, v.w);
#pragma unroll 2
            for (int m = (e.x >> 8) - 1; m > 0; --m) {
                c += kAggStride;
                v = c[0];
                a01 = __fadd2_rn(a01, make_float2(v.x, v.y));
                a23 = __fadd2_rn(a23, make_float2(v.z, v.w));
            }
            atomicAdd(node + e.y, make_float4(a01.x, a01.y, a23.x, a23.y));
        }
    }
}

}  // namespace mpm
