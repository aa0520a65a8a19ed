// Particle-array access shared by the transfer kernels.
//
// Particle arrays are structure-of-arrays with component stride P.np:
// x[D], v[D], C[D][D], E[D][D] (row-major), 2D + 2D^2 components, where
// E = F - I is the strain form of the deformation gradient.  Grids are one
// float4 per node.
#pragma once

#include <utility>

#include "kernels.h"
#include "packed.cuh"

namespace mpm {

// Launch a per-substep kernel; with P.pdl the launch allows programmatic
// dependent launch (the kernel begins with pdl_wait()).
// launch_chain_smem also gives the launch smem bytes of dynamic shared memory.
template <typename... KArgs, typename... Args>
cudaError_t launch_chain_smem(const Params& P, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = P.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_chain(const Params& P, void (*kernel)(KArgs...), dim3 grid, dim3 block,
                         cudaStream_t st, Args&&... args) {
    return launch_chain_smem(P, kernel, grid, block, 0, st, std::forward<Args>(args)...);
}

template <int D>
struct Layout {
    // F slot holds E = F - I
    static constexpr int X = 0, V = D, C = 2 * D, F = 2 * D + D * D, N = 2 * D + 2 * D * D;
};

template <int D>
__device__ __forceinline__ float4 pack4(float a, const float (&v)[D]) {
    return make_float4(a, v[0], v[1 % D], D == 3 ? v[2 % D] : 0.0f);
}

template <int D>
__device__ __forceinline__ void unpack3(const float4& g, float (&v)[D]) {
    v[0] = g.x;
    v[1 % D] = g.y;
    if (D == 3) v[2 % D] = g.z;
}

// A load that stays where it is written (asm volatile, so it is neither
// merged with an earlier load of the same address nor moved): reloading a
// value after a long stretch of code frees its registers in between.
__device__ __forceinline__ float reload(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

template <int D>
__device__ __forceinline__ void reload_mat(const float* __restrict__ s, int base, long long np, int p,
                                           float (&M)[D][D]) {
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b) M[a][b] = reload(s + (long long)(base + a * D + b) * np + p);
}

// The particle state is read once per kernel (a streaming read, evict-first),
// so that it does not push the stencil nodes the gathers reuse out of L1
// (3D locomotion, 1M particles: forward 97.6 -> 95.2 us per launch).
template <int D>
__device__ __forceinline__ void load_vec(const float* __restrict__ s, int base, long long np, int p,
                                         float (&v)[D]) {
#pragma unroll
    for (int a = 0; a < D; ++a) v[a] = __ldcs(s + (long long)(base + a) * np + p);
}

// Position of particle p: the X slot of the state plus x0 (the state holds
// the displacement u = x - x0; x0 null: the slot holds x itself).
template <int D>
__device__ __forceinline__ void load_position(const float* __restrict__ s, const float* __restrict__ x0,
                                              long long np, int p, float (&x)[D]) {
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const float u = __ldcs(s + (long long)a * np + p);
        x[a] = x0 ? __fadd_rn(u, __ldg(x0 + (long long)a * np + p)) : u;
    }
}

template <int D>
__device__ __forceinline__ void load_mat(const float* __restrict__ s, int base, long long np, int p,
                                         float (&M)[D][D]) {
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b) M[a][b] = __ldcs(s + (long long)(base + a * D + b) * np + p);
}

template <int D>
__device__ __forceinline__ void store_vec(float* __restrict__ s, int base, long long np, int p,
                                          const float (&v)[D]) {
#pragma unroll
    for (int a = 0; a < D; ++a) s[(long long)(base + a) * np + p] = v[a];
}

template <int D>
__device__ __forceinline__ void store_mat(float* __restrict__ s, int base, long long np, int p,
                                          const float (&M)[D][D]) {
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b) s[(long long)(base + a * D + b) * np + p] = M[a][b];
}

// Particle values parked in the warp's scatter slab while no register should
// hold them: component c of a lane at float c * 32 + lane.  park() copies from
// global memory without passing through registers (cp.async); a lane reads
// back only its own copies, after park_wait().
__device__ __forceinline__ void park(float4* sm, int c, const float* src) {
    float* dst = reinterpret_cast<float*>(sm) + c * 32 + (threadIdx.x & 31);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void park_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the last N committed groups have arrived
template <int N>
__device__ __forceinline__ void park_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// (volatile, as reload(): the value is read where it is written, not kept)
__device__ __forceinline__ float parked(const float4* sm, int c) {
    const float* src = reinterpret_cast<const float*>(sm) + c * 32 + (threadIdx.x & 31);
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"((unsigned)__cvta_generic_to_shared(src)));
    return v;
}

template <int D>
__device__ __forceinline__ void park_mat(float4* sm, int c, const float* __restrict__ s, int base, long long np, int p) {
#pragma unroll
    for (int k = 0; k < D * D; ++k) park(sm, c + k, s + (long long)(base + k) * np + p);
}
template <int D>
__device__ __forceinline__ void parked_mat(const float4* sm, int c, float (&M)[D][D]) {
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b) M[a][b] = parked(sm, c + a * D + b);
}

constexpr int kStencil2 = 9, kStencil3 = 27;
template <int D>
constexpr int stencil_size() { return D == 2 ? kStencil2 : kStencil3; }

// ---------------------------------------------------------------------------
// forward particle kernel
// ---------------------------------------------------------------------------
// Clears a.zero4 (grid-stride over the whole launch); fused mode only.
__device__ __forceinline__ void clear_buffer(const StepArgs& a) {
    if (a.zero4 == nullptr) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < a.zero_n; i += stride)
        a.zero4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Grid velocity at offset (o0, om, ol) of the stencil whose base node is
// grid[0] (2D: the offset is (om, ol)), packed: read from V (separate grid
// kernel), or the grid operation (Eq. 16-18) applied to the node's
// accumulator (fused).
template <int D, bool FUSE, bool BOXES = true>
__device__ __forceinline__ typename NodePack<D>::Vel load_node_velocity(const float4* __restrict__ grid,
                                                                        const Stencil<D>& s, const Params& P, int o0,
                                                                        int om, int ol, int step) {
    const float4 g = __ldg(grid + ((D == 3 ? o0 * P.res + om : om) * P.res + ol));
    if (!FUSE) return NodePack<D>::vel(g);
    float mv[D], gv[D];
    int c[D];
    unpack3<D>(make_float4(g.y, g.z, g.w, 0.0f), mv);
    if (D == 3) c[0] = s.base[0] + o0;
    c[D - 2] = s.base[D - 2] + om;
    c[D - 1] = s.base[D - 1] + ol;
    grid_velocity<D, BOXES>(P, c, g.x, mv, gv, step);
    return NodePack<D>::vel(gv);
}

// The adjoint (mbar, mvbar) of that node: from the grid adjoint kernel, or
// (FUSE) the reverse of the grid operation on the node's accumulator grid[.]
// and velocity adjoint vbar[.].
template <int D, bool FUSE, bool BOXES = true>
__device__ __forceinline__ typename NodePack<D>::Mass load_node_adjoint(const float4* __restrict__ grid,
                                                                        const float4* __restrict__ vbar,
                                                                        const Stencil<D>& s, const Params& P, int o0,
                                                                        int om, int ol, int step) {
    const int node = (D == 3 ? o0 * P.res + om : om) * P.res + ol;
    const float4 g = __ldg(grid + node);
    if (!FUSE) return NodePack<D>::mass(g);
    float mv[D], vb[D], mvb[D], mb;
    int c[D];
    unpack3<D>(make_float4(g.y, g.z, g.w, 0.0f), mv);
    unpack3<D>(__ldg(vbar + node), vb);
    if (D == 3) c[0] = s.base[0] + o0;
    c[D - 2] = s.base[D - 2] + om;
    c[D - 1] = s.base[D - 1] + ol;
    grid_velocity_adjoint<D, BOXES>(P, c, g.x, mv, vb, mb, mvb, step);
    return NodePack<D>::mass(mb, mvb);
}

}  // namespace mpm
