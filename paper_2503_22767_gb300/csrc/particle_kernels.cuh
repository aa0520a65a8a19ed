// Particle kernels of the magneto-elastic MLS-MPM substep and its reverse.
//
// Forward (arxiv 2503.22767, Section 2.2): the particle kernel fuses the G2P
// of substep n (Eq. 19-22) with the P2G of substep n+1 (Eq. 14-15 with the
// SIMP-scaled stress of Eq. 7/31-33), so between substeps a particle's state
// is read once and written once.  Reverse (Section 2.3): the particle kernel
// fuses the P2G^T of substep n with the G2P^T of substep n-1.
//
// Particle arrays are structure-of-arrays with component stride P.np:
// x[D], v[D], C[D][D], E[D][D] (row-major), i.e. 2D + 2D^2 components, where
// E = F - I is the strain form of the deformation gradient (see
// mpm_device.cuh: it keeps small strains exact to float32 precision).
// Grids are float4 per node ([inst][node]): accumulators (m, mv), velocities
// (v, 0), adjoints (mbar, mvbar).
//
// The kernels are templates over the dimension and the fused stages; each
// dimension and direction is instantiated in a translation unit of its own
// (kernels_particle2.cu, kernels_forward3.cu, kernels_adjoint3.cu), so they
// compile in parallel.
#pragma once

#include <type_traits>

#include "kernels.h"
#include "particle_io.cuh"
#include "stencil_sums.cuh"
#include "warp_scatter.cuh"

namespace mpm {

// Resident 256-thread blocks per SM that the register allocation must allow
// (the compiler caps registers at 65536 / (256 x this)).  The transfer kernels
// are latency-bound, so occupancy is traded against spills: the 3D forward
// kernel is held to 64 registers, and the adjoint kernel is compiled for 2
// (<= 128 registers), 3 (<= 80) and, in 2D, 4 (<= 64) blocks, chosen per
// launch (Params::adj_blocks; 4 acts as 3 in 3D).
//
// In 3D two rules go beyond the option.  A body that one wave of 128-register
// kernels holds (Params::wave, 77,824 particles on 152 SMs) gains nothing from
// more warps per SM, so both kernels take 128 registers: design gradient of
// 64,000 particles 3,418 -> 3,069 us, of 14,304 1,493 -> 1,416; of 79,816, just
// past the wave, it would lose 14%.  Larger bodies in blocks of up to 128
// threads run the adjoint with five blocks of 128 threads per SM (96
// registers, 36 instead of 244 bytes of spill loads): 64,000 particles 3,460
// -> 3,380 us, 3 x 200,000 15,380 -> 15,335, 1,000,000 25.01 -> 24.91 ms;
// blocks of 256 keep 80 registers (96 would leave two of them: +7%).
constexpr int kMinBlocksForward3 = 4;
constexpr int kMinBlocksOneWave = 2;
constexpr int kBlocksOf128 = 5;  // MINB of the adjoint kernel for blocks of up to 128 threads
// 2D: with the aggregated P2G (large launches) at most 48 registers (40 warps
// per SM, no spills; the 2D batch's forward launch went from 83 to 79 us);
// with per-lane atomics 64 (a small body's blocks are far from filling the GPU)
constexpr int kMinBlocksForward2 = 4, kMinBlocksForward2Agg = 5;

namespace {

inline int particle_blocks(long long n, int block) { return (int)((n + block - 1) / block); }

// The forward step of particle p (G2P of substep a.n_g2p and/or P2G of
// a.n_p2g); every lane of a warp calls it together, with particles
// 32w .. 32w + 31 (w = p / 32).  sm: this warp's warp_slots<D, P2G>()
// float4 of shared memory (the scatter slab of P2G).
// EXT: P.ext is set (solid boxes or a non-uniform field); without it the
// code for them is left out.  CHAIN: the kernel is one launch of a chain
// with programmatic dependent launch (k_forward); a persistent kernel calls
// this between its own grid-wide barriers instead.  AGG_P2G: the P2G scatter
// is aggregated over the lanes of one base node (scatter_aggregated).
template <int D, bool G2P, bool P2G, bool WRITE_ALL, bool FUSE, bool EXT, bool CHAIN,
          bool AGG_P2G = aggregate_scatter<D>()>
__device__ __forceinline__ void forward_particle(const Params& P, const StepArgs& a, int p, float4* sm) {
    using L = Layout<D>;
    // Early loads: with the grid operation in its own kernel, this kernel's
    // predecessor is that grid kernel, which writes none of the particle
    // arrays read first here.  Every kernel of the chain waits before it
    // triggers its dependents, so when this kernel starts, the particle
    // kernel before the grid kernel has completed, and the state loads can
    // overlap the grid kernel's tail.
    constexpr bool kEarly = CHAIN && G2P && !FUSE;
    // the P2G scatter is aggregated over the lanes of one cell (scatter_aggregated)
    constexpr bool AGG = P2G && AGG_P2G;
    const bool active = p < P.n_total;
    const int inst = active ? find_instance(a.inst_off, P.n_inst, p) : -1;
    const long long np = P.np;
    int flags = 0;
    // x: the X slot (the displacement u = x - x0 when a.x0 is set); every
    // stencil and field evaluation uses the position x0 + u (pos below)
    // xo: x0 (0 without a.x0), loaded with the state for G2P and again after
    // the G2P node loop for P2G, so that it holds no registers in the loop
    float x[D], v[D], C[D][D], F[D][D], xo[D];
    float phi = 0.0f, mp = 0.0f;
    // In 2D with per-lane atomics (small bodies: a chain of short launches)
    // the design and field of P2G are loaded with the state, so that their
    // latency passes while the kernel waits for its predecessor (half-size
    // walker, forward only: 1,664 -> 1,607 us per 400 substeps, with 64
    // instead of 48 registers allowed).  The launches that fill the GPU need
    // the registers more: loaded early, the 2D batch lost 1.7%; in 3D, copied
    // early into the scatter slab, 1,000,000 particles lost 8%.
    constexpr bool kHoist = D == 2 && P2G && !AGG_P2G;
    float Br[D], Ba[D];
    auto load_design = [&]() {
#pragma unroll
        for (int i = 0; i < D; ++i) {
            Br[i] = a.mag[(long long)i * np + p];
            Ba[i] = __ldg(a.field + ((long long)inst * P.n_steps + a.n_p2g) * D + i);
        }
    };
    auto position = [&](float (&pos)[D]) {
#pragma unroll
        for (int i = 0; i < D; ++i) pos[i] = __fadd_rn(x[i], xo[i]);
    };
    auto load_state = [&]() {
        load_vec<D>(a.s_in, L::X, np, p, x);
#pragma unroll
        for (int i = 0; i < D; ++i) xo[i] = a.x0 ? __ldg(a.x0 + (long long)i * np + p) : 0.0f;
        load_mat<D>(a.s_in, L::F, np, p, F);
        phi = a.phi[p];
        mp = phi * P.rho0 * P.p_vol;  // Eq. 33
        if (!G2P) {
            load_vec<D>(a.s_in, L::V, np, p, v);
            load_mat<D>(a.s_in, L::C, np, p, C);
        }
        if (kHoist) load_design();
    };
    if (kEarly && active) load_state();
    if (CHAIN) {
        pdl_wait();
        pdl_trigger();
        if (FUSE) clear_buffer(a);
    }
    if (!kEarly && active) load_state();
    if (G2P) {
        float mom_x[1] = {0.0f};
        Stencil<D> s;
#pragma unroll
        for (int i = 0; i < D; ++i) s.base[i] = 0;
        if (active) {
            float pos[D];
            position(pos);
            if (!make_stencil<D>(pos, P, s)) flags |= kErrDomain;
        }
        const float4* __restrict__ Vg = FUSE ? a.accG : a.V;
        if (active) {
            const float4* __restrict__ Vi = Vg + (long long)inst * P.nodes;
            // Eq. 19-20 with x_i - x_p = (o - r) dx for stencil offset o:
            //   v = sum w V,  C = (4/dx) sum w V (o - r)^T
            const float4* __restrict__ Vn = Vi + base_node<D>(s, P.res);
            typename NodePack<D>::Vel vp, Mp[D];
            gather_velocity<D>(
                s,
                [&](int o0, int om, int ol) {
                    return load_node_velocity<D, FUSE, EXT>(Vn, s, P, o0, om, ol, a.n_g2p);
                },
                vp, Mp);
            NodePack<D>::get(vp, v);
            if (P2G && a.x0 && !kHoist) {  // x0 again for the P2G position; the load overlaps the G2P tail
#pragma unroll
                for (int i = 0; i < D; ++i) xo[i] = reload(a.x0 + (long long)i * np + p);
            }
            float Fn[D][D];
#pragma unroll
            for (int j = 0; j < D; ++j) {
                float m[D];
                NodePack<D>::get(Mp[j], m);
                const float c4 = (j == D - 1 ? 0.5f : 4.0f) * P.inv_dx;
#pragma unroll
                for (int i = 0; i < D; ++i) C[i][j] = c4 * m[i];
                x[j] += P.dt * v[j];                              // Eq. 21 (on u = x - x0)
            }
            // Eq. 22 in strain form: E' = E + dt C (I + E)
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    float acc = C[i][j];
#pragma unroll
                    for (int k = 0; k < D; ++k) acc += C[i][k] * F[k][j];
                    Fn[i][j] = F[i][j] + P.dt * acc;
                }
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) F[i][j] = Fn[i][j];
            float Jm1 = det_minus_one<D>(F);
            if (!(Jm1 > -1.0f) || !isfinite(Jm1)) flags |= kErrNumeric;
            store_vec<D>(a.s_out, L::X, np, p, x);
            store_mat<D>(a.s_out, L::F, np, p, F);
            if (WRITE_ALL) {
                // v and C of a stored state are read only by the adjoint, a
                // segment later (the next substep's G2P computes its own):
                // streaming stores keep them from evicting the grids from L2
                // (2D batch, store passes: forward 89.6 -> 84.0 us per launch)
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    __stcs(a.s_out + (long long)(L::V + i) * np + p, v[i]);
#pragma unroll
                    for (int j = 0; j < D; ++j) __stcs(a.s_out + (long long)(L::C + i * D + j) * np + p, C[i][j]);
                }
            }
            mom_x[0] = mp * v[0];
        }
        // Eq. 40's momentum row: a large body's sum cancels to a small part of
        // its terms, so thousands of warps add in 64 bits, spread over slots
        // so that they do not queue for one address
        if (P.loss_kind == 1 && a.mom_acc != nullptr)
            warp_add_per_instance<1>(mom_x, inst,
                                     a.mom_acc + (long long)a.n_g2p * P.n_inst * a.slots + ((p >> 5) & (a.slots - 1)),
                                     a.slots);
    }
    if (P2G) {
        // this warp's box of listed cells, read after the scatter (3D)
        if (D == 3 && a.blk.flag != nullptr) prefetch_l1(a.blk.wbox + (p >> 5));
        Stencil<D> s;
        float A[D][D], u[D];
        int nb = 0;
        float4* __restrict__ ai = a.acc + (long long)(active ? inst : 0) * P.nodes;
        if (active) {
            float pos[D];
            position(pos);
            if (!make_stencil<D>(pos, P, s)) flags |= kErrDomain;
            StressParts<D> S;
            stress_parts<D>(F, phi, P, S);
            if (!(S.J > 0.0f)) flags |= kErrNumeric;
            float Pk[D][D];
            if (!kHoist) load_design();
            if (EXT && P.ext->fgrad) {
                const float* Gn = P.ext->fgrad + ((long long)inst * P.n_steps + a.n_p2g) * D * D;
                field_at_particle<D>(Gn, pos, Ba);
                // body force of the non-uniform field, folded into the momentum
                // m v (f and m both vanish with phi, so m > 0 whenever f != 0)
                float f[D];
                magnetic_force<D>(Gn, F, Br, S.s, P, f);
                if (mp > 0.0f) {
#pragma unroll
                    for (int i = 0; i < D; ++i) v[i] += P.dt * f[i] / mp;
                }
            }
            piola<D>(S, Br, Ba, Pk);
            const float sc = P.dt * P.kappa * P.p_vol;
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    float pft = Pk[i][j];  // (P F^T)_ij with F = I + E
#pragma unroll
                    for (int k = 0; k < D; ++k) pft += Pk[i][k] * F[j][k];
                    // MLS-MPM affine momentum (Eq. 15 with the time step and the
                    // x_i - x_p offset of the MLS-MPM form): m C - dt (4/dx^2) V P F^T
                    A[i][j] = mp * C[i][j] - sc * pft;
                }
            // Eq. 15 with x_i - x_p = (o - r) dx: node momentum w (u + dx A o),
            // u = m v - dx A r
#pragma unroll
            for (int i = 0; i < D; ++i) {
                float ar = 0.0f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    A[i][j] *= P.dx;
                    ar += A[i][j] * s.r[j];
                }
                u[i] = mp * v[i] - ar;
            }
            nb = base_node<D>(s, P.res);
        } else {  // a lane past the end takes part in the aggregated scatter with zeros
#pragma unroll
            for (int i = 0; i < D; ++i) {
                u[i] = 0.0f;
                s.base[i] = 0;
#pragma unroll
                for (int j = 0; j < D; ++j) A[i][j] = 0.0f;
#pragma unroll
                for (int j = 0; j < 3; ++j) s.w[i][j] = 0.0f;
            }
        }
        // node (o0, .., ol) receives w (mp, u + dx A o)  (Eq. 14 in the first component)
        using NP = NodePack<D>;
        const typename NP::Mass U = NP::mass(mp, u);
        typename NP::Mass As[D];
#pragma unroll
        for (int j = 0; j < D; ++j) {
            float col[D];
#pragma unroll
            for (int i = 0; i < D; ++i) col[i] = A[i][j];
            As[j] = NP::mass(0.0f, col);
        }
        if constexpr (AGG) {
            scatter_aggregated<D>(nb, inst, active, a.acc, P.nodes, P.res, sm,
                                  NodeValues<D, typename NP::Mass>{s, U, As, U, 0.0f});
            // the warp lists the node blocks its stencils reach beyond its box
            // (a.blk is uniform over the launch, so the whole warp takes part)
            if constexpr (D == 3) {
                if (a.blk.flag != nullptr) mark_blocks(a.blk, p >> 5, active, inst, s.base, P.res, a.blk.wbox[p >> 5]);
            }
        } else if (active) {
            float4* __restrict__ an = ai + nb;
            NodeValues<D, typename NP::Mass> value{s, U, As, U, 0.0f};
#pragma unroll
            for (int k = 0; k < stencil_size<D>(); ++k) atomicAdd(an + node_offset<D>(k, P.res), value(k));
        }
    }
    if (flags) atomicOr(a.err, flags);
}

// 3D: at most 64 registers (32 warps per SM) to keep more gathers in flight
template <int D, bool AGG>
constexpr int forward_min_blocks() {
    return D == 3 ? kMinBlocksForward3 : AGG ? kMinBlocksForward2Agg : kMinBlocksForward2;
}
template <int D, bool G2P, bool P2G, bool WRITE_ALL, bool FUSE, bool EXT, bool AGG = aggregate_scatter<D>(),
          int MINB = forward_min_blocks<D, AGG>()>
__global__ void __launch_bounds__(256, MINB) k_forward(Params P, StepArgs a) {
    extern __shared__ float4 s_warp[];
    forward_particle<D, G2P, P2G, WRITE_ALL, FUSE, EXT, true, AGG>(
        P, a, blockIdx.x * blockDim.x + threadIdx.x, s_warp + (threadIdx.x >> 5) * warp_slots<D, P2G, AGG>());
}


// ---------------------------------------------------------------------------
// adjoint particle kernel
//   P2GT: reverse of P2G at substep n = a.n_p2g; completes the particle
//         adjoint of state n (x, v, C, F), accumulates design gradients.
//   G2PT: reverse of G2P at substep m (= n-1 when fused, else n): consumes
//         the adjoint of state m+1, scatters Vbar, writes the partial
//         adjoint (x, F) of state m.
// ---------------------------------------------------------------------------
// FUSE: P2G^T evaluates the grid adjoint per stencil node from (accP, VbarIn);
// FUSE_V: G2P^T takes the grid velocity from accG through the grid operation.
// EXT: P.ext is set (solid boxes or a non-uniform field), as in k_forward.
// CHAIN and the calling convention as in forward_particle; sm: this warp's
// warp_slots<D, G2PT>() float4 (the scatter slab of G2P^T).  RELIEF: the
// register budget is tight (96 registers or fewer, in 3D also 128), so the
// state and stress of P2G^T are reloaded and recomputed after its node loop
// (3D at 128 registers: 216 -> 12 bytes of spill loads; 64,000 particles 3,050
// -> 3,015 us, 82,944 in a non-uniform field 2,530 -> 2,443).
template <int D, bool P2GT, bool G2PT, bool FUSE, bool FUSE_V, bool EXT, bool CHAIN, bool RELIEF>
__device__ __forceinline__ void adjoint_particle(const Params& P, const StepArgs& a, int p, float4* sm) {
    using L = Layout<D>;
    // Early loads as in k_forward: the fused kernel without grid-adjoint
    // fusion follows the grid adjoint kernel, which writes none of the
    // particle arrays of state n, the partial adjoint or the design.
    constexpr bool kEarly = CHAIN && P2GT && G2PT && !FUSE;
    // The late P2G^T epilogue (kLate): under the 80-register budget of the 3D
    // kernel it cuts the spills from 188 to 88 bytes per thread (3D
    // locomotion, 1M particles: 198.1 -> 196.0 us per launch, 3 x 200,000
    // particles: 119.3 -> 117.4 us).  The 2D budgets spill nothing in the
    // plain order and lose with this one (2D batch: 108.3 -> 112.3 us).
    constexpr bool kLate = RELIEF && D == 3;
    // The matrices of the fused 3D kernel wait in the scatter slab (idle until
    // the scatter at the end; 4 x 9 floats a lane fill it): C, E and Fbar of
    // state n and E of state m, copied there without registers while the
    // kernel still waits for its predecessor (as loads where each is used, C
    // read three times and E twice: 3D plate, 3 x 200,000 particles, design
    // gradient 16,220 us; parked: 15,955).
    constexpr bool kPark = kLate && P2GT && G2PT;
    constexpr int kParkC = 0, kParkE = D * D, kParkFb = 2 * D * D, kParkEm = 3 * D * D;
    const bool active = p < P.n_total;
    const int inst = active ? find_instance(a.inst_off, P.n_inst, p) : -1;
    const long long np = P.np;
    int flags = 0;
    // adjoint of the state between the two halves (state n if P2GT)
    float xb[D], vb[D], Cb[D][D], Fb[D][D];
    float Cn[D][D];  // C of state n (= m+1), needed by G2P^T
    float x_n[D], v_n[D], F_n[D][D], phi_n = 0.0f;  // state n and design (P2G^T)
    // 2D: the design and field with the state, as in the forward kernel (2D
    // walker's design gradient 5,355 -> 5,270 us; the 3D plate lost 0.5%)
    float Br[D], Ba[D];
    auto load_design = [&]() {
#pragma unroll
        for (int i = 0; i < D; ++i) {
            Br[i] = a.mag[(long long)i * np + p];
            Ba[i] = __ldg(a.field + ((long long)inst * P.n_steps + a.n_p2g) * D + i);
        }
    };
    // 2D with registers to spare (the 128-register budget of small bodies): the
    // adjoint of F, the state of m and the locomotion seed too (walker 5,160 ->
    // 5,030 -> 4,860 us; the 64-register launches of the batch lost 1%)
    constexpr bool kAhead = D == 2 && P2GT && G2PT && !RELIEF;
    float x_m[D], F_m[D][D];
    constexpr bool kSeed = D == 2 && !RELIEF;
    float M_n = 0.0f, dl_n = 0.0f, mom_n = 0.0f;
    auto load_seed = [&]() {
        if (P.loss_kind == 1 && a.n_p2g >= 1) {
            M_n = a.Minst[inst];
            dl_n = a.dloss[inst];
            mom_n = a.mom[(long long)(a.n_p2g - 1) * P.n_inst + inst];
        }
    };
    auto load_state_n = [&]() {
        if (kSeed) load_seed();
        if (kAhead) {
            load_mat<D>(a.adj, L::F, np, p, Fb);
            load_position<D>(a.s_aux, a.x0, np, p, x_m);
            load_mat<D>(a.s_aux, L::F, np, p, F_m);
        }
        load_position<D>(a.s_in, a.x0, np, p, x_n);  // the position x0 + u
        load_vec<D>(a.s_in, L::V, np, p, v_n);
        // C and E are read again after the P2G^T node loop under RELIEF:
        // plain loads, so that the second read finds them cached
        if (kPark) {
            park_mat<D>(sm, kParkC, a.s_in, L::C, np, p);
            park_mat<D>(sm, kParkE, a.s_in, L::F, np, p);
            park_commit();
            park_mat<D>(sm, kParkFb, a.adj, L::F, np, p);
            park_mat<D>(sm, kParkEm, a.s_aux, L::F, np, p);
            park_commit();
        } else
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) {
                Cn[i][j] = RELIEF ? __ldg(a.s_in + (long long)(L::C + i * D + j) * np + p)
                                  : __ldcs(a.s_in + (long long)(L::C + i * D + j) * np + p);
                F_n[i][j] = RELIEF ? __ldg(a.s_in + (long long)(L::F + i * D + j) * np + p)
                                   : __ldcs(a.s_in + (long long)(L::F + i * D + j) * np + p);
            }
        load_vec<D>(a.adj, L::X, np, p, xb);
        phi_n = a.phi[p];
        if (D == 2) load_design();
    };
    if (kEarly && active) load_state_n();
    if (P2GT && G2PT && active) {
        // x and E of state m = n-1 (G2P^T) come from the segment store in HBM;
        // request them now so that their loads after P2G^T find them in L2
#pragma unroll
        for (int c = 0; c < D; ++c) prefetch_l2(a.s_aux + (long long)(L::X + c) * np + p);
        if (!kPark) {
#pragma unroll
            for (int c = 0; c < D * D; ++c) prefetch_l2(a.s_aux + (long long)(L::F + c) * np + p);
        }
    }
    if (P2GT && active) {  // the design and its gradients, read late in P2G^T
        prefetch_l2(a.gphi + p);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            prefetch_l2(a.mag + (long long)c * np + p);
            prefetch_l2(a.gmag + (long long)c * np + p);
        }
    }
    if (CHAIN) {
        pdl_wait();
        pdl_trigger();
        clear_buffer(a);
    }
    if (P2GT && !kEarly && active) load_state_n();
    constexpr bool AGG = G2PT && aggregate_scatter<D>();
    float bab[D];
#pragma unroll
    for (int i = 0; i < D; ++i) bab[i] = 0.0f;
    // non-uniform field: G of this substep (uniform over the launch), and the
    // particle's contribution to dL/dG
    const bool has_fgrad = EXT && P2GT && P.ext->fgrad;
    float gG[D * D];
#pragma unroll
    for (int i = 0; i < D * D; ++i) gG[i] = 0.0f;
    if (P2GT) {
        if (active) {
            const int n = a.n_p2g;
            const float* Gn = has_fgrad ? P.ext->fgrad + ((long long)inst * P.n_steps + n) * D * D : nullptr;
            float(&x)[D] = x_n;
            float(&v)[D] = v_n;
            float(&F)[D][D] = F_n;
            const float phi = phi_n;
            const float mp = phi * P.rho0 * P.p_vol;
            float Pk[D][D], A[D][D];
            if (D == 3) load_design();
            if (Gn) field_at_particle<D>(Gn, x, Ba);
            Stencil<D> s;
            if (!make_stencil<D>(x, P, s)) flags |= kErrDomain;
            if (kPark) {
                park_wait<1>();
                parked_mat<D>(sm, kParkE, F);
                parked_mat<D>(sm, kParkC, Cn);
            }
            StressParts<D> S;
            stress_parts<D>(F, phi, P, S);
            piola<D>(S, Br, Ba, Pk);
            const float sc = P.dt * P.kappa * P.p_vol;
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    float pft = Pk[i][j];  // (P F^T)_ij with F = I + E
#pragma unroll
                    for (int k = 0; k < D; ++k) pft += Pk[i][k] * F[j][k];
                    A[i][j] = mp * Cn[i][j] - sc * pft;
                }
            // Node sums with x_i - x_p = (o - r) dx (o the stencil offset):
            //   S0 = sum w mvb,  T = sum w mvb (o - r)^T,  mbs = sum w mb
            // give vbar = mp S0, Abar = dx T and
            // mbar_p = mbs + S0 . v + C : Abar.  The node's contribution to
            // the particle's momentum is
            //   mb mp + mvb . (mp v + dx A (o - r)),
            // whose weighted sum's derivative with respect to r is dx xbar
            // (adjoint_sums).
            float u[D], dA[D][D];  // dA[c][i] = dx A_ic
#pragma unroll
            for (int i = 0; i < D; ++i) {
#pragma unroll
                for (int j = 0; j < D; ++j) dA[j][i] = P.dx * A[i][j];
                u[i] = mp * v[i];
            }
            if (Gn) {  // the body force is part of the particle's momentum term
                float f[D];
                magnetic_force<D>(Gn, F, Br, S.s, P, f);
#pragma unroll
                for (int i = 0; i < D; ++i) u[i] += P.dt * f[i];
            }
            using NP = NodePack<D>;
            const int nb = base_node<D>(s, P.res);
            const float4* __restrict__ gi = (FUSE ? a.accP : a.gadj) + (long long)inst * P.nodes + nb;
            const float4* __restrict__ vbi = FUSE ? a.VbarIn + (long long)inst * P.nodes + nb : nullptr;
            float S0[D], mbs, xg[D];
            typename NP::Mom Tp[D];
            {
                typename NP::Mass Sp;
                typename NP::Mom Ap[D];
#pragma unroll
                for (int c = 0; c < D; ++c) Ap[c] = NP::mom(dA[c]);
                adjoint_sums<D, true>(
                    s,
                    [&](int o0, int om, int ol) {
                        return load_node_adjoint<D, FUSE, EXT>(gi, vbi, s, P, o0, om, ol, a.n_p2g);
                    },
                    NP::mass(mp, u), Ap, Sp, Tp, xg);
                NP::get(Sp, mbs, S0);
            }
            // The node loop needs none of C, E, the stress (all used for A
            // before it) and Fbar of state n.  Under a tight register budget
            // (RELIEF) they are read again, and the stress recomputed, here, so
            // their registers are free during the loop (the recomputation is
            // cheaper than the spills); with registers to spare they stay live.
            // kLate: E, the stress and Fbar are formed only where first used,
            // and P element by element.
            if (kPark) {
                park_wait<0>();
                parked_mat<D>(sm, kParkC, Cn);
            } else if (RELIEF) {
                reload_mat<D>(a.s_in, L::C, np, p, Cn);
            }
            if (RELIEF && !kLate) reload_mat<D>(a.s_in, L::F, np, p, F);
            if (!kLate && !kAhead) load_mat<D>(a.adj, L::F, np, p, Fb);
            if (RELIEF && !kLate) {
                stress_parts<D>(F, phi, P, S);
                piola<D>(S, Br, Ba, Pk);
            }
            float Ab[D][D], mpb = mbs;
#pragma unroll
            for (int j = 0; j < D; ++j) {
                float tj[D];
                NP::get_mom(Tp[j], tj);
                xb[j] += P.inv_dx * xg[j];
                vb[j] = mp * S0[j];
                mpb += S0[j] * v[j];
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    Ab[i][j] = (j == D - 1 ? 0.125f : 1.0f) * P.dx * tj[i];
                    mpb += Cn[i][j] * Ab[i][j];
                }
            }
            // A = mp C - sc P F^T:  Pbar = -sc Abar F,  Fbar -= sc Abar^T P
            float Pb[D][D];
            if (!kLate) {
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int j = 0; j < D; ++j) Cb[i][j] = mp * Ab[i][j];
            }
            if (kPark) parked_mat<D>(sm, kParkE, F);
            else if (kLate) reload_mat<D>(a.s_in, L::F, np, p, F);
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    float pb = Ab[i][j], fb = 0.0f;  // (Abar F)_ij with F = I + E
#pragma unroll
                    for (int k = 0; k < D; ++k) {
                        pb += Ab[i][k] * F[k][j];
                        if (!kLate) fb += Ab[k][i] * Pk[k][j];  // (Abar^T P)_ij
                    }
                    Pb[i][j] = -sc * pb;
                    if (!kLate) Fb[i][j] -= sc * fb;
                }
            if (kLate) {
                stress_parts<D>(F, phi, P, S);
                if (kPark) parked_mat<D>(sm, kParkFb, Fb);
                else load_mat<D>(a.adj, L::F, np, p, Fb);
                // P_kj as piola() forms it, used by its three products at once
                const float smu = S.s * (1.0f / kMu0);
#pragma unroll
                for (int k = 0; k < D; ++k)
#pragma unroll
                    for (int j = 0; j < D; ++j) {
                        const float pk = S.sE * (S.a * S.dev[k][j] + S.b * S.H[k][j]) - smu * Ba[k] * Br[j];
#pragma unroll
                        for (int i = 0; i < D; ++i) Fb[i][j] -= sc * (Ab[k][i] * pk);
                    }
            }
            float phib = 0.0f, brb[D];
#pragma unroll
            for (int i = 0; i < D; ++i) brb[i] = 0.0f;
            piola_adjoint<D>(F, phi, S, Br, Ba, Pb, P, Fb, phib, brb, bab);
            if (kLate) {
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int j = 0; j < D; ++j) Cb[i][j] = mp * Ab[i][j];
            }
            float gph = phib + mpb * P.rho0 * P.p_vol;
            if (Gn) {
                // B at the particle = B_a + G (x - x_c): dL/dB_a stays in bab,
                // dL/dG += bab (x - x_c)^T, xbar += G^T bab
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int j = 0; j < D; ++j) {
                        gG[i * D + j] += bab[i] * (x[j] - 0.5f);
                        xb[j] += __ldg(Gn + i * D + j) * bab[i];
                    }
                // body force f = c G^T (F B~_r), c = s V / mu0, whose adjoint is
                // fbar = dt sum_i w mvb_i = dt S0
                const float c = S.s * P.p_vol * (1.0f / kMu0);
                float FB[D], Gfb[D], fraw = 0.0f;
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    FB[i] = Br[i];
                    Gfb[i] = 0.0f;
#pragma unroll
                    for (int k = 0; k < D; ++k) {
                        FB[i] += F[i][k] * Br[k];
                        Gfb[i] += __ldg(Gn + i * D + k) * (P.dt * S0[k]);
                    }
                }
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    fraw += Gfb[i] * FB[i];
#pragma unroll
                    for (int k = 0; k < D; ++k) {
                        Fb[i][k] += c * Gfb[i] * Br[k];
                        brb[k] += c * Gfb[i] * ((i == k ? 1.0f : 0.0f) + F[i][k]);
                        gG[i * D + k] += c * FB[i] * (P.dt * S0[k]);
                    }
                }
                const float ds = P.simp_q > 0 ? (float)P.simp_q * int_pow(phi, P.simp_q - 1) : 0.0f;
                gph += ds * P.p_vol * (1.0f / kMu0) * fraw;
            }
            // locomotion seed on state n (n >= 1), Eq. 40
            if (P.loss_kind == 1 && n >= 1) {
                if (!kSeed) load_seed();
                const float M = M_n, dl = dl_n;
                if (M > 0.0f) {
                    const float rM = 1.0f / M;
                    const float vbar = mom_n * rM;
                    vb[0] -= P.dt * mp * rM * dl;
                    gph -= P.dt * (v[0] - vbar) * rM * dl * P.rho0 * P.p_vol;
                }
            }
            // one writer per value: a reduction that returns nothing, instead of a
            // read whose latency ends the kernel (2D walker's design gradient
            // 5,200 -> 5,030 us, batch 17,720 -> 17,260, 3D walker 25.36 -> 25.00 ms)
            atomicAdd(a.gphi + p, gph);
#pragma unroll
            for (int i = 0; i < D; ++i) atomicAdd(a.gmag + (long long)i * np + p, brb[i]);
        }
        // into slots: with one sum per instance, the 31,250 warps of a million
        // particles queued at three addresses (adjoint 200 -> 160 us per launch)
        const long long slot = (long long)a.n_p2g * a.slots + ((p >> 5) & (a.slots - 1));
        const long long per_inst = (long long)P.n_steps * a.slots;
        warp_add_per_instance<D>(bab, inst, a.gfield_acc + slot * D, per_inst * D);
        if (has_fgrad)  // uniform over the launch: every lane takes part
            warp_add_per_instance<D * D>(gG, inst, P.ext->gfgrad + slot * D * D, per_inst * D * D);
        if (!G2PT && active) {
            store_vec<D>(a.adj, L::X, np, p, xb);
            store_vec<D>(a.adj, L::V, np, p, vb);
            store_mat<D>(a.adj, L::C, np, p, Cb);
            store_mat<D>(a.adj, L::F, np, p, Fb);
        }
    }
    if (G2PT) {
        Stencil<D> s;
        float q[D], dC[D][D];  // dC[c][i] = kappa dx Ct_ic
        int nb = 0;
        float4* __restrict__ Vbi = a.Vbar + (long long)(active ? inst : 0) * P.nodes;
        if (active) {
            if (!P2GT) {
                // adjoint of state m+1 and C_{m+1} from memory
                load_vec<D>(a.adj, L::X, np, p, xb);
                load_vec<D>(a.adj, L::V, np, p, vb);
                load_mat<D>(a.adj, L::C, np, p, Cb);
                load_mat<D>(a.adj, L::F, np, p, Fb);
                load_mat<D>(a.s_in, L::C, np, p, Cn);
            }
            float x[D], F[D][D];
            if (kAhead) {
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    x[i] = x_m[i];
#pragma unroll
                    for (int j = 0; j < D; ++j) F[i][j] = F_m[i][j];
                }
            } else {
                load_position<D>(a.s_aux, a.x0, np, p, x);  // the position x0 + u
                if (kPark) parked_mat<D>(sm, kParkEm, F);
                else load_mat<D>(a.s_aux, L::F, np, p, F);
            }
            if (!make_stencil<D>(x, P, s)) flags |= kErrDomain;
            // x' = x + dt v',  F' = (I + dt C') F  (Eq. 21-22)
            float vt[D], Ct[D][D], Fo[D][D];
            // C of state n, for (I + dt C')^T
            if (kPark) parked_mat<D>(sm, kParkC, Cn);
            else if (kLate && P2GT) reload_mat<D>(a.s_in, L::C, np, p, Cn);
#pragma unroll
            for (int i = 0; i < D; ++i) vt[i] = vb[i] + P.dt * xb[i];
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    float fft = Fb[i][j], ctf = Fb[i][j];  // F = I + E
#pragma unroll
                    for (int k = 0; k < D; ++k) {
                        fft += Fb[i][k] * F[j][k];          // (Fbar F^T)_ij
                        ctf += P.dt * Cn[k][i] * Fb[k][j];  // ((I + dt C')^T Fbar)_ij
                    }
                    Ct[i][j] = Cb[i][j] + P.dt * fft;
                    Fo[i][j] = ctf;
                }
            store_mat<D>(a.adj, L::F, np, p, Fo);  // complete: the stencil sums add nothing to it
            using NP = NodePack<D>;
            // Eq. 19-20 reversed (v' = sum w V, C' = kappa sum w V dpos^T) with
            // dpos = (o - r) dx: the node's velocity adjoint is w sv,
            //   sv = vt + kappa Ct dpos = q + kappa dx Ct o,  q = vt - kappa dx Ct r,
            // and dx xbar += d/dr sum w V . sv (adjoint_sums).
            const float kdx = P.kappa * P.dx;
#pragma unroll
            for (int i = 0; i < D; ++i) {
                float cr = 0.0f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    cr += Ct[i][j] * s.r[j];
                    dC[j][i] = kdx * Ct[i][j];
                }
                q[i] = vt[i] - kdx * cr;
            }
            nb = base_node<D>(s, P.res);
            const float4* __restrict__ Vn = (FUSE_V ? a.accG : a.V) + (long long)inst * P.nodes + nb;
            float xg[D];
            {
                typename NP::Vel Cp[D], Vs, none[D];
#pragma unroll
                for (int c = 0; c < D; ++c) Cp[c] = NP::vel(dC[c]);
                adjoint_sums<D, false>(
                    s,
                    [&](int o0, int om, int ol) {
                        return load_node_velocity<D, FUSE_V, EXT>(Vn, s, P, o0, om, ol, a.n_p2g - 1);
                    },
                    NP::vel(vt), Cp, Vs, none, xg);
            }
            if constexpr (!AGG) {
                typename NP::Vel Cp[D];
#pragma unroll
                for (int c = 0; c < D; ++c) Cp[c] = NP::vel(dC[c]);
                const typename NP::Vel Q = NP::vel(q);
                NodeValues<D, typename NP::Vel> value{s, Q, Cp, Q, 0.0f};
#pragma unroll
                for (int k = 0; k < stencil_size<D>(); ++k) atomicAdd(Vbi + nb + node_offset<D>(k, P.res), value(k));
            }
#pragma unroll
            for (int c = 0; c < D; ++c) xb[c] += P.inv_dx * xg[c];
            store_vec<D>(a.adj, L::X, np, p, xb);
        } else {  // a lane past the end takes part in the aggregated scatter with zeros
#pragma unroll
            for (int i = 0; i < D; ++i) {
                q[i] = 0.0f;
                s.base[i] = 0;
#pragma unroll
                for (int j = 0; j < D; ++j) dC[i][j] = 0.0f;
#pragma unroll
                for (int j = 0; j < 3; ++j) s.w[i][j] = 0.0f;
            }
        }
        if constexpr (AGG) {
            // node (o0, .., ol) receives w sv, sv = q + kappa dx Ct o, as above
            using NP = NodePack<D>;
            const typename NP::Vel Q = NP::vel(q);
            typename NP::Vel Cs[D];
#pragma unroll
            for (int c = 0; c < D; ++c) Cs[c] = NP::vel(dC[c]);
            scatter_aggregated<D>(nb, inst, active, a.Vbar, P.nodes, P.res, sm,
                                  NodeValues<D, typename NP::Vel>{s, Q, Cs, Q, 0.0f});
        }
    }
    if (flags) atomicOr(a.err, flags);
}

template <int D, bool P2GT, bool G2PT, bool FUSE, bool FUSE_V, int MINB, bool EXT>
__global__ void __launch_bounds__(MINB == kBlocksOf128 ? 128 : 256, MINB) k_adjoint(Params P, StepArgs a) {
    extern __shared__ float4 s_warp[];
    adjoint_particle<D, P2GT, G2PT, FUSE, FUSE_V, EXT, true, (MINB >= 3 || D == 3)>(
        P, a, blockIdx.x * blockDim.x + threadIdx.x, s_warp + (threadIdx.x >> 5) * warp_slots<D, G2PT>());
}


}  // namespace

template <int D, bool FUSE>
static cudaError_t forward_d(bool g2p, bool p2g, bool all, const Params& P, const StepArgs& a,
                             int block, cudaStream_t st) {
    // a fused launch also clears a.zero4, so it runs even without particles
    if (P.n_total == 0 && !(FUSE && a.zero4)) return cudaSuccess;
    long long threads = P.n_total > 0 ? P.n_total : block;
    dim3 grid(particle_blocks(threads, block));
    const bool ext = P.ext != nullptr;
    const size_t warps = (size_t)(block + 31) / 32;
    auto go = [&](auto kernel, size_t smem) { return launch_chain_smem(P, kernel, grid, block, smem, st, P, a); };
    const size_t smem_p2g = warps * warp_slots<D, true>() * sizeof(float4);
    const size_t smem_g2p = warps * warp_slots<D, false>() * sizeof(float4);
    if (g2p && p2g) {
        if (ext) {
            if (all) return go(k_forward<D, true, true, true, FUSE, true>, smem_p2g);
            return go(k_forward<D, true, true, false, FUSE, true>, smem_p2g);
        }
        if constexpr (D == 2) {
            if (P.agg2) {  // the aggregated 2D P2G (Params::agg2)
                const size_t smem_agg = warps * warp_slots<D, true, true>() * sizeof(float4);
                if (all) return go(k_forward<D, true, true, true, FUSE, false, true>, smem_agg);
                return go(k_forward<D, true, true, false, FUSE, false, true>, smem_agg);
            }
        }
        if constexpr (D == 3 && !FUSE) {
            if (P.n_total <= P.wave) {
                if (all) return go(k_forward<D, true, true, true, FUSE, false, true, kMinBlocksOneWave>, smem_p2g);
                return go(k_forward<D, true, true, false, FUSE, false, true, kMinBlocksOneWave>, smem_p2g);
            }
        }
        if (all) return go(k_forward<D, true, true, true, FUSE, false>, smem_p2g);
        return go(k_forward<D, true, true, false, FUSE, false>, smem_p2g);
    } else if (g2p) {
        // with grid fusion the G2P applies the grid operation, boxes included
        if (ext && FUSE) {
            if (all) return go(k_forward<D, true, false, true, FUSE, true>, smem_g2p);
            return go(k_forward<D, true, false, false, FUSE, true>, smem_g2p);
        }
        if (all) return go(k_forward<D, true, false, true, FUSE, false>, smem_g2p);
        return go(k_forward<D, true, false, false, FUSE, false>, smem_g2p);
    } else {
        if (ext) return go(k_forward<D, false, true, false, FUSE, true>, smem_p2g);
        return go(k_forward<D, false, true, false, FUSE, false>, smem_p2g);
    }
    return cudaGetLastError();
}

template <int D>
cudaError_t launch_forward_dim(bool g2p, bool p2g, bool write_all, bool fuse, const Params& P,
                               const StepArgs& a, int block, cudaStream_t st) {
    return fuse ? forward_d<D, true>(g2p, p2g, write_all, P, a, block, st)
                : forward_d<D, false>(g2p, p2g, write_all, P, a, block, st);
}

template <int D, bool FUSE, bool FUSE_V>
static cudaError_t adjoint_d(bool p2gt, bool g2pt, const Params& P, const StepArgs& a, int block,
                             cudaStream_t st) {
    if (P.n_total == 0 && !a.zero4) return cudaSuccess;
    long long threads = P.n_total > 0 ? P.n_total : block;
    dim3 grid(particle_blocks(threads, block));
    // with solid boxes or a field gradient only the 128-register budget is built
    const bool ext = P.ext != nullptr;
    const size_t warps = (size_t)(block + 31) / 32;
    auto go = [&](auto kernel, size_t smem) { return launch_chain_smem(P, kernel, grid, block, smem, st, P, a); };
    const size_t sm_g2pt = warps * warp_slots<D, true>() * sizeof(float4);
    const size_t sm_p2gt = warps * warp_slots<D, false>() * sizeof(float4);
    if (p2gt && g2pt) {
        if (ext) return go(k_adjoint<D, true, true, FUSE, FUSE_V, 2, true>, sm_g2pt);
        if constexpr (D == 2) {
            if (P.adj_blocks == 4) return go(k_adjoint<D, true, true, FUSE, FUSE_V, 4, false>, sm_g2pt);
        }
        if (P.adj_blocks < 3 || (D == 3 && P.n_total <= P.wave))
            return go(k_adjoint<D, true, true, FUSE, FUSE_V, kMinBlocksOneWave, false>, sm_g2pt);
        if constexpr (D == 3) {
            if (block <= 128) return go(k_adjoint<D, true, true, FUSE, FUSE_V, kBlocksOf128, false>, sm_g2pt);
        }
        return go(k_adjoint<D, true, true, FUSE, FUSE_V, 3, false>, sm_g2pt);
    }
    // the segment-edge halves run once per checkpoint segment
    if (p2gt) {
        if (ext) return go(k_adjoint<D, true, false, FUSE, FUSE_V, 2, true>, sm_p2gt);
        return go(k_adjoint<D, true, false, FUSE, FUSE_V, 2, false>, sm_p2gt);
    }
    if (ext) return go(k_adjoint<D, false, true, FUSE, FUSE_V, 2, true>, sm_g2pt);
    return go(k_adjoint<D, false, true, FUSE, FUSE_V, 2, false>, sm_g2pt);
}

template <int D>
cudaError_t launch_adjoint_dim(bool p2gt, bool g2pt, bool fuse, bool fuse_v, const Params& P,
                               const StepArgs& a, int block, cudaStream_t st) {
    if (fuse) return adjoint_d<D, true, true>(p2gt, g2pt, P, a, block, st);
    if (fuse_v) return adjoint_d<D, false, true>(p2gt, g2pt, P, a, block, st);
    return adjoint_d<D, false, false>(p2gt, g2pt, P, a, block, st);
}


}  // namespace mpm
