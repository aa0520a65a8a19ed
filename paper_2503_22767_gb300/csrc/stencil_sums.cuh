// Stencil sums of node values, axis by axis (the gathers of the transfer
// kernels).
//
// The quadratic B-spline weights of one axis, with t = r - 1 in [-1/2, 1/2)
// and the three node values f0, f1, f2 taken as f1, D = f2 - f0 and
// Q = f0 - 2 f1 + f2, give
//   sum w f          = f1 + (t/2) D + (1/8 + t^2/2) Q
//   sum w (o - r) f  = (D + t (3 - 4 t^2) Q) / 8        (o the node's offset)
// so the centred moment (the affine matrix C of Eq. 20) comes from node
// differences, without the subtraction of two large sums.  A row along the
// last axis takes this form; across rows and planes the sums run with the
// axis' weights.  Node values are packed pairs (packed.cuh): the kernels are
// bound by instruction issue.
#pragma once

#include "mpm_device.cuh"
#include "packed.cuh"

namespace mpm {

// s x - y
__device__ __forceinline__ Pack2 psub(const Pack2& x, const Pack2& y) { return pfma(dup2(-1.0f), y, x); }
__device__ __forceinline__ Pack3 psub(const Pack3& x, const Pack3& y) { return pfma(dup2(-1.0f), y, x); }
__device__ __forceinline__ Pack4 psub(const Pack4& x, const Pack4& y) { return pfma(dup2(-1.0f), y, x); }

// v = sum w V, M[a] = sum w (o - r)_a V over the stencil; the last axis'
// moment comes out times 8.  load(o0, om, ol) gives the velocity of the node
// at that offset (2D: o0 is 0 and the offset is (om, ol)).
template <int D, typename Load>
__device__ __forceinline__ void gather_velocity(const Stencil<D>& s, Load load, typename NodePack<D>::Vel& v,
                                                typename NodePack<D>::Vel (&M)[D]) {
    using Vel = typename NodePack<D>::Vel;
    constexpr int A1 = D - 2, L = D - 1;
    const float t = s.r[L] - 1.0f;
    const float2 ht = dup2(0.5f * t), al = dup2(0.125f + 0.5f * t * t), b8 = dup2(t * (3.0f - 4.0f * t * t));
#pragma unroll
    for (int o0 = 0; o0 < (D == 3 ? 3 : 1); ++o0) {
        Vel h, m1, m8;  // sums over the rows of this plane
#pragma unroll
        for (int om = 0; om < 3; ++om) {
            const Vel f0 = load(o0, om, 0), f1 = load(o0, om, 1), f2 = load(o0, om, 2);
            const Vel d = psub(f2, f0), q = pfma(dup2(-2.0f), f1, padd(f0, f2));
            const Vel r = pfma(al, q, pfma(ht, d, f1)), rm = pfma(b8, q, d);
            const float2 w = dup2(s.w[A1][om]), wm = dup2(s.w[A1][om] * ((float)om - s.r[A1]));
            h = om == 0 ? pmul(w, r) : pfma(w, r, h);
            m1 = om == 0 ? pmul(wm, r) : pfma(wm, r, m1);
            m8 = om == 0 ? pmul(w, rm) : pfma(w, rm, m8);
        }
        if constexpr (D == 3) {
            const float2 w = dup2(s.w[0][o0]), wm = dup2(s.w[0][o0] * ((float)o0 - s.r[0]));
            v = o0 == 0 ? pmul(w, h) : pfma(w, h, v);
            M[0] = o0 == 0 ? pmul(wm, h) : pfma(wm, h, M[0]);
            M[1] = o0 == 0 ? pmul(w, m1) : pfma(w, m1, M[1]);
            M[2] = o0 == 0 ? pmul(w, m8) : pfma(w, m8, M[2]);
        } else {
            v = h;
            M[0] = m1;
            M[1] = m8;
        }
    }
}

}  // namespace mpm
