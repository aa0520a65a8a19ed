// Stencil sums of node values, axis by axis (the gathers of the transfer
// kernels).
//
// The quadratic B-spline weights of one axis, with t = r - 1 in [-1/2, 1/2)
// and the three node values f0, f1, f2 taken as f1, D = f2 - f0 and
// Q = f0 - 2 f1 + f2, give
//   sum w f          = f1 + (t/2) D + (1/8 + t^2/2) Q
//   sum w (o - r) f  = (D + t (3 - 4 t^2) Q) / 8        (o the node's offset)
//   sum w' f         = (D + 2 t Q) / 2                  (' = d/dr)
//   (sum w (o - r) f)' = (3/8 - 3 t^2/2) Q
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

// The sums of a transfer's reverse.  The node values f are contracted with
// the field U + sum_a (o - r)_a A[a] that the forward transfer spreads (f .
// field at the node: the objective's sensitivity to the node's weight), and
//   S = sum w f,   T[a] = sum w (o - r)_a f   (MASS; the last axis' moment
//                                              comes out times 8)
//   xg[a] = d/dr_a sum w f . (U + sum_b (o - r)_b A[b])
// come out.  load(o0, om, ol) as in gather_velocity, packed like U.  MASS: f
// and U hold mass and momentum, A and T momentum; else all are velocities.
//
// In the 3D adjoint kernel (80 registers, latency-bound, 55-60% issue) this
// took the launch from 115.5 to 104.6 M warp instructions and from 158.0 to
// 153.3 us per 1,000,000 particles (ncu) against scalar sums with one
// contraction per node; a rolled plane loop (less code, 248 instead of 208
// bytes of spill loads) gave 1% back.
template <int D, bool MASS, typename V, typename M, typename Load>
__device__ __forceinline__ void adjoint_sums(const Stencil<D>& s, Load load, const V& U, const M (&A)[D], V& S,
                                             M (&T)[D], float (&xg)[D]) {
    constexpr int A1 = D - 2, L = D - 1;
    const float t = s.r[L] - 1.0f;
    const float2 ht = dup2(0.5f * t), al = dup2(0.125f + 0.5f * t * t), b8 = dup2(t * (3.0f - 4.0f * t * t)),
                 t2 = dup2(2.0f * t);
    // the field at o = 0 of every axis but the last, and what the last axis adds
    V U0 = pfma(dup2(-s.r[A1]), A[A1], U);
    if (D == 3) U0 = pfma(dup2(-s.r[0]), A[0], U0);
    auto part = [](const V& x) {
        if constexpr (MASS) return NodePack<D>::mom(x);
        else return x;
    };
    const M A8 = pmul(dup2(0.125f), A[L]), Ag = pmul(dup2(0.75f - 3.0f * t * t), A[L]);
#pragma unroll
    for (int o0 = 0; o0 < (D == 3 ? 3 : 1); ++o0) {
        V Ur = U0, h;
        M m1, m8;  // the row's field; sums over the rows of this plane
        float la, lb, lc;
#pragma unroll
        for (int om = 0; om < 3; ++om) {
            if (om > 0) Ur = padd(Ur, A[A1]);
            const V f0 = load(o0, om, 0), f1 = load(o0, om, 1), f2 = load(o0, om, 2);
            const V d = psub(f2, f0), q = pfma(dup2(-2.0f), f1, padd(f0, f2));
            const V r = pfma(al, q, pfma(ht, d, f1)), rd = pfma(t2, q, d);
            const M rm = pfma(b8, part(q), part(d));
            const float ha = pdot2(Ur, r, A8, rm), hb = pdot2(Ur, rd, Ag, part(q));  // hb: twice the derivative
            const float w = s.w[A1][om], dw = s.dw[A1][om], wm = w * ((float)om - s.r[A1]);
            h = om == 0 ? pmul(dup2(w), r) : pfma(dup2(w), r, h);
            if (MASS) {
                m1 = om == 0 ? pmul(dup2(wm), part(r)) : pfma(dup2(wm), part(r), m1);
                m8 = om == 0 ? pmul(dup2(w), rm) : pfma(dup2(w), rm, m8);
            }
            la = om == 0 ? w * ha : fmaf(w, ha, la);
            lb = om == 0 ? dw * ha : fmaf(dw, ha, lb);
            lc = om == 0 ? w * hb : fmaf(w, hb, lc);
        }
        if constexpr (D == 3) {
            const float w = s.w[0][o0], dw = s.dw[0][o0], wm = w * ((float)o0 - s.r[0]);
            S = o0 == 0 ? pmul(dup2(w), h) : pfma(dup2(w), h, S);
            if (MASS) {
                T[0] = o0 == 0 ? pmul(dup2(wm), part(h)) : pfma(dup2(wm), part(h), T[0]);
                T[1] = o0 == 0 ? pmul(dup2(w), m1) : pfma(dup2(w), m1, T[1]);
                T[2] = o0 == 0 ? pmul(dup2(w), m8) : pfma(dup2(w), m8, T[2]);
            }
            xg[0] = o0 == 0 ? dw * la : fmaf(dw, la, xg[0]);
            xg[1] = o0 == 0 ? w * lb : fmaf(w, lb, xg[1]);
            xg[2] = o0 == 0 ? w * lc : fmaf(w, lc, xg[2]);
            if (o0 < 2) U0 = padd(U0, A[0]);
        } else {
            S = h;
            if (MASS) {
                T[0] = m1;
                T[1] = m8;
            }
            xg[0] = lb;
            xg[1] = lc;
        }
    }
    // d(o - r)/dr of the axes summed with their weights' derivatives
    xg[A1] -= pdot(A[A1], part(S));
    if (D == 3) xg[0] -= pdot(A[0], part(S));
    xg[L] *= 0.5f;
}

}  // namespace mpm
