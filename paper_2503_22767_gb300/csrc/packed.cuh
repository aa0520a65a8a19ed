// Packed float32 vectors of the stencil sums.
//
// sm_103a issues two float32 FMAs in one instruction (fma.rn.f32x2, at half
// the issue rate of the scalar FMA: the same arithmetic rate for half the
// issue slots), and the transfer kernels are bound by instruction issue.  So
// the node values of a stencil (a float4 from memory: (v, 0) or (m, m v)) are
// summed as register pairs.  Each component is rounded as the scalar
// operation rounds it.
#pragma once

#include <cuda_runtime.h>

namespace mpm {

__device__ __forceinline__ float2 dup2(float s) { return make_float2(s, s); }

// One pair, a pair and a scalar, two pairs: the vectors of 2 (2D velocity),
// 3 (3D velocity; 2D mass and momentum) and 4 (3D mass and momentum) floats.
struct Pack2 {
    float2 a;
};
struct Pack3 {
    float2 a;
    float b;
};
struct Pack4 {
    float2 a, b;
};

// the momentum part of a Pack4, in place
struct Pack12 {
    float a;
    float2 b;
};

__device__ __forceinline__ Pack12 pmul(float2 s, const Pack12& x) { return {s.x * x.a, __fmul2_rn(s, x.b)}; }
__device__ __forceinline__ Pack12 pfma(float2 s, const Pack12& x, const Pack12& y) {
    return {fmaf(s.x, x.a, y.a), __ffma2_rn(s, x.b, y.b)};
}
__device__ __forceinline__ float pdot(const Pack12& x, const Pack12& y) {
    const float2 t = __fmul2_rn(x.b, y.b);
    return t.x + fmaf(x.a, y.a, t.y);
}

__device__ __forceinline__ Pack2 padd(const Pack2& x, const Pack2& y) { return {__fadd2_rn(x.a, y.a)}; }
__device__ __forceinline__ Pack3 padd(const Pack3& x, const Pack3& y) {
    return {__fadd2_rn(x.a, y.a), __fadd_rn(x.b, y.b)};
}
__device__ __forceinline__ Pack4 padd(const Pack4& x, const Pack4& y) {
    return {__fadd2_rn(x.a, y.a), __fadd2_rn(x.b, y.b)};
}

// s x, with s in both halves of the pair
__device__ __forceinline__ Pack2 pmul(float2 s, const Pack2& x) { return {__fmul2_rn(s, x.a)}; }
__device__ __forceinline__ Pack3 pmul(float2 s, const Pack3& x) { return {__fmul2_rn(s, x.a), s.x * x.b}; }
__device__ __forceinline__ Pack4 pmul(float2 s, const Pack4& x) { return {__fmul2_rn(s, x.a), __fmul2_rn(s, x.b)}; }

// s x + y
__device__ __forceinline__ Pack2 pfma(float2 s, const Pack2& x, const Pack2& y) { return {__ffma2_rn(s, x.a, y.a)}; }
__device__ __forceinline__ Pack3 pfma(float2 s, const Pack3& x, const Pack3& y) {
    return {__ffma2_rn(s, x.a, y.a), fmaf(s.x, x.b, y.b)};
}
__device__ __forceinline__ Pack4 pfma(float2 s, const Pack4& x, const Pack4& y) {
    return {__ffma2_rn(s, x.a, y.a), __ffma2_rn(s, x.b, y.b)};
}

// x . y
__device__ __forceinline__ float pdot(const Pack2& x, const Pack2& y) {
    const float2 t = __fmul2_rn(x.a, y.a);
    return t.x + t.y;
}
__device__ __forceinline__ float pdot(const Pack3& x, const Pack3& y) {
    const float2 t = __fmul2_rn(x.a, y.a);
    return t.x + fmaf(x.b, y.b, t.y);
}
__device__ __forceinline__ float pdot(const Pack4& x, const Pack4& y) {
    const float2 t = __ffma2_rn(x.b, y.b, __fmul2_rn(x.a, y.a));
    return t.x + t.y;
}

// x . y + z . w
__device__ __forceinline__ float pdot2(const Pack2& x, const Pack2& y, const Pack2& z, const Pack2& w) {
    const float2 t = __ffma2_rn(z.a, w.a, __fmul2_rn(x.a, y.a));
    return t.x + t.y;
}
__device__ __forceinline__ float pdot2(const Pack3& x, const Pack3& y, const Pack3& z, const Pack3& w) {
    const float2 t = __ffma2_rn(z.a, w.a, __fmul2_rn(x.a, y.a));
    return t.x + fmaf(z.b, w.b, fmaf(x.b, y.b, t.y));
}
__device__ __forceinline__ float pdot2(const Pack4& x, const Pack4& y, const Pack4& z, const Pack4& w) {
    float2 t = __ffma2_rn(z.a, w.a, __fmul2_rn(x.a, y.a));
    t = __ffma2_rn(z.b, w.b, __ffma2_rn(x.b, y.b, t));
    return t.x + t.y;
}

// a Pack4 with a momentum part: x + (0, y), s (0, y) + x, x . y + (0, z) . w
__device__ __forceinline__ Pack4 padd(const Pack4& x, const Pack12& y) {
    return {make_float2(x.a.x, x.a.y + y.a), __fadd2_rn(x.b, y.b)};
}
__device__ __forceinline__ Pack4 pfma(float2 s, const Pack12& y, const Pack4& x) {
    return {make_float2(x.a.x, fmaf(s.x, y.a, x.a.y)), __ffma2_rn(s, y.b, x.b)};
}
__device__ __forceinline__ float pdot2(const Pack4& x, const Pack4& y, const Pack12& z, const Pack12& w) {
    float2 t = __fmul2_rn(x.a, y.a);
    t.y = fmaf(z.a, w.a, t.y);
    t = __ffma2_rn(z.b, w.b, __ffma2_rn(x.b, y.b, t));
    return t.x + t.y;
}

// Node velocities (v, 0) and node mass and momentum (m, m v) per dimension.
template <int D>
struct NodePack;

template <>
struct NodePack<2> {
    using Vel = Pack2;
    using Mass = Pack3;
    // the momentum part: in 2D with the mass in its place (0 in slopes; with it
    // taken out, the 64-register adjoint spilled and lost 2%)
    using Mom = Mass;
    static __device__ __forceinline__ Mom mom(const Mass& x) { return x; }
    static __device__ __forceinline__ Mom mom(const float (&v)[2]) { return {make_float2(0.0f, v[0]), v[1]}; }
    static __device__ __forceinline__ void get_mom(const Mom& x, float (&v)[2]) { v[0] = x.a.y, v[1] = x.b; }
    static __device__ __forceinline__ Vel vel(const float4& g) { return {make_float2(g.x, g.y)}; }
    static __device__ __forceinline__ Vel vel(const float (&v)[2]) { return {make_float2(v[0], v[1])}; }
    static __device__ __forceinline__ Mass mass(const float4& g) { return {make_float2(g.x, g.y), g.z}; }
    static __device__ __forceinline__ Mass mass(float m, const float (&v)[2]) { return {make_float2(m, v[0]), v[1]}; }
    static __device__ __forceinline__ float4 node(const Vel& x) { return make_float4(x.a.x, x.a.y, 0.0f, 0.0f); }
    static __device__ __forceinline__ float4 node(const Mass& x) { return make_float4(x.a.x, x.a.y, x.b, 0.0f); }
    static __device__ __forceinline__ void get(const Vel& x, float (&v)[2]) { v[0] = x.a.x, v[1] = x.a.y; }
    static __device__ __forceinline__ void get(const Mass& x, float& m, float (&v)[2]) {
        m = x.a.x, v[0] = x.a.y, v[1] = x.b;
    }
};

template <>
struct NodePack<3> {
    using Vel = Pack3;
    using Mass = Pack4;
    using Mom = Pack12;
    static __device__ __forceinline__ Mom mom(const Mass& x) { return {x.a.y, x.b}; }
    static __device__ __forceinline__ Mom mom(const float (&v)[3]) { return {v[0], make_float2(v[1], v[2])}; }
    static __device__ __forceinline__ void get_mom(const Mom& x, float (&v)[3]) { v[0] = x.a, v[1] = x.b.x, v[2] = x.b.y; }
    static __device__ __forceinline__ Vel vel(const float4& g) { return {make_float2(g.x, g.y), g.z}; }
    static __device__ __forceinline__ Vel vel(const float (&v)[3]) { return {make_float2(v[0], v[1]), v[2]}; }
    static __device__ __forceinline__ Mass mass(const float4& g) { return {make_float2(g.x, g.y), make_float2(g.z, g.w)}; }
    static __device__ __forceinline__ Mass mass(float m, const float (&v)[3]) {
        return {make_float2(m, v[0]), make_float2(v[1], v[2])};
    }
    static __device__ __forceinline__ float4 node(const Vel& x) { return make_float4(x.a.x, x.a.y, x.b, 0.0f); }
    static __device__ __forceinline__ float4 node(const Mass& x) { return make_float4(x.a.x, x.a.y, x.b.x, x.b.y); }
    static __device__ __forceinline__ void get(const Vel& x, float (&v)[3]) { v[0] = x.a.x, v[1] = x.a.y, v[2] = x.b; }
    static __device__ __forceinline__ void get(const Mass& x, float& m, float (&v)[3]) {
        m = x.a.x, v[0] = x.a.y, v[1] = x.b.x, v[2] = x.b.y;
    }
};

}  // namespace mpm
