// FP32 bounds of the HOLD pair step (tau_pair in hold_pair.cuh): lo <= tau <= hi
// for every pair, from about 70 FP32 instructions.
//
// Positions and velocities are pairs of floats (hi + lo, 48 bits), so a
// difference keeps a relative error of 2^-22 as a vector as long as its length is
// above 2^-20 of the body's own largest coordinate. With it and approximate
// reciprocals and roots (relative error 2^-22 each),
//   t_ff = eta sqrt(r^3 / gm) and t_fl = eta r / v      have a relative error below 2^-18;
//   cos = r.v / (r v)                                    an absolute error below 2^-19;
//   d_ff = 1.5 T cos, T = t_ff v / r                     below 1.5 T 2^-17.4;
//   d_fl = eta S cos, S = 1 + gm / (r v^2)               below eta S 2^-18,
// both capped at 1, so D = 1 - d/2 >= 1/2 has a relative error below 0.75 T 2^-17.4 / D
// and eta S 2^-19 / D. The bounds take K (1 + T / D) and K (1 + eta S / D) with
// K = 2^-16 as the relative errors of t / D. For bodies of equal velocity (a cluster
// starting from rest), which the caller compares, t_ff alone counts and d_ff = 0. Outside
// the ranges that keep every intermediate a normal number, and for differences too
// close to cancel, the pair gets lo = -1 and hi = infinity: it is always evaluated
// exactly. The ranges are those of units in which lengths, masses times G and with them
// speeds are of order 1 up to powers of the number of bodies (PairBody32::scale).
#pragma once

#include <cuda_runtime.h>

namespace gbfmm {

struct PairBody32 {
    float4 a, b, c;  // xh xl yh yl | zh zl uh ul | vh vl wh wl
    float m;
    __device__ __forceinline__ PairBody32() {}
    __device__ __forceinline__ PairBody32(double x, double y, double z, double u, double v, double w, double mass) {
        a.x = (float)x; a.y = (float)(x - (double)a.x);
        a.z = (float)y; a.w = (float)(y - (double)a.z);
        b.x = (float)z; b.y = (float)(z - (double)b.x);
        b.z = (float)u; b.w = (float)(u - (double)b.z);
        c.x = (float)v; c.y = (float)(v - (double)c.x);
        c.z = (float)w; c.w = (float)(w - (double)c.z);
        m = (float)mass;
    }
    // to other units: lengths, speeds by powers of two, masses by any factor (t = eta r / v and
    // t^2 = eta^2 r^3 / (G m) keep their order in units of length L, speed V and mass L V^2)
    __device__ __forceinline__ void scale(float l, float v, float g) {
        a.x *= l; a.y *= l; a.z *= l; a.w *= l; b.x *= l; b.y *= l;
        b.z *= v; b.w *= v; c.x *= v; c.y *= v; c.z *= v; c.w *= v;
        m *= g;
    }
};

// the body's own constants: the smallest squared distance and speed that its
// coordinates leave accurate, G and eta
struct PairScale32 {
    float r2min, v2min, G, eta;
    bool ok;
    __device__ __forceinline__ PairScale32(const PairBody32& s, double Gd, double etad) {
        const float x = fmaxf(fabsf(s.a.x), fmaxf(fabsf(s.a.z), fabsf(s.b.x))) * 0x1p-20f;
        const float v = fmaxf(fabsf(s.b.z), fmaxf(fabsf(s.c.x), fabsf(s.c.z))) * 0x1p-20f;
        r2min = fmaxf(0x1p-60f, x * x);
        v2min = fmaxf(0x1p-60f, v * v);
        G = (float)Gd;
        eta = (float)etad;
        ok = eta > 0x1p-20f && eta < 0x1p10f;
    }
};

// equal numbers, by integer tests (an FP64 comparison would cost an FP64 instruction)
__device__ __forceinline__ bool same_number(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return x == y || (x | y) << 1 == 0;  // (zeros of either sign)
}

// same_velocity(): whether the bodies' FP64 velocities are equal; asked only where the difference is
// too close to cancel.
template <typename Same>
__device__ __forceinline__ void pair_bounds32(const PairBody32& p, const PairBody32& q, const PairScale32& s, bool sym,
                                              Same same_velocity, float& lo, float& hi) {
    constexpr float K = 0x1p-16f;
    const float dx = (q.a.x - p.a.x) + (q.a.y - p.a.y), dy = (q.a.z - p.a.z) + (q.a.w - p.a.w),
                dz = (q.b.x - p.b.x) + (q.b.y - p.b.y);
    const float ux = (q.b.z - p.b.z) + (q.b.w - p.b.w), uy = (q.c.x - p.c.x) + (q.c.y - p.c.y),
                uz = (q.c.z - p.c.z) + (q.c.w - p.c.w);
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz)), v2 = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
    const float gm = s.G * (p.m + q.m);
    const bool ok = s.ok && r2 >= s.r2min && r2 <= 0x1p40f && gm >= 0x1p-60f && gm <= 0x1p20f;
    const bool moving = v2 >= s.v2min && v2 <= 0x1p60f;
    const float ir = rsqrtf(r2), iv = rsqrtf(v2), r = r2 * ir;
    const float c = r2 * r * __fdividef(1.0f, gm);
    const float tff = s.eta * (c * rsqrtf(c)), tfl = s.eta * r * iv;
    float aff = tff, afl = tfl, kff = K, kfl = K;
    if (sym) {
        const float cosv = fmaf(dx, ux, fmaf(dy, uy, dz * uz)) * ir * iv;
        const float T = tff * ir * (v2 * iv), S = s.eta * (1.0f + gm * ir * (iv * iv));
        const float iff = __fdividef(1.0f, 1.0f - 0.5f * fminf(1.5f * T * cosv, 1.0f));
        const float ifl = __fdividef(1.0f, 1.0f - 0.5f * fminf(S * cosv, 1.0f));
        aff = tff * iff;
        afl = tfl * ifl;
        kff = fmaf(K * T, iff, K);
        kfl = fmaf(K * S, ifl, K);
    }
    // a (1 - k) <= a / (1 + k) and, for k <= 1/4, a / (1 - k) <= a (1 + 2 k)
    lo = fminf(aff * (1.0f - kff), afl * (1.0f - kfl));
    const float hff = kff <= 0.25f ? aff * fmaf(2.0f, kff, 1.0f) : __int_as_float(0x7f800000);
    const float hfl = kfl <= 0.25f ? afl * fmaf(2.0f, kfl, 1.0f) : __int_as_float(0x7f800000);
    hi = fminf(hff, hfl);
    // (a NaN bound fails the comparison and counts as out of range)
    if (!(ok && moving && kff < 1e30f && kfl < 1e30f && hi > 0.0f)) {
        const bool rest = ok && v2 < s.v2min && same_velocity();
        lo = rest ? tff * (1.0f - K) : -1.0f;
        hi = rest ? tff * (1.0f + 2.0f * K) : __int_as_float(0x7f800000);
    }
}

}  // namespace gbfmm
