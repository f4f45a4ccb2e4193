// Per-pixel arithmetic of compositing, shared by the compositor's two forms so
// that a pixel's value does not depend on which of them renders it.
#pragma once

#include "gs_internal.cuh"

namespace gsb {

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// A 16-byte copy from global to shared memory that the thread waits for later.
__device__ __forceinline__ void copy16(float4* dst, const float4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// One pixel's blend step for a splat whose alpha is `al` (already >= 1/255);
// returns the weight w = alpha T added (0 when the step stops instead):
// T' = T (1 - alpha), evaluated as T - w; stop (splat not added) when
// T' < 1e-4.  The arithmetic is pinned to explicit round-to-nearest operations
// so every tile shape and every pixel slot evaluates exactly the same.
__device__ __forceinline__ float blend(float al, const float4& C, float z, float& T, float& r, float& g, float& b,
                                       float& d, bool& done) {
    const float w = __fmul_rn(al, T);
    const float Tn = __fsub_rn(T, w);
    if (Tn < 1e-4f) {
        done = true;
        return 0.0f;
    }
    r = __fmaf_rn(w, C.x, r);
    g = __fmaf_rn(w, C.y, g);
    b = __fmaf_rn(w, C.z, b);
    d = __fmaf_rn(w, z, d);
    T = Tn;
    return w;
}

// alpha = min(0.99, o exp(-q/2)) = min(0.99, 2^(log2 o - (l00 dx + l01 dy)^2 - (l11 dy)^2))
// where B = (l00, l01, l11) is the conic's upper Cholesky factor scaled by
// sqrt(log2(e)/2): q is evaluated as a sum of two squares.  Evaluated at a
// lane's two pixel centres (fpx, fpy.x) and (fpx, fpy.y) with the paired FP32
// instructions of sm_100+ (two round-to-nearest operations per instruction).
// CLAMP = false leaves out the 0.99 cap, for splats of opacity <= 0.98 (their
// alpha stays below it).
template <bool CLAMP = true>
__device__ __forceinline__ float2 splat_alpha2(const float4& A, const float4& B, float fpx, float2 fpy) {
    const float dx = fpx - A.x;
    const float2 dy = __fadd2_rn(fpy, make_float2(-A.y, -A.y));
    const float bx = __fmul_rn(B.x, dx);
    const float2 t = __ffma2_rn(make_float2(B.y, B.y), dy, make_float2(bx, bx));
    const float2 s = __fmul2_rn(make_float2(B.z, B.z), dy);
    // camera splats are staged with A.z = log2(o), folded into the exponent:
    // alpha = 2^(log2 o - t^2 - s^2), two paired FMAs before the ex2
    const float2 pw =
        __ffma2_rn(make_float2(-t.x, -t.y), t, __ffma2_rn(make_float2(-s.x, -s.y), s, make_float2(A.z, A.z)));
    const float2 a = make_float2(ex2_approx(pw.x), ex2_approx(pw.y));
    if constexpr (!CLAMP) return a;
    return make_float2(fminf(0.99f, a.x), fminf(0.99f, a.y));
}

// blend() for a lane's two pixels at once: pixel k takes the splat where uk
// is set.  A pixel that does not take it keeps its state exactly (its weight
// is 0, and fma(0, c, x) = x for the finite, non-negative sums here).  Returns
// the sum of the two weights added.
__device__ __forceinline__ float blend2(float2 al, bool u0, bool u1, const float4& C, float z, float2& T, float2& r,
                                        float2& g, float2& b, float2& d, bool& done0, bool& done1) {
    const float2 am = make_float2(u0 ? al.x : 0.0f, u1 ? al.y : 0.0f);
    const float2 x = __fmul2_rn(am, T);
    const float2 Tn = __fadd2_rn(T, make_float2(-x.x, -x.y));
    const bool s0 = u0 && Tn.x < 1e-4f, s1 = u1 && Tn.y < 1e-4f;
    done0 = done0 || s0;
    done1 = done1 || s1;
    const float2 w = make_float2(s0 ? 0.0f : x.x, s1 ? 0.0f : x.y);
    r = __ffma2_rn(w, make_float2(C.x, C.x), r);
    g = __ffma2_rn(w, make_float2(C.y, C.y), g);
    b = __ffma2_rn(w, make_float2(C.z, C.z), b);
    d = __ffma2_rn(w, make_float2(z, z), d);
    T = make_float2(s0 ? T.x : Tn.x, s1 ? T.y : Tn.y);
    return w.x + w.y;
}

// Whether a splat can reach alpha >= 1/255 at any pixel centre of the 8x8
// subtile whose first centre is (x0, y0): the minimum of its quadratic form
// q = (l00 dx + l01 dy)^2 + (l11 dy)^2 over the rectangle spanned by the
// centres, against log2(255 o) (B.w).  q is convex, so with the splat centre
// outside the rectangle the minimum lies on an edge, where it is the clamped
// stationary point of a 1D quadratic.  The test only skips splats that no
// pixel of the subtile blends: it keeps a relative margin of 1e-3 plus 1e-3
// on the threshold, far above the rounding of q here and in the blend loop.
__device__ __forceinline__ bool reaches_rect(const float4& A, const float4& B, float x0, float y0) {
    const float ax = x0 - A.x, bx = ax + 7.0f;  // dx range
    const float ay = y0 - A.y, by = ay + 7.0f;  // dy range
    if (ax <= 0.0f && bx >= 0.0f && ay <= 0.0f && by >= 0.0f) return true;
    const float l00 = B.x, l01 = B.y, l11 = B.z;
    auto q = [&](float dx, float dy) {
        const float t = fmaf(l01, dy, l00 * dx);
        const float u = l11 * dy;
        return fmaf(t, t, u * u);
    };
    // vertical edges dx = const: stationary dy = -l00 l01 dx / (l01^2 + l11^2);
    // horizontal edges dy = const: stationary dx = -l01 dy / l00.  Fast
    // divisions: q is evaluated exactly at whatever point is used, and a
    // stationary point off by a few ulp raises q only to second order.
    const float kv = __fdividef(-l00 * l01, fmaf(l01, l01, l11 * l11));
    const float kh = __fdividef(-l01, l00);
    const float q1 = q(ax, fminf(fmaxf(kv * ax, ay), by));
    const float q2 = q(bx, fminf(fmaxf(kv * bx, ay), by));
    const float q3 = q(fminf(fmaxf(kh * ay, ax), bx), ay);
    const float q4 = q(fminf(fmaxf(kh * by, ax), bx), by);
    const float qmin = fminf(fminf(q1, q2), fminf(q3, q4));
    return qmin <= fmaf(B.w, 1.001f, 1e-3f);
}

// Stores one camera pixel: the float image, or the observation form (rgb8 /
// depth16), where the clamped colour goes through the env's appearance
// transform (exposure gain 2^e, contrast c about 0.5, brightness offset b), is
// clamped again and rounded to 8 bits, and depth is rounded to half precision.
struct PixelStore {
    float gain = 1.0f, con = 1.0f, bri = 0.0f;
    __device__ __forceinline__ PixelStore(const CompParams& P, int el) {
        if (P.rgb8 && P.appear) {
            const gs_appearance ap = P.appear[el];
            gain = exp2f(ap.exposure);
            con = ap.contrast;
            bri = ap.brightness;
        }
    }
    __device__ __forceinline__ void put(const CompParams& P, size_t pix, float T, float r, float g, float b,
                                        float d) const {
        const float cr = fminf(fmaxf(r, 0.0f), 1.0f), cg = fminf(fmaxf(g, 0.0f), 1.0f),
                    cb = fminf(fmaxf(b, 0.0f), 1.0f);
        const float a = 1.0f - T;
        const float dep = a > 0.0f ? d / a : 0.0f;
        if (P.rgb8) {
            auto q = [&](float v) {
                // no appearance given: the identity, exactly ((v - 0.5) + 0.5 would round)
                if (P.appear) v = fmaf(fmaf(v, gain, -0.5f), con, 0.5f + bri);
                return (uint8_t)__float2int_rn(fminf(fmaxf(v, 0.0f), 1.0f) * 255.0f);
            };
            P.rgb8[3 * pix] = q(cr);
            P.rgb8[3 * pix + 1] = q(cg);
            P.rgb8[3 * pix + 2] = q(cb);
        } else {
            P.rgb[3 * pix] = cr;
            P.rgb[3 * pix + 1] = cg;
            P.rgb[3 * pix + 2] = cb;
        }
        if (P.depth16) P.depth16[pix] = __half_as_ushort(__float2half_rn(dep));
        else if (P.depth) P.depth[pix] = dep;
        if (P.alpha) P.alpha[pix] = a;
    }
};

}  // namespace gsb
