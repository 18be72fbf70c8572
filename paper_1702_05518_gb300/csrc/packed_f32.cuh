// packed_f32.cuh -- Blackwell's two-lane FP32 arithmetic (add/sub/mul/fma .rn.f32x2: one instruction
// per pair, each lane rounded as the scalar operation would be) and the Box-Muller pairs of a
// Philox block in it.
#pragma once

#include <cstdint>

#include "gmrf_device.cuh"

namespace gmrf {

// Two FP32 values (low half: the even chain) in one 64-bit register.
using f2 = unsigned long long;

__device__ __forceinline__ f2 pk(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// a * b + c, rounded once per lane
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Four chain values (two pairs) at p, 16-byte aligned.
__device__ __forceinline__ void ld2x2(const float *p, f2 &a, f2 &b)
{
    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
    a = t.x;
    b = t.y;
}
__device__ __forceinline__ void st2x2(float *p, f2 a, f2 b) { *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(a, b); }

__device__ __forceinline__ f2 splat(float v) { return pk(v, v); }
__device__ __forceinline__ f2 lanes_f(uint32_t a, uint32_t b) { return pk(static_cast<float>(a), static_cast<float>(b)); }

// The two Box-Muller pairs of one Philox block, (w.x, w.y) in the low lanes and (w.z, w.w) in
// the high lanes, with the operations of box_muller_f32 lane by lane (so the normals are those of
// the scalar routine, bit for bit): -2 ln u from the base-2 logarithm for u < 3/4 and from the
// atanh series in v = 1 - u above, r = that times its reciprocal square root, and the angle
// reduced on the word to a quadrant and a Taylor-series sine and cosine.  Returns the normals of
// chains (0, 1) and (2, 3) of the block as pairs.
__device__ __forceinline__ void box_muller_block_f32x2(uint4 w, f2 &z01, f2 &z23)
{
    const f2 k32 = splat(0x1p-32f), k33 = splat(0x1p-33f);
    const f2 ua = fma2(lanes_f(w.x, w.z), k32, k33);
    float ua0, ua1;
    upk(ua, ua0, ua1);
    const f2 l1 = mul2(pk(lg2_approx(ua0), lg2_approx(ua1)), splat(-1.3862943611198906f));
    const f2 v = fma2(lanes_f(~w.x, ~w.z), k32, k33);
    float d0, d1;
    upk(sub2(splat(2.0f), v), d0, d1);
    const f2 t = mul2(v, pk(rcp_approx(d0), rcp_approx(d1)));
    const f2 t2 = mul2(t, t);
    const f2 p = fma2(fma2(fma2(fma2(splat(1.0f / 9.0f), t2, splat(1.0f / 7.0f)), t2, splat(1.0f / 5.0f)), t2,
                           splat(1.0f / 3.0f)),
                      t2, splat(1.0f));
    const f2 l2 = mul2(mul2(splat(4.0f), t), p);
    float l1a, l1b, l2a, l2b;
    upk(l1, l1a, l1b);
    upk(l2, l2a, l2b);
    const float q0 = w.x >= 0xC0000000u ? l2a : l1a, q1 = w.z >= 0xC0000000u ? l2b : l1b;
    const f2 q2 = pk(q0, q1);
    const f2 r = mul2(q2, pk(rsqrt_approx(q0), rsqrt_approx(q1)));
    const uint32_t s0 = w.y + 0x20000000u, s1 = w.w + 0x20000000u;
    const f2 dd = add2(sub2(pk(__uint_as_float(0x3F800000u | ((s0 >> 7) & 0x7FFFFFu)),
                               __uint_as_float(0x3F800000u | ((s1 >> 7) & 0x7FFFFFu))),
                            splat(1.5f)),
                       splat(0x1p-24f));
    const f2 dsq = mul2(dd, dd);
    const f2 ps = fma2(fma2(fma2(fma2(splat(1.6044118478735982e-4f), dsq, splat(-4.6817541353186881e-3f)), dsq,
                                 splat(7.9692626246167046e-2f)),
                            dsq, splat(-6.4596409750624625e-1f)),
                       dsq, splat(1.5707963267948966f));
    float sn[2], cs[2];
    upk(mul2(dd, ps), sn[0], sn[1]);
    upk(fma2(fma2(fma2(fma2(splat(9.1926027483942659e-4f), dsq, splat(-2.0863480763352961e-2f)), dsq,
                       splat(2.5366950790104802e-1f)),
                  dsq, splat(-1.2337005501361697f)),
             dsq, splat(1.0f)),
        cs[0], cs[1]);
    const uint32_t quad[2] = {s0 >> 30, s1 >> 30};
    float cq[2], sq[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        cq[h] = (quad[h] & 1u) ? -sn[h] : cs[h];
        sq[h] = (quad[h] & 1u) ? cs[h] : sn[h];
        if (quad[h] & 2u) {
            cq[h] = -cq[h];
            sq[h] = -sq[h];
        }
    }
    // each pair's radius times its (cos, sin): the chains' order, with no transposition
    float r0, r1;
    upk(r, r0, r1);
    z01 = mul2(splat(r0), pk(cq[0], sq[0]));
    z23 = mul2(splat(r1), pk(cq[1], sq[1]));
}

}  // namespace gmrf
