// Packed FP32 arithmetic and the pair terms shared by the direct pair kernels
// (pair.cu) and the hierarchical ones (tree.cu).
#pragma once

#include "vesis_internal.cuh"

namespace vesis {

// 1/sqrt(x) on the SFU without the subnormal range handling: every argument
// here is at least r_min^2, so flushing subnormals changes nothing.
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two FP32 values in one 64-bit register, for the packed f32x2 arithmetic
// of sm_100-class SMs: one instruction performs the same IEEE operation on
// both halves, so the FP32 pipe is fed with half the issue slots.
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk2(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ void upk2(f2 v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}

__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// One staged atom, every value duplicated into both halves of a pair.
struct AtomPairs {
    f2 x, y, z, q;   // position, charge
    f2 a, nb;        // A = 4 eps sigma^12, -B = -4 eps sigma^6
};

// One atom against the PTS cells of a thread, two cells per packed
// instruction; CLAMP applies r_min.
template <bool CLAMP, int PTS>
__device__ __forceinline__ void energy_atom(const AtomPairs &at, f2 px, f2 py, const f2 *pz,
                                            float rmin2, f2 *lj, f2 *ex, f2 *ey, f2 *ez)
{
    const f2 dx = sub2(px, at.x);
    const f2 dy = sub2(py, at.y);
    const f2 dxy2 = fma2(dx, dx, mul2(dy, dy));
#pragma unroll
    for (int p = 0; p < PTS / 2; ++p) {
        const f2 dz = sub2(pz[p], at.z);
        const f2 r2 = fma2(dz, dz, dxy2);
        float r2a, r2b;
        upk2(r2, r2a, r2b);
        if (CLAMP) {
            r2a = fmaxf(r2a, rmin2);
            r2b = fmaxf(r2b, rmin2);
        }
        const f2 ri = pk2(rsqrt_ftz(r2a), rsqrt_ftz(r2b));
        const f2 ri2 = mul2(ri, ri);
        const f2 ri3 = mul2(ri2, ri);
        const f2 ri6 = mul2(ri3, ri3);
        const f2 tl = fma2(at.a, ri6, at.nb);    // A r^-6 - B
        lj[p] = fma2(ri6, tl, lj[p]);
        const f2 qr3 = mul2(at.q, ri3);
        ex[p] = fma2(qr3, dx, ex[p]);
        ey[p] = fma2(qr3, dy, ey[p]);
        ez[p] = fma2(qr3, dz, ez[p]);
    }
}

// The grid kernel's form of the same pair, for the thread's two atoms at
// once (packed pairs; nk3 = -3 kq).  The cells of one z-pencil share x and
// y, so dx, dy and dx^2 + dy^2 come in once per pencil, and the pencil's sum
// of cd d_x is dx times its sum of cd.  With r^-8 (c1 r^-6 + c2) + nk3 r^-5
// (d.E) = r^-5 [r^-3 (c1 r^-6 + c2) + nk3 (d.E)], a pair adds
//   sc += cd,  fz += cd dz,  g += r^-3 E     (the E part times kq at the end)
// in 18 packed operations.  Clamped pairs keep only r^-3 E.
struct CellQuad {
    f2 z, ex, ey, ez;   // cell z and field, each duplicated into both halves
};

__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

template <bool CLAMP>
__device__ __forceinline__ void grad_pair2(const CellQuad &c, f2 dx, f2 dy, f2 dxy2, f2 az,
                                           f2 c1, f2 c2, f2 nk3, float rmin2, f2 &sc,
                                           f2 &fz, f2 &gx, f2 &gy, f2 &gz)
{
    const f2 dz = sub2(c.z, az);
    const f2 r2 = fma2(dz, dz, dxy2);
    float ra, rb;
    upk2(r2, ra, rb);
    f2 ri;
    bool ua = true, ub = true;   // not clamped
    if (CLAMP) {
        ua = ra >= rmin2;
        ub = rb >= rmin2;
        ri = pk2(rsqrt_ftz(fmaxf(ra, rmin2)), rsqrt_ftz(fmaxf(rb, rmin2)));
    } else {
        ri = pk2(rsqrt_ftz(ra), rsqrt_ftz(rb));
    }
    const f2 ri2 = mul2(ri, ri);
    const f2 ri3 = mul2(ri2, ri);
    const f2 ri6 = mul2(ri3, ri3);
    const f2 ri5 = mul2(ri3, ri2);
    const f2 t1 = fma2(c1, ri6, c2);
    const f2 dE = fma2(dx, c.ex, fma2(dy, c.ey, mul2(dz, c.ez)));
    f2 cd = mul2(ri5, fma2(ri3, t1, mul2(nk3, dE)));
    if (CLAMP) {
        float ca, cb;
        upk2(cd, ca, cb);
        cd = pk2(ua ? ca : 0.f, ub ? cb : 0.f);
    }
    sc = add2(sc, cd);
    fz = fma2(cd, dz, fz);
    gx = fma2(ri3, c.ex, gx);
    gy = fma2(ri3, c.ey, gy);
    gz = fma2(ri3, c.ez, gz);
}

// hi + lo += v with the rounding error of the addition kept in lo (Knuth's
// two-sum, both halves of the pairs at once)
__device__ __forceinline__ void two_sum_acc(f2 &hi, f2 &lo, f2 v)
{
    const f2 s = add2(hi, v);
    const f2 bb = sub2(s, hi);
    lo = add2(lo, add2(sub2(hi, sub2(s, bb)), sub2(v, bb)));
    hi = s;
}

}  // namespace vesis
