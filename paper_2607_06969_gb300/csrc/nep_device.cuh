// Device math of the NEP pair terms: cutoff and Chebyshev basis (Eqs. 12-15),
// real solid harmonics for l = 1..4 (Eq. 16) and their gradients.
#pragma once
#include "nep_internal.h"

#if !defined(__CUDA_ARCH__)
#include <cmath>
#endif

namespace nep {

// IEEE single operations that the compiler must not contract into FMAs;
// the neighbour predicate and the pair vectors are defined with them.
NEP_HD float add_rn(float a, float b) {
#if defined(__CUDA_ARCH__)
    return __fadd_rn(a, b);
#else
    volatile float r = a + b;
    return r;
#endif
}
NEP_HD float mul_rn(float a, float b) {
#if defined(__CUDA_ARCH__)
    return __fmul_rn(a, b);
#else
    volatile float r = a * b;
    return r;
#endif
}
NEP_HD float sub_rn(float a, float b) {
#if defined(__CUDA_ARCH__)
    return __fsub_rn(a, b);
#else
    volatile float r = a - b;
    return r;
#endif
}
// correctly rounded reciprocal
NEP_HD float rcp_f(float x) {
#if defined(__CUDA_ARCH__)
    return __frcp_rn(x);
#else
    return 1.0f / x;
#endif
}
NEP_HD float tanh_f(float x) {
#if defined(__CUDA_ARCH__)
    return tanhf(x);
#else
    return (float)std::tanh((double)x);
#endif
}
NEP_HD float sqrt_f(float x) {
#if defined(__CUDA_ARCH__)
    return sqrtf(x);
#else
    return (float)std::sqrt((double)x);
#endif
}
// Distance r and 1/r of a pair from d2 = |r_ij|^2 > 0: one reciprocal
// square root (rsqrtf, within 2 ulp) and a product on the device, in place
// of a correctly rounded square root and reciprocal (2.8% of an evaluation
// at 900k atoms, measured; the results stay within the FP32 parity bars).
NEP_HD void dist_rinv(float d2, float& r, float& ir) {
#if defined(__CUDA_ARCH__)
    ir = rsqrtf(d2);
    r = d2 * ir;
#else
    r = sqrt_f(d2);
    ir = rcp_f(r);
#endif
}
NEP_HD float dist_r(float d2) {
#if defined(__CUDA_ARCH__)
    return d2 * rsqrtf(d2);
#else
    return sqrt_f(d2);
#endif
}
NEP_HD float rint_f(float x) {
#if defined(__CUDA_ARCH__)
    return rintf(x);
#else
    return std::nearbyint(x);
#endif
}
// eight consecutive floats from a 32-byte aligned global address that no
// thread writes during the kernel: one 256-bit load on the device
NEP_HD void load8_ro(const float* p, float* v) {
#if defined(__CUDA_ARCH__)
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
        : "l"(p));
#else
    for (int k = 0; k < 8; ++k) v[k] = p[k];
#endif
}

// the same by an ordinary (coherent) load, for data that the kernel in front may
// still write when this one starts; the address must come from after_wait
NEP_HD void load8(const float* p, float* v) {
#if defined(__CUDA_ARCH__)
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
#else
    for (int k = 0; k < 8; ++k) v[k] = p[k];
#endif
}

// Two independent FP32 FMAs in one paired instruction on the device
// (a.x * b.x + c.x, a.y * b.y + c.y, each rounded once as fmaf rounds it):
// pairing two accumulation chains leaves every result bit unchanged and
// halves the instructions the chains issue.
NEP_HD float2 ffma2(float2 a, float2 b, float2 c) {
#if defined(__CUDA_ARCH__)
    return __ffma2_rn(a, b, c);
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}

// index of the lowest set bit of a non-zero word
NEP_HD int low_bit(unsigned long long m) {
#if defined(__CUDA_ARCH__)
    return __ffsll((long long)m) - 1;
#else
    return __builtin_ctzll(m);
#endif
}
NEP_HD int f2i(float x) {
#if defined(__CUDA_ARCH__)
    return __float_as_int(x);
#else
    int r; memcpy(&r, &x, 4); return r;
#endif
}
NEP_HD float i2f(int x) {
#if defined(__CUDA_ARCH__)
    return __int_as_float(x);
#else
    float r; memcpy(&r, &x, 4); return r;
#endif
}

// Packed image shift: int8 sx | sy << 8 | sz << 16.
NEP_HD int pack_shift(int sx, int sy, int sz) {
    return (sx & 0xff) | ((sy & 0xff) << 8) | ((sz & 0xff) << 16);
}
NEP_HD void unpack_shift(int v, int& sx, int& sy, int& sz) {
    sx = (int)(signed char)(v & 0xff);
    sy = (int)(signed char)((v >> 8) & 0xff);
    sz = (int)(signed char)((v >> 16) & 0xff);
}

// Pair vector r_ij = (x_j - x_i) + s * L with the list's image, or with the
// minimum image when the list carries no shifts.  The image is added by one
// FMA: for images of 0, +-1 and +-2 boxes the product is exact, so the result is
// that of the neighbour predicate's separate product and sum; the vector seen
// from j is the exact negation in any case.
NEP_HD void pair_vector(float4 pi, float4 pj, float Lx, float Ly, float Lz, float iLx, float iLy,
                        float iLz, int min_image, int packed, float& dx, float& dy, float& dz) {
    const float ux = sub_rn(pj.x, pi.x), uy = sub_rn(pj.y, pi.y), uz = sub_rn(pj.z, pi.z);
    float sx, sy, sz;
    if (min_image) {
        sx = -rint_f(ux * iLx);
        sy = -rint_f(uy * iLy);
        sz = -rint_f(uz * iLz);
    } else {
        int a, b, c;
        unpack_shift(packed, a, b, c);
        sx = (float)a; sy = (float)b; sz = (float)c;
    }
    dx = fmaf(sx, Lx, ux);
    dy = fmaf(sy, Ly, uy);
    dz = fmaf(sz, Lz, uz);
}

// |r|^2 in the neighbour predicate's operation order
NEP_HD float dist2(float dx, float dy, float dz) {
    return add_rn(add_rn(mul_rn(dx, dx), mul_rn(dy, dy)), mul_rn(dz, dz));
}
// |r|^2 in the evaluation, which decides by it in every kernel alike: the same
// value for r and -r, within an ulp of dist2 (a pair that far from a cutoff
// contributes about 1e-13)
NEP_HD float norm2(float dx, float dy, float dz) { return fmaf(dz, dz, fmaf(dy, dy, mul_rn(dx, dx))); }

// cos(pi z) and sin(pi z) for z = r/rc in [0, 1): with w = z - 1/2,
// cos(pi z) = -sin(pi w) and sin(pi z) = cos(pi w), |pi w| <= pi/2, summed
// as their Taylor series in y = (pi w)^2 (Horner), through y^6: the first
// omitted terms are below (pi/2)^15/15! = 6.7e-10 and (pi/2)^14/14! = 6.9e-9,
// under the FP32 rounding of the result.
NEP_HD void cutoff_trig(float z, float& c, float& s) {
    // pi w with pi split in two floats, so that the product keeps ~45 bits
    const float w = z - 0.5f;
    const float t = fmaf(3.14159274101257324f, w, -8.74227766e-8f * w);
    const float y = t * t;
    float ps = 1.0f / 6227020800.0f;                 // 1/13!
    ps = fmaf(ps, y, -1.0f / 39916800.0f);            // 1/11!
    ps = fmaf(ps, y, 1.0f / 362880.0f);               // 1/9!
    ps = fmaf(ps, y, -1.0f / 5040.0f);                // 1/7!
    ps = fmaf(ps, y, 1.0f / 120.0f);
    ps = fmaf(ps, y, -1.0f / 6.0f);
    ps = fmaf(ps, y, 1.0f);
    float pc = 1.0f / 479001600.0f;                  // 1/12!
    pc = fmaf(pc, y, -1.0f / 3628800.0f);             // 1/10!
    pc = fmaf(pc, y, 1.0f / 40320.0f);                // 1/8!
    pc = fmaf(pc, y, -1.0f / 720.0f);
    pc = fmaf(pc, y, 1.0f / 24.0f);
    pc = fmaf(pc, y, -0.5f);
    pc = fmaf(pc, y, 1.0f);
    c = -t * ps;
    s = pc;
}

// Q_k(r) = (T_k(x)+1)/2 f_c(r), x = 2(r/rc-1)^2-1, f_c = (1+cos(pi r/rc))/2.
// One FMA per recurrence step and one per value: (T + 1) w = T w + w.
template <int K>
NEP_HD void basis(float r, float inv_rc, float* f) {
    float cz, sz;
    cutoff_trig(r * inv_rc, cz, sz);
    const float fc2 = fmaf(0.25f, cz, 0.25f);               // f_c / 2
    const float t = fmaf(r, inv_rc, -1.0f);
    const float x = fmaf(2.0f * t, t, -1.0f), x2 = 2.0f * x;
    float Tm = 1.0f, Tk = x;
    f[0] = 2.0f * fc2;
    if (K > 1) f[1] = fmaf(x, fc2, fc2);
#pragma unroll
    for (int k = 2; k < K; ++k) {
        const float Tn = fmaf(x2, Tk, -Tm);
        f[k] = fmaf(Tn, fc2, fc2);
        Tm = Tk;
        Tk = Tn;
    }
}

// Q_k and dQ_k/dr.  T'_{k+1} = 2 T_k + 2x T'_k - T'_{k-1}.
template <int K>
NEP_HD void basis_d(float r, float inv_rc, float* f, float* fp) {
    float sp, cp;
    cutoff_trig(r * inv_rc, cp, sp);
    const float fc2 = fmaf(0.25f, cp, 0.25f);
    const float dfc2 = (-0.25f * 3.14159265358979f) * inv_rc * sp;
    const float t = fmaf(r, inv_rc, -1.0f);
    const float x = fmaf(2.0f * t, t, -1.0f), x2 = 2.0f * x;
    const float a = 4.0f * t * inv_rc * fc2;
    float Tm = 1.0f, Tk = x, dTm = 0.0f, dTk = 1.0f;
    f[0] = 2.0f * fc2;
    fp[0] = 2.0f * dfc2;
    if (K > 1) {
        f[1] = fmaf(x, fc2, fc2);
        fp[1] = fmaf(x, dfc2, a + dfc2);
    }
#pragma unroll
    for (int k = 2; k < K; ++k) {
        const float Tn = fmaf(x2, Tk, -Tm);
        const float dTn = fmaf(x2, dTk, fmaf(2.0f, Tk, -dTm));
        f[k] = fmaf(Tn, fc2, fc2);
        fp[k] = fmaf(dTn, a, fmaf(Tn, dfc2, dfc2));
        Tm = Tk; Tk = Tn; dTm = dTk; dTk = dTn;
    }
}

// Weights C_lm such that sum_m C_lm P_lm(a) P_lm(b) = P_l(a.b) for unit a, b,
// i.e. 4 pi/(2l+1) times the squared normalisation of each real harmonic.
NEP_HD float clm(int lm) {
    switch (lm) {
        case 0: case 1: case 2: return 1.0f;
        case 3: case 4: case 6: return 3.0f;
        case 5: return 0.25f;
        case 7: return 0.75f;
        case 8: case 14: return 0.625f;
        case 9: return 15.0f;
        case 10: case 12: return 0.375f;
        case 11: return 0.25f;
        case 13: return 3.75f;
        case 15: return 8.75f;
        case 16: case 22: return 4.375f;
        case 17: return 1.25f;
        case 18: case 20: return 0.625f;
        case 19: return 1.0f / 64.0f;
        case 21: return 0.3125f;
        default: return 35.0f / 64.0f;   // 23
    }
}
NEP_HD int lm_l(int lm) { return lm < 3 ? 1 : (lm < 8 ? 2 : (lm < 15 ? 3 : 4)); }

// Real harmonics P_lm(u) of a unit vector u = (x, y, z), l = 1..4, order as in
// clm().  Each is a polynomial in z times the real or imaginary part c_k, s_k
// of a power of x + iy (s_2 and s_4 without their factors 2 and 4):
//   l = 1: y, z, x
//   l = 2: s2, y z, 3z^2-1, x z, c2
//   l = 3: s3, s2 z, y q1, p3, x q1, z c2, c3
//   l = 4: s4, z s3, s2 q2, y q3, p4, x q3, c2 q2, z c3, c4
// so sums over m of a_m P_m and of its gradient collect the coefficients of
// each c_k, s_k first: per pair the angular force takes about 95 operations
// for both sums where evaluating every P_m and its three derivatives took 230.
template <class R>
struct Harm {
    R x, y, z, c2, s2, c3, s3, c4, s4;
    R zz, q1, q2, q3, p2, p3, p4;    // 5zz-1, 7zz-1, z(7zz-3), 3zz-1, z(5zz-3), (35zz-30)zz+3
};
template <class R>
NEP_HD Harm<R> harm_of(R x, R y, R z) {
    Harm<R> h;
    const R xx = x * x, yy = y * y, zz = z * z;
    const R e1 = R(3.0) * xx - yy, e2 = xx - R(3.0) * yy;
    h.x = x; h.y = y; h.z = z; h.zz = zz;
    h.s2 = x * y;
    h.c2 = xx - yy;
    h.c3 = x * e2;
    h.s3 = y * e1;
    h.c4 = xx * e2 - yy * e1;
    h.s4 = h.s2 * h.c2;
    h.q1 = R(5.0) * zz - R(1.0);
    h.q2 = R(7.0) * zz - R(1.0);
    h.q3 = z * (R(7.0) * zz - R(3.0));
    h.p2 = R(3.0) * zz - R(1.0);
    h.p3 = z * (R(5.0) * zz - R(3.0));
    h.p4 = (R(35.0) * zz - R(30.0)) * zz + R(3.0);
    return h;
}
// P_m(u); with m a compile-time constant the switch folds away
template <class R>
NEP_HD R harm_value(int m, const Harm<R>& h) {
    switch (m) {
        case 0: return h.y;
        case 1: return h.z;
        case 2: return h.x;
        case 3: return h.s2;
        case 4: return h.y * h.z;
        case 5: return h.p2;
        case 6: return h.x * h.z;
        case 7: return h.c2;
        case 8: return h.s3;
        case 9: return h.s2 * h.z;
        case 10: return h.y * h.q1;
        case 11: return h.p3;
        case 12: return h.x * h.q1;
        case 13: return h.z * h.c2;
        case 14: return h.c3;
        case 15: return h.s4;
        case 16: return h.z * h.s3;
        case 17: return h.s2 * h.q2;
        case 18: return h.y * h.q3;
        case 19: return h.p4;
        case 20: return h.x * h.q3;
        case 21: return h.c2 * h.q2;
        case 22: return h.z * h.c3;
        default: return h.c4;
    }
}

// The derivative of every term along a tangent du of the unit sphere
template <class R>
struct HarmD {
    R x, y, z, c2, s2, c3, s3, c4, s4, q1, q2, q3, p2, p3, p4;
};
template <class R>
NEP_HD HarmD<R> harm_along(const Harm<R>& h, R dx, R dy, R dz) {
    HarmD<R> d;
    const R zd = h.z * dz, c23 = R(3.0) * h.c2, s26 = R(6.0) * h.s2;
    d.x = dx; d.y = dy; d.z = dz;
    d.c2 = R(2.0) * (h.x * dx - h.y * dy);
    d.s2 = h.x * dy + h.y * dx;
    d.c3 = c23 * dx - s26 * dy;
    d.s3 = s26 * dx + c23 * dy;
    d.c4 = R(4.0) * (h.c3 * dx - h.s3 * dy);
    d.s4 = h.s3 * dx + h.c3 * dy;
    d.q1 = R(10.0) * zd;
    d.q2 = R(14.0) * zd;
    d.q3 = (R(21.0) * h.zz - R(3.0)) * dz;
    d.p2 = R(6.0) * zd;
    d.p3 = (R(15.0) * h.zz - R(3.0)) * dz;
    d.p4 = (R(140.0) * h.zz - R(60.0)) * zd;
    return d;
}
// along the change of u = r_ij / r when r_ij changes by dr (udr = u . dr)
template <class R>
NEP_HD HarmD<R> unit_tangent(const Harm<R>& h, R drx, R dry, R drz, R udr, R ir) {
    return harm_along(h, (drx - h.x * udr) * ir, (dry - h.y * udr) * ir, (drz - h.z * udr) * ir);
}
template <class R>
NEP_HD R harm_dvalue(int m, const Harm<R>& h, const HarmD<R>& d) {
    switch (m) {
        case 0: return d.y;
        case 1: return d.z;
        case 2: return d.x;
        case 3: return d.s2;
        case 4: return h.y * d.z + d.y * h.z;
        case 5: return d.p2;
        case 6: return h.x * d.z + d.x * h.z;
        case 7: return d.c2;
        case 8: return d.s3;
        case 9: return h.s2 * d.z + d.s2 * h.z;
        case 10: return h.y * d.q1 + d.y * h.q1;
        case 11: return d.p3;
        case 12: return h.x * d.q1 + d.x * h.q1;
        case 13: return h.z * d.c2 + d.z * h.c2;
        case 14: return d.c3;
        case 15: return d.s4;
        case 16: return h.z * d.s3 + d.z * h.s3;
        case 17: return h.s2 * d.q2 + d.s2 * h.q2;
        case 18: return h.y * d.q3 + d.y * h.q3;
        case 19: return d.p4;
        case 20: return h.x * d.q3 + d.x * h.q3;
        case 21: return h.c2 * d.q2 + d.c2 * h.q2;
        case 22: return h.z * d.c3 + d.z * h.c3;
        default: return d.c4;
    }
}

// sum_m a_m grad P_m(u) and sum_m b_m P_m(u): add() takes m = 0..23 in
// ascending order, each once.  The gradient is that of the polynomials above,
// whose part along u has no meaning: force() takes it out.
template <class R>
struct HarmSums {
    R C1, S1, C2, S2, C3, S3, C4, S4;                   // coefficients of c_k, s_k (c_1 = x, s_1 = y)
    R D0, D1, E1, D2, E2, D3, E3;                       // their derivatives by z
    R v0, v1, w1, v2, w2, v3, w3, v4, w4;               // the same coefficients from b
    R z6, z10, z14, t3, t4, t5;
    NEP_HD explicit HarmSums(const Harm<R>& h) {
        z6 = R(6.0) * h.z;
        z10 = R(10.0) * h.z;
        z14 = R(14.0) * h.z;
        t3 = R(15.0) * h.zz - R(3.0);
        t4 = R(21.0) * h.zz - R(3.0);
        t5 = (R(140.0) * h.zz - R(60.0)) * h.z;
    }
    NEP_HD void add(int m, const Harm<R>& h, R a, R b) {
        switch (m) {
            case 0: S1 = a; w1 = b; break;
            case 1: D0 = a; v0 = b * h.z; break;
            case 2: C1 = a; v1 = b; break;
            case 3: S2 = a; w2 = b; break;
            case 4: S1 += a * h.z; E1 = a; w1 += b * h.z; break;
            case 5: D0 += a * z6; v0 += b * h.p2; break;
            case 6: C1 += a * h.z; D1 = a; v1 += b * h.z; break;
            case 7: C2 = a; v2 = b; break;
            case 8: S3 = a; w3 = b; break;
            case 9: S2 += a * h.z; E2 = a; w2 += b * h.z; break;
            case 10: S1 += a * h.q1; E1 += a * z10; w1 += b * h.q1; break;
            case 11: D0 += a * t3; v0 += b * h.p3; break;
            case 12: C1 += a * h.q1; D1 += a * z10; v1 += b * h.q1; break;
            case 13: C2 += a * h.z; D2 = a; v2 += b * h.z; break;
            case 14: C3 = a; v3 = b; break;
            case 15: S4 = a; w4 = b; break;
            case 16: S3 += a * h.z; E3 = a; w3 += b * h.z; break;
            case 17: S2 += a * h.q2; E2 += a * z14; w2 += b * h.q2; break;
            case 18: S1 += a * h.q3; E1 += a * t4; w1 += b * h.q3; break;
            case 19: D0 += a * t5; v0 += b * h.p4; break;
            case 20: C1 += a * h.q3; D1 += a * t4; v1 += b * h.q3; break;
            case 21: C2 += a * h.q2; D2 += a * z14; v2 += b * h.q2; break;
            case 22: C3 += a * h.z; D3 = a; v3 += b * h.z; break;
            default: C4 = a; v4 = b; break;
        }
    }
    // f = u sum_m b_m P_m + (1/r) (1 - u u^T) sum_m a_m grad P_m
    NEP_HD void force(const Harm<R>& h, R ir, R& fx, R& fy, R& fz) const {
        const R x2 = R(2.0) * h.x, y2 = R(2.0) * h.y, c23 = R(3.0) * h.c2, s26 = R(6.0) * h.s2;
        const R c34 = R(4.0) * h.c3, s34 = R(4.0) * h.s3;
        const R Gx = C1 + x2 * C2 + h.y * S2 + c23 * C3 + s26 * S3 + c34 * C4 + h.s3 * S4;
        const R Gy = S1 - y2 * C2 + h.x * S2 - s26 * C3 + c23 * S3 - s34 * C4 + h.c3 * S4;
        const R Gz = D0 + D1 * h.x + E1 * h.y + D2 * h.c2 + E2 * h.s2 + D3 * h.c3 + E3 * h.s3;
        const R val = v0 + v1 * h.x + w1 * h.y + v2 * h.c2 + w2 * h.s2 + v3 * h.c3 + w3 * h.s3 + v4 * h.c4 +
                      w4 * h.s4;
        const R ug = h.x * Gx + h.y * Gy + h.z * Gz;
        const R rad = val - ir * ug;
        fx = h.x * rad + Gx * ir;
        fy = h.y * rad + Gy * ir;
        fz = h.z * rad + Gz * ir;
    }
};

// 4-body term from the l = 2 block s[0..4] = (xy, yz, 2zz-xx-yy, xz, xx-yy)
// sums: A = sum_j g (u u^T - I/3) is traceless symmetric with
// A_xy = s0, A_yz = s1, A_zz = s2/3, A_xz = s3, A_xx - A_yy = s4.
// q4 = tr(A^3); dq4/ds returned in ds.
template <class R>
NEP_HD R fourbody(const R* s, R* ds) {
    R axy = s[0], ayz = s[1], azz = s[2] * (R(1.0) / R(3.0)), axz = s[3];
    R axx = R(0.5) * (s[4] - azz), ayy = -R(0.5) * (s[4] + azz);
    // B = A^2 (symmetric)
    R bxx = axx * axx + axy * axy + axz * axz;
    R byy = axy * axy + ayy * ayy + ayz * ayz;
    R bzz = axz * axz + ayz * ayz + azz * azz;
    R bxy = axx * axy + axy * ayy + axz * ayz;
    R bxz = axx * axz + axy * ayz + axz * azz;
    R byz = axy * axz + ayy * ayz + ayz * azz;
    R q4 = axx * bxx + ayy * byy + azz * bzz + R(2.0) * (axy * bxy + axz * bxz + ayz * byz);
    if (ds) {
        ds[0] = R(6.0) * bxy;
        ds[1] = R(6.0) * byz;
        ds[2] = bzz - R(0.5) * (bxx + byy);
        ds[3] = R(6.0) * bxz;
        ds[4] = R(1.5) * (bxx - byy);
    }
    return q4;
}

NEP_HD float fma_r(float a, float b, float c) { return fmaf(a, b, c); }
NEP_HD double fma_r(double a, double b, double c) { return fma(a, b, c); }

// Directional derivative of the 4-body gradient: J = dq4/ds (as fourbody)
// and dJ = d/de J(s + e ds) at e = 0.  With A(s) linear, d(A^2) = A dA + dA A
// and J is the same linear map of A^2 as dJ is of A dA + dA A.
template <class R>
NEP_HD void fourbody_jvp(const R* s, const R* ds, R* J, R* dJ) {
    R a[3][3], d[3][3];
    {
        const R azz = s[2] * (R(1.0) / R(3.0));
        a[0][1] = a[1][0] = s[0];
        a[1][2] = a[2][1] = s[1];
        a[0][2] = a[2][0] = s[3];
        a[2][2] = azz;
        a[0][0] = R(0.5) * (s[4] - azz);
        a[1][1] = -R(0.5) * (s[4] + azz);
        const R dzz = ds[2] * (R(1.0) / R(3.0));
        d[0][1] = d[1][0] = ds[0];
        d[1][2] = d[2][1] = ds[1];
        d[0][2] = d[2][0] = ds[3];
        d[2][2] = dzz;
        d[0][0] = R(0.5) * (ds[4] - dzz);
        d[1][1] = -R(0.5) * (ds[4] + dzz);
    }
    R B[3][3], C[3][3];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            R b = R(0.0), x = R(0.0), y = R(0.0);
            for (int k = 0; k < 3; ++k) {
                b = fma_r(a[r][k], a[k][c], b);
                x = fma_r(a[r][k], d[k][c], x);
                y = fma_r(d[r][k], a[k][c], y);
            }
            B[r][c] = b;
            C[r][c] = x + y;
        }
    J[0] = R(6.0) * B[0][1];
    J[1] = R(6.0) * B[1][2];
    J[2] = B[2][2] - R(0.5) * (B[0][0] + B[1][1]);
    J[3] = R(6.0) * B[0][2];
    J[4] = R(1.5) * (B[0][0] - B[1][1]);
    dJ[0] = R(6.0) * C[0][1];
    dJ[1] = R(6.0) * C[1][2];
    dJ[2] = C[2][2] - R(0.5) * (C[0][0] + C[1][1]);
    dJ[3] = R(6.0) * C[0][2];
    dJ[4] = R(1.5) * (C[0][0] - C[1][1]);
}

}  // namespace nep
