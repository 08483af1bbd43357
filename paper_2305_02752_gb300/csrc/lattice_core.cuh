// Collision arithmetic shared by the lattice kernels (AA in-place streaming
// and the two-array streaming of the Lees-Edwards boundary): the BGK update
// with the Guo source in pair form, and the dispatch over storage types.
#pragma once

#include <type_traits>

#include "hemo_internal.cuh"

namespace hemo {

// BGK collision with the Guo source at one node: from the 19 deviations d
// arriving at the node and the force F, the post-collision deviations p
// (before any wall term), the density and the velocity with F/2.
//
// Per direction, with d^eq = f^eq - w and S the Guo source,
//   p = (1 - om) d + om d^eq + S,
//   d^eq = w (rho - 1) + w rho (3 c.u + 4.5 (c.u)^2 - 1.5 u.u),
//   S = (1 - om/2) w (3 (c.F - u.F) + 9 (c.u)(c.F)).
// Directions come in opposite pairs (c, -c): the terms even in c are shared
// and the odd ones change sign, so each pair costs one c.u and one c.F.  In
// exact arithmetic the collision keeps the mass and adds F to the momentum;
// the rest population and the axis pairs' odd parts are computed so that
// rounded arithmetic keeps both too.
template <typename R>
__device__ __forceinline__ R recip(R x) {
    if constexpr (std::is_same<R, float>::value) return __frcp_rn(x);  // correctly rounded, as 1 / x
    else return R(1) / x;
}

template <typename R>
__device__ __forceinline__ void bgk_guo(const R (&d)[Q], R Fx, R Fy, R Fz, R om, R (&p)[Q], R &rho, R &ux, R &uy,
                                        R &uz) {
    // moments of the deviations: rho - 1 = sum d (summed without the 1, so
    // that FP32 keeps the density deviation's own precision), rho u = sum d c
    // + F/2
    R drho = R(0), mx = R(0), my = R(0), mz = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        drho += d[i];
        if (cx(i)) mx += cx(i) > 0 ? d[i] : -d[i];
        if (cy(i)) my += cy(i) > 0 ? d[i] : -d[i];
        if (cz(i)) mz += cz(i) > 0 ? d[i] : -d[i];
    }
    rho = R(1) + drho;
    const R inv = recip(rho);
    ux = (mx + R(0.5) * Fx) * inv;
    uy = (my + R(0.5) * Fy) * inv;
    uz = (mz + R(0.5) * Fz) * inv;
    const R uu = ux * ux + uy * uy + uz * uz;
    const R uF = ux * Fx + uy * Fy + uz * Fz;
    const R om1 = R(1) - om, src = R(1) - R(0.5) * om;
    // even part A + (c.u) (B (c.u) + C (c.F)) of om d^eq + S and odd part
    // G (c.u) + H (c.F), for the axis weight 1/18; the diagonal weight 1/36
    // is exactly half of it
    const R w1 = R(1.0 / 18.0), ow = om * w1, sw = src * w1;
    const R A = ow * (drho - R(1.5) * rho * uu) - R(3) * sw * uF;
    const R B = R(4.5) * ow * rho, C = R(9) * sw, G = R(3) * ow * rho, H = R(3) * sw;
    // The weights' rounding (18 fl(1/18) = 1 + 7e-9 in FP32) would scale the
    // momentum by the same factor in every collision, a drift that adds up
    // over the steps.  The odd parts of the three axis pairs are therefore
    // the remainders that make the post-collision momentum m + F (what the
    // formulas give in exact arithmetic), and the rest population the
    // remainder that conserves mass.
    R sx = R(0), sy = R(0), sz = R(0), se = R(0), od[6];
#pragma unroll
    for (int a = 7; a < Q; a += 2) {  // diagonal pairs: even part now, odd part kept
        const R cu = R(cx(a)) * ux + R(cy(a)) * uy + R(cz(a)) * uz;
        const R cF = R(cx(a)) * Fx + R(cy(a)) * Fy + R(cz(a)) * Fz;
        const R even = R(0.5) * (A + cu * (B * cu + C * cF));
        const R odd = R(0.5) * (G * cu + H * cF);
        p[a] = om1 * d[a] + even;
        p[a + 1] = om1 * d[a + 1] + even;
        od[(a - 7) / 2] = odd;
        se += even;
        if (cx(a)) sx += cx(a) > 0 ? odd : -odd;
        if (cy(a)) sy += cy(a) > 0 ? odd : -odd;
        if (cz(a)) sz += cz(a) > 0 ? odd : -odd;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // axis pairs (1, 2), (3, 4), (5, 6)
        const int a = 1 + 2 * k;
        const R cu = k == 0 ? ux : (k == 1 ? uy : uz);
        const R cF = k == 0 ? Fx : (k == 1 ? Fy : Fz);
        const R mk = k == 0 ? mx : (k == 1 ? my : mz);
        const R sk = k == 0 ? sx : (k == 1 ? sy : sz);
        const R even = A + cu * (B * cu + C * cF);
        const R odd = R(0.5) * (om * mk + cF) - sk;  // sum over pairs of 2 c odd = om m + F
        se += even;
        p[a] = om1 * d[a] + even + odd;
        p[a + 1] = om1 * d[a + 1] + even - odd;
    }
    p[0] = om1 * d[0] + (om * drho - R(2) * se);  // sum over directions of om d^eq + S = om (rho - 1)
#pragma unroll
    for (int a = 7; a < Q; a += 2) {
        p[a] += od[(a - 7) / 2];
        p[a + 1] -= od[(a - 7) / 2];
    }
}

// Moments of the deviations from the opposite pairs' sums s and differences t
// (FP64: 39 operations instead of 48)
template <typename R>
__device__ __forceinline__ void pair_moments(const R (&d)[Q], R (&s)[9], R (&t)[9], R &drho, R (&m)[3]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        s[k] = d[2 * k + 1] + d[2 * k + 2];
        t[k] = d[2 * k + 1] - d[2 * k + 2];
    }
    drho = d[0];
#pragma unroll
    for (int k = 0; k < 9; ++k) drho += s[k];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        m[a] = t[a];
#pragma unroll
        for (int k = 3; k < 9; ++k) {
            const int i = 2 * k + 1, c = a == 0 ? cx(i) : (a == 1 ? cy(i) : cz(i));
            if (c) m[a] += c > 0 ? t[k] : -t[k];
        }
    }
}

// The same update in FP64, where the FP64 pipe bounds the kernels that call it
// (one warp instruction in 19 cycles per SM): the even parts om d^eq + S are a
// quadratic form in c, A + 3 sum_ab c_a c_b u_a V_b with V = g u + H F, and the
// odd ones linear, 2 c.W with W = g u + H F / 2 (axis weight; g = om rho / 12,
// H = 1/6 - om / 12), so both come from 3 + 6 products instead of products per
// direction, and the pairs' sums and differences carry them: 150 operations per
// node instead of 300 (products with the zero components of c are not folded
// in FP64).  48 x 39 x 64 channel: 74 -> 53 us (moments 22 -> 19);
// 32^3 box: 20 -> 15.7 us.
// A, u_a V_a and W enter the rest population and the axis pairs as they enter
// the other directions, so the remainders keep mass and momentum as above.
__device__ __forceinline__ void bgk_guo(const double (&d)[Q], double Fx, double Fy, double Fz, double om, double (&p)[Q],
                                        double &rho, double &ux, double &uy, double &uz) {
    double s[9], t[9], drho, m[3];
    pair_moments<double>(d, s, t, drho, m);
    rho = 1.0 + drho;
    const double inv = 1.0 / rho, F[3] = {Fx, Fy, Fz}, hF[3] = {0.5 * Fx, 0.5 * Fy, 0.5 * Fz};
    double u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = (m[a] + hF[a]) * inv;
    ux = u[0];
    uy = u[1];
    uz = u[2];
    const double om1 = 1.0 - om, hom = 0.5 * om, h = 0.5 - hom, om12 = om * (1.0 / 12.0);
    const double g = om12 * rho, H = 1.0 / 6.0 - om12, Hh = 0.5 * H;
    double V[3], W[3], q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double gu = g * u[a];
        V[a] = gu + H * F[a];
        W[a] = gu + Hh * F[a];
        q[a] = u[a] * V[a];
    }
    const double tr = q[0] + q[1] + q[2];
    const double A = om * (1.0 / 18.0) * drho - tr;  // ow (drho - 1.5 rho u.u) - 3 sw u.F
    const double K = 0.5 * A + 1.5 * tr;
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // axis pairs: odd parts as remainders
        const double e = h * s[a] + (A + 3.0 * q[a]);
        const double o = h * t[a] + ((hom * m[a] + hF[a]) - 4.0 * W[a]);
        p[2 * a + 1] = e + o;
        p[2 * a + 2] = e - o;
    }
#pragma unroll
    for (int k = 3; k < 9; ++k) {  // diagonal pairs (1, sg) in the plane (a, b)
        const int i = 2 * k + 1, a = cx(i) ? 0 : 1, b = cz(i) ? 2 : 1, sg = b == 2 ? cz(i) : cy(i);
        const double base = K - 1.5 * q[3 - a - b], x = u[a] * V[b] + u[b] * V[a];
        const double e = h * s[k] + (sg > 0 ? base + 1.5 * x : base - 1.5 * x);
        const double o = h * t[k] + (sg > 0 ? W[a] + W[b] : W[a] - W[b]);
        p[i] = e + o;
        p[i + 1] = e - o;
    }
    p[0] = om1 * d[0] + (om * drho - 12.0 * A - 18.0 * tr);  // - 2 times the even parts of the nine pairs
}

// Two floats in a 64-bit register: one instruction for both
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pk(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ F2 pk(float a) { return pk(a, a); }
__device__ __forceinline__ float2 unpk(F2 p) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p.v));
    return r;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// bgk_guo<float> of two nodes at once, for 16-bit storage, whose kernels are
// bound by instruction issue.  The same bits as two calls of it: every product
// that the compiler fuses with an addition there is fused here.
__device__ __forceinline__ void bgk_guo(const F2 (&d)[Q], F2 Fx, F2 Fy, F2 Fz, F2 om, F2 (&p)[Q], F2 &rho, F2 &ux,
                                        F2 &uy, F2 &uz) {
    F2 drho = d[0] + d[1], m[3];
#pragma unroll
    for (int i = 2; i < Q; ++i) drho = drho + d[i];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        m[k] = d[2 * k + 1] - d[2 * k + 2];
#pragma unroll
        for (int i = 7; i < Q; ++i) {
            const int c = k == 0 ? cx(i) : (k == 1 ? cy(i) : cz(i));
            if (c) m[k] = c > 0 ? m[k] + d[i] : m[k] - d[i];
        }
    }
    const F2 half = pk(0.5f), one = pk(1.f), w1 = pk((float)(1.0 / 18.0));
    rho = one + drho;
    const float2 r = unpk(rho);
    const F2 inv = pk(recip(r.x), recip(r.y));
    ux = fma2(half, Fx, m[0]) * inv;
    uy = fma2(half, Fy, m[1]) * inv;
    uz = fma2(half, Fz, m[2]) * inv;
    const F2 uu = fma2(uz, uz, fma2(ux, ux, uy * uy));
    const F2 uF = fma2(uz, Fz, fma2(ux, Fx, uy * Fy));
    const F2 om1 = one - om, src = fma2(pk(-0.5f), om, one);
    const F2 ow = om * w1, sw = src * w1, H = pk(3.f) * sw, nH = pk(-3.f) * sw, C = pk(9.f) * sw;
    const F2 in = fma2(pk(-1.5f) * rho, uu, drho);
    const F2 A = fma2(ow, in, nH * uF);
    const F2 B = pk(4.5f) * ow * rho, G = pk(3.f) * ow * rho;
    F2 sx, sy, sz, se, od[6];
#pragma unroll
    for (int a = 7; a < Q; a += 2) {  // diagonal pairs (1, sg) in a plane
        const bool up = (cx(a) ? cy(a) + cz(a) : cz(a)) > 0;
        const F2 u0 = cx(a) ? ux : uy, u1 = cz(a) ? uz : uy, F0 = cx(a) ? Fx : Fy, F1 = cz(a) ? Fz : Fy;
        const F2 cu = up ? u0 + u1 : u0 - u1, cF = up ? F0 + F1 : F0 - F1;
        const F2 even = half * fma2(cu, fma2(B, cu, C * cF), A);
        const F2 odd = half * fma2(G, cu, H * cF);
        p[a] = fma2(om1, d[a], even);
        p[a + 1] = fma2(om1, d[a + 1], even);
        od[(a - 7) / 2] = odd;
        se = a == 7 ? even : se + even;
        // (7, 9: the xy plane; 11, 13: xz; 15, 17: yz)
        if (cx(a)) sx = a == 7 ? odd : sx + odd;
        if (cy(a)) sy = a == 7 ? odd : (cy(a) > 0 ? sy + odd : sy - odd);
        if (cz(a)) sz = a == 11 ? odd : (cz(a) > 0 ? sz + odd : sz - odd);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int a = 1 + 2 * k;
        const F2 cu = k == 0 ? ux : (k == 1 ? uy : uz), cF = k == 0 ? Fx : (k == 1 ? Fy : Fz);
        const F2 sk = k == 0 ? sx : (k == 1 ? sy : sz);
        const F2 even = fma2(cu, fma2(B, cu, C * cF), A);
        const F2 odd = half * fma2(om, m[k], cF) - sk;
        se = se + even;
        p[a] = fma2(om1, d[a], even) + odd;
        p[a + 1] = fma2(om1, d[a + 1], even) - odd;
    }
    p[0] = fma2(om1, d[0], fma2(om, drho, pk(-2.f) * se));
#pragma unroll
    for (int a = 7; a < Q; a += 2) {
        p[a] = p[a] + od[(a - 7) / 2];
        p[a + 1] = p[a + 1] - od[(a - 7) / 2];
    }
}

// storage type by precision: FP64 arithmetic only with FP64 storage
#define HEMO_DISPATCH_T(prec, R, CALL)                           \
    do {                                                         \
        if constexpr (std::is_same<R, double>::value) {          \
            using T = double;                                    \
            CALL;                                                \
        } else if ((prec) == HEMO_F32) {                         \
            using T = float;                                     \
            CALL;                                                \
        } else if ((prec) == HEMO_F16DEV) {                      \
            using T = __half;                                    \
            CALL;                                                \
        } else {                                                 \
            using T = __nv_bfloat16;                             \
            CALL;                                                \
        }                                                        \
    } while (0)

}  // namespace hemo
