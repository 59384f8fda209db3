// Rotation sub-steps of a free particle in FP32 pairs.
//
// An FP64 warp instruction holds its SM sub-partition for 64 cycles on this
// GPU and the n_s sub-steps of a step are one chain (26 such instructions
// each), so in FP64 they took 110 us per step for n_s = 100.  A step of one
// particle with n_s = 100, the DEM kernel of an FP64 lattice: 114 us in FP64, 62
// as some 600 FP32 instructions of one lane, 36 with a lane per
// component.
//
// The scheme is that of rotate_free_quad (k_particles.cu), in the variables
//   u = h w_b / 2 (the half angle of a sub-step), tau = (h/2)^2 T_b,
//   d = (c, s): s = u sin|u| / |u|, c = cos|u|:
//     uh  = u + G + P(u)                  G_l = tau_l / I_l
//     tau' = tau - 2 c s x tau + 2 s x (s x tau)
//     u'  = uh + G' + P(uh + G' + P(uh))  P_l(u) = cI_l u_{l+1} u_{l+2}
//     D'  = D (x) d.
// What makes pairs of FP32 enough is what they hold: not the state, but its
// change within the step.
//   u = U_0 + 2 k G_0 + delta after k sub-steps, U_0 and G_0 in FP64 and put
//   together in FP64 at the end; delta holds the gyroscopic terms and the
//   turning of the torque, a small part of u;
//   tau = tau_0 + theta; D = (sqrt(1 - |beta|^2), beta) from the identity, so
//   |beta| is the half angle of the whole step, and q_0 (x) D is formed in FP64.
// A pair carries 2^-48 of delta, theta and beta, which are at most 2^-8 of the
// state under the conditions of rot32_applies: below FP64's rounding of the
// state in each of its n_s steps.  Products that enter them are pairs too;
// single FP32 is left for terms of second order (P(uh) - P(u) inside the inner
// fixed-point sweep, s x (s x tau), 1 - c, |s| - |u|, (1 - D_0) s), whose
// rounding is under 2^-54 of the state by the same conditions.  Measured
// against 128-bit arithmetic over 1 to 400 sub-steps and angular velocities
// from rest to the limit: see tests/test_rot32.py, which compiles this file
// for the host.
#pragma once

#ifdef __CUDACC__
#define ROT32_FN __host__ __device__ __forceinline__
#else
#include <cmath>
#define ROT32_FN inline
#endif

namespace lbmmb {

// value = h + l, |l| <= ulp(h) (not always rounded to nearest)
struct Pair {
    float h, l;
};

ROT32_FN float rot_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fmaf(a, b, c);
#endif
}
ROT32_FN float rot_add(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    volatile float r = a + b;
    return r;
#endif
}
ROT32_FN float rot_mul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    volatile float r = a * b;
    return r;
#endif
}
// v as a pair (on the device without FP64 conversions, see from_double)
ROT32_FN Pair rot_split(double v) {
    Pair p;
#ifdef __CUDA_ARCH__
    p.h = from_double<float>(v);
    p.l = from_double<float>(v - to_double(p.h));
#else
    p.h = (float)v;
    p.l = (float)(v - (double)p.h);
#endif
    return p;
}
// a + b exactly as h + l (Knuth)
ROT32_FN Pair two_sum(float a, float b) {
    Pair r;
    r.h = rot_add(a, b);
    const float bb = rot_add(r.h, -a);
    r.l = rot_add(rot_add(a, -rot_add(r.h, -bb)), rot_add(b, -bb));
    return r;
}
ROT32_FN Pair renorm(Pair a) {
    Pair r;
    r.h = rot_add(a.h, a.l);
    r.l = rot_add(a.l, -rot_add(r.h, -a.h));
    return r;
}
ROT32_FN Pair padd(Pair a, Pair b) {
    Pair s = two_sum(a.h, b.h);
    s.l = rot_add(s.l, rot_add(a.l, b.l));
    return renorm(s);
}
ROT32_FN Pair pmul(Pair a, Pair b) {
    Pair r;
    r.h = rot_mul(a.h, b.h);
    r.l = rot_fma(a.l, b.h, rot_fma(a.h, b.l, rot_fma(a.h, b.h, -r.h)));
    return r;
}
// a x b - c x d
ROT32_FN Pair pcross(Pair a, Pair b, Pair c, Pair d) {
    const Pair p = pmul(a, b), q = pmul(c, d);
    Pair s = two_sum(p.h, -q.h);
    s.l = rot_add(s.l, rot_add(p.l, -q.l));
    return renorm(s);
}

struct Rot32 {
    Pair cI[3], iI[3];   // Euler coefficients, 1 / I
    Pair U0[3], G0[3];   // at the start: h w_b / 2, (h/2)^2 T_b / I
    Pair t0[3];          // (h/2)^2 T_b
};
struct Rot32Result {
    Pair delta[3], beta[3];
    bool ok;
};

constexpr float kRot32MaxHalfAngle2 = 1.0f / (1 << 30);  // |uh| <= 2^-15 in every sub-step

// Whether the pairs carry FP64's accuracy: u0max is |h w_b / 2| at the start
// plus the torque's share over the step; half the limits on a sub-step's and
// the whole step's half angle are left to the gyroscopic terms, which cannot
// double |w_b| within so small an angle (|cI| <= 1 as of any mass
// distribution).  Fewer than kRot32MinSub sub-steps are left in FP64, where
// the last roundings weigh more than the sub-steps' and the time is short
// (n_s = 1 and 2 measured within 1.7 of FP64's error, from 10 on below it).
constexpr int kRot32MinSub = 8;
ROT32_FN bool rot32_applies(float u0max, int n_sub, float cImax) {
    return n_sub >= kRot32MinSub && u0max <= 1.0f / (1 << 16) && u0max * (float)n_sub <= 1.0f / (1 << 9) &&
           cImax <= 1.0001f;
}

// The sub-steps, written for one component at a time: X gives a component's
// neighbours.  The host holds the three in an array (N = 3); on the device each
// is a lane's (N = 1) and neighbours are shuffled.
//
// A lane's sub-step is about 330 instructions beside a chain of pair operations
// nearly as long: products and sums are put together so that what is known
// early is added early, and one sum is left after each of P, X, g' and P(v1).
// (One lane for all three components, and the sums in the order of the formulas:
// about 870 cycles a sub-step.)
template <class X>
ROT32_FN bool rot32_steps(const X &x, const Pair (&cI)[X::N], const Pair (&iI)[X::N], const Pair (&U0)[X::N],
                          const Pair (&G0)[X::N], const Pair (&t0)[X::N], int n_sub, Pair (&delta)[X::N],
                          Pair (&beta)[X::N]) {
    constexpr int N = X::N;
    const Pair zero = {0.f, 0.f};
    Pair base[N], th[N], t[N], g[N], u[N];
#pragma unroll
    for (int l = 0; l < N; l++) {
        delta[l] = beta[l] = th[l] = g[l] = zero;
        base[l] = u[l] = U0[l];
        t[l] = t0[l];
    }
    bool ok = true;
    for (int k = 0; k < n_sub; k++) {
        Pair P[N], uh[N], e0[N], pre[N], dpre[N], sa[N], sb[N], so[N], Xc[N], v1[N], nb[N];
        float cm1[N];
#pragma unroll
        for (int l = 0; l < N; l++) {
            const Pair Gg = padd(G0[l], g[l]);
            P[l] = pmul(pmul(cI[l], x.at(u, l, 1)), x.at(u, l, 2));
            uh[l] = padd(padd(u[l], Gg), P[l]);
            e0[l].h = rot_add(Gg.h, P[l].h);  // uh - u
        }
#pragma unroll
        for (int l = 0; l < N; l++) {
            so[l] = uh[l];
            sa[l] = x.at(uh, l, 1);
            sb[l] = x.at(uh, l, 2);
            const float a2 = rot_fma(uh[l].h, uh[l].h, rot_fma(sa[l].h, sa[l].h, rot_mul(sb[l].h, sb[l].h)));
            ok = ok && a2 <= kRot32MaxHalfAngle2;
            const float es = rot_mul(a2, rot_fma(a2, 1.0f / 120.0f, -1.0f / 6.0f));
            cm1[l] = rot_mul(a2, rot_fma(a2, 1.0f / 24.0f, -0.5f));
            so[l].l = rot_fma(so[l].h, es, so[l].l);
            sa[l].l = rot_fma(sa[l].h, es, sa[l].l);
            sb[l].l = rot_fma(sb[l].h, es, sb[l].l);
        }
#pragma unroll
        for (int l = 0; l < N; l++) {
            Xc[l] = pcross(sa[l], x.at(t, l, 2), sb[l], x.at(t, l, 1));
            // P(uh) = P(u) + cI (u_a e_b + e_a u_b + e_a e_b), the second term in FP32
            const float ea = x.at_h(e0, l, 1), eb = x.at_h(e0, l, 2), ua = x.at_h(u, l, 1), ub = x.at_h(u, l, 2);
            const float dP = rot_mul(cI[l].h, rot_fma(ua, eb, rot_mul(ea, rot_add(ub, eb))));
            Pair q = P[l];
            q.l = rot_add(q.l, dP);
            pre[l] = padd(padd(uh[l], G0[l]), renorm(q));
            dpre[l] = padd(delta[l], padd(g[l], P[l]));
        }
#pragma unroll
        for (int l = 0; l < N; l++) {
            // theta' = theta - 2 X + 2 s x X - 2 (c - 1) X
            const Pair m2X = {rot_mul(-2.0f, Xc[l].h), rot_mul(-2.0f, Xc[l].l)};
            th[l] = padd(th[l], m2X);
            const float Y = rot_fma(sa[l].h, x.at_h(Xc, l, 2), -rot_mul(sb[l].h, x.at_h(Xc, l, 1)));
            th[l].l = rot_add(th[l].l, rot_mul(2.0f, rot_fma(-cm1[l], Xc[l].h, Y)));
            th[l] = renorm(th[l]);
            t[l] = padd(t0[l], th[l]);
            g[l] = pmul(iI[l], th[l]);
            v1[l] = padd(pre[l], g[l]);
            dpre[l] = padd(dpre[l], g[l]);
        }
#pragma unroll
        for (int l = 0; l < N; l++) {
            // D (x) d: beta + s + beta x s + (D_0 - 1) s + (c - 1) beta
            const Pair ba = x.at(beta, l, 1), bb = x.at(beta, l, 2);
            const float d0m1 = rot_mul(-0.5f, rot_fma(beta[l].h, beta[l].h, rot_fma(ba.h, ba.h, rot_mul(bb.h, bb.h))));
            Pair w = pcross(ba, sb[l], bb, sa[l]);
            w.l = rot_add(w.l, rot_fma(d0m1, so[l].h, rot_mul(cm1[l], beta[l].h)));
            nb[l] = padd(beta[l], padd(renorm(so[l]), w));
        }
#pragma unroll
        for (int l = 0; l < N; l++) {
            // delta' = delta + g + g' + P(u) + P(v1)
            const Pair P1 = pmul(pmul(cI[l], x.at(v1, l, 1)), x.at(v1, l, 2));
            const Pair g2 = {2.0f * G0[l].h, 2.0f * G0[l].l};
            base[l] = padd(base[l], g2);
            u[l] = padd(padd(base[l], dpre[l]), P1);
            delta[l] = padd(dpre[l], P1);
            beta[l] = nb[l];
        }
    }
    return ok;
}

// All three components in one thread.
struct RotArray {
    static constexpr int N = 3;
    ROT32_FN Pair at(const Pair (&v)[3], int l, int o) const { return v[(l + o) % 3]; }
    ROT32_FN float at_h(const Pair (&v)[3], int l, int o) const { return v[(l + o) % 3].h; }
};
ROT32_FN Rot32Result rot32_run(const Rot32 &R, int n_sub) {
    Rot32Result o;
    o.ok = rot32_steps(RotArray(), R.cI, R.iI, R.U0, R.G0, R.t0, n_sub, o.delta, o.beta);
    return o;
}

}  // namespace lbmmb
