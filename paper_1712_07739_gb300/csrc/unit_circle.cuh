// The unit-circle rule of kernel_math.cuh in moment form, and the contraction of
// h with a segment: the per-pair arithmetic of the near field.
//
// The rule sums, over the Q points z_k of the half circle normal to T,
//     h_vpq = 1 / (4 pi Q) sum_k [ z_q F_vp - T_q (zz)^-1_vp ],
// F_vp the derivative of -(zz)^-1_vp along T.  With (zz)^-1 = adj / det, both
// polynomials in z (degrees 4 and 6), that is a linear functional of adj,
//     h_vpq = L[z_q adj_vp],   L[p] = sum_k y_k p(z_k) - sum_k w_k (T . grad p)(z_k),
//     w = 1 / det,  y = w^2 (T . grad det),
// symmetric in the five factors of a degree-5 monomial.  On the circle
// z = c a + s b (a, b the circle's axes, c and s the point's cosine and sine), so a
// polynomial p(c a + s b + eps T) needs only its coefficients in c^i s^j (order
// eps^0) and in c^i s^j eps, and L needs only eleven moments,
//     Th_m = sum_k w_k c^(4-m) s^m,   Ps_m = sum_k y_k c^(5-m) s^m.
// The loop over the circle points therefore evaluates two polynomials (det: 7
// coefficients, its derivative: 6) and adds to 11 sums, instead of inverting a 3 x 3
// matrix and forming F at every point; points phi and -phi share the even and odd
// parts of every polynomial, so a pair of points costs 37 multiply-adds and two
// reciprocals (the pointwise form: 114 and one reciprocal for each point).  The
// coefficients before the loop and the rows of stress and two strains after it cost
// about 430 multiply-adds in a cubic medium with axes along x, y, z and 850 in any
// other, whatever Q is.  The sums run over the same points as the pointwise form, so the
// two agree to rounding (FP64: 1e-15; FP32, chain from the separation to h / R^2
// against FP64, C11 = 1.684, C12 = 1.214, C44 = 0.754: 1.6e-7 RMS here, 2.2e-7
// pointwise with an unrefined reciprocal square root).
#pragma once
#include "kernel_math.cuh"

// Constants of a medium as the near-field kernels take them (by value, kernel parameters), the moduli
// divided by a power of two near the largest: the rules below form 1 / det^2, a sixth power
template <typename R>
struct NearMedium {
    int Q, np;                   // circle points; pairs (phi, -phi) with 0 < phi < pi / 2
    R k1, k3, k6;                // isotropic: strain_iso's factors (1 / (16 pi mu (1 - nu)) in the same unit is folded into the Burgers vectors)
    R d1, d2, e0;                // cubic: det = d0 + d1 s2 + d2 s3 with s2, s3 the symmetric functions of z_i^2; e0 = d0 + d1 / 2
    R rc[3], rn[4], re[2], rs[4];  // cubic: factors of rows_cubic
    R y12, ydiag, y44;           // cubic: C12, C11 - C12, C44 (contraction)
    R C[36];                     // Voigt stiffness
    R Z[36];                     // (zz)_m = sum_x Z[6 m + x] (z z)_x, pairs in the order of hs
    float2 Z2[36];               // the same, twice, for packed arithmetic
};

// Rows of the moment table, one per pair (phi, -phi): ten pairs of values
//   (c6, c5s) (c4s2, c3s3) (c2s4, cs5) | (c5, c4s) (c3s2, c2s3) (cs4, s5) | (c4, c3s) (c2s2, cs3) | (s4, s6) (unused)
constexpr int kMomRow = 20;
// A block keeps the table of up to this many pairs in shared memory (Q <= 513); a larger rule
// computes its rows as it goes
constexpr int kMomMax = 256;

template <typename R>
__device__ __forceinline__ void moment_row(int k, int Q, R *t) {
    double s, c;
    sincospi(double(k) / double(Q), &s, &c);
    const double c2 = c * c, s2 = s * s, cs = c * s, c4 = c2 * c2, s4 = s2 * s2;
    t[0] = R(c4 * c2), t[1] = R(c4 * cs), t[2] = R(c4 * s2), t[3] = R(c2 * s2 * cs), t[4] = R(c2 * s4), t[5] = R(cs * s4);
    t[6] = R(c4 * c), t[7] = R(c4 * s), t[8] = R(c2 * c * s2), t[9] = R(c2 * s2 * s), t[10] = R(c * s4), t[11] = R(s4 * s);
    t[12] = R(c4), t[13] = R(c2 * cs), t[14] = R(c2 * s2), t[15] = R(cs * s2), t[16] = R(s4), t[17] = R(s4 * s2);
    t[18] = t[19] = R(0);
}

__device__ __forceinline__ float recip(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Newton's iteration from the hardware's approximation: two steps square its error of 2^-20 twice,
// four multiply-adds where the correctly rounded quotient takes a longer chain with its range checks
__device__ __forceinline__ double recip(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(fma(-x, y, 1.0), y, y);
    return fma(fma(-x, y, 1.0), y, y);
}

// the rows 1 .. np of a block's table (nothing for a rule too large for it)
template <typename R>
__device__ __forceinline__ void moment_table(int Q, int np, R *tab) {
    if (np > kMomMax) return;
    for (int k = threadIdx.x; k < np; k += blockDim.x) moment_row<R>(k + 1, Q, tab + kMomRow * k);
}

// One pair of points added to the moments, FP32: packed pairs hold the even and the odd
// part of a polynomial (one instruction for both)
__device__ __forceinline__ void moment_step(const float *t, const float det[7], const float dd[6], float Th[5],
                                            float Ps[6]) {
    const float4 *q = reinterpret_cast<const float4 *>(t);
    const float4 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3], q4 = q[4];
    const float2 t0 = make_float2(q0.x, q0.y), t1 = make_float2(q0.z, q0.w), t2 = make_float2(q1.x, q1.y),
                 t3 = make_float2(q1.z, q1.w), t4 = make_float2(q2.x, q2.y), t5 = make_float2(q2.z, q2.w),
                 t6 = make_float2(q3.x, q3.y), t7 = make_float2(q3.z, q3.w);
    float2 x = mul2(make_float2(det[0], det[1]), t0);
    float2 e = mul2(make_float2(dd[0], dd[1]), t3);
    x = fma2(make_float2(det[2], det[3]), t1, x);
    e = fma2(make_float2(dd[2], dd[3]), t4, e);
    x = fma2(make_float2(det[4], det[5]), t2, x);
    e = fma2(make_float2(dd[4], dd[5]), t5, e);
    const float ev = fmaf(det[6], q4.y, x.x);
    const float wp = recip(ev + x.y), wm = recip(ev - x.y);
    const float yp = (e.x + e.y) * (wp * wp), ym = (e.x - e.y) * (wm * wm);
    const float2 W = make_float2(wp + wm, wp - wm), Y = make_float2(yp + ym, yp - ym);
    const float2 a0 = fma2(W, t6, make_float2(Th[0], Th[1])), a1 = fma2(W, t7, make_float2(Th[2], Th[3]));
    const float2 p0 = fma2(Y, t3, make_float2(Ps[0], Ps[1])), p1 = fma2(Y, t4, make_float2(Ps[2], Ps[3])),
                 p2 = fma2(Y, t5, make_float2(Ps[4], Ps[5]));
    Th[0] = a0.x, Th[1] = a0.y, Th[2] = a1.x, Th[3] = a1.y;
    Th[4] = fmaf(W.x, q4.x, Th[4]);
    Ps[0] = p0.x, Ps[1] = p0.y, Ps[2] = p1.x, Ps[3] = p1.y, Ps[4] = p2.x, Ps[5] = p2.y;
}
__device__ __forceinline__ void moment_step(const double *t, const double det[7], const double dd[6], double Th[5],
                                            double Ps[6]) {
    const double ev = det[0] * t[0] + det[2] * t[2] + det[4] * t[4] + det[6] * t[17];
    const double od = det[1] * t[1] + det[3] * t[3] + det[5] * t[5];
    const double e = dd[0] * t[6] + dd[2] * t[8] + dd[4] * t[10], o = dd[1] * t[7] + dd[3] * t[9] + dd[5] * t[11];
    const double dp = ev + od, dm = ev - od;
    const double r = recip(dp * dm);  // one division for the two reciprocals
    const double wp = dm * r, wm = dp * r;
    const double yp = (e + o) * (wp * wp), ym = (e - o) * (wm * wm);
    const double ws = wp + wm, wd = wp - wm, ys = yp + ym, yd = yp - ym;
    Th[0] += ws * t[12], Th[1] += wd * t[13], Th[2] += ws * t[14], Th[3] += wd * t[15], Th[4] += ws * t[16];
    Ps[0] += ys * t[6], Ps[1] += yd * t[7], Ps[2] += ys * t[8], Ps[3] += yd * t[9], Ps[4] += ys * t[10];
    Ps[5] += yd * t[11];
}

// rules beyond the shared table: the same sums, each row computed where it is used
template <typename R>
__device__ __noinline__ void moments_long(int Q, int np, const R det[7], const R dd[6], R Th[5], R Ps[6]) {
    __align__(16) R row[kMomRow];
    for (int k = 1; k <= np; ++k) {
        moment_row<R>(k, Q, row);
        moment_step(row, det, dd, Th, Ps);
    }
}

// Th, Ps of the whole rule from det and its derivative along T
template <typename R>
__device__ __forceinline__ void moments(const NearMedium<R> &m, const R *tab, const R det[7], const R dd[6], R Th[5],
                                        R Ps[6]) {
    const R w0 = recip(det[0]);  // phi = 0: c = 1, s = 0
    Th[0] = w0, Ps[0] = dd[0] * (w0 * w0);
    Th[1] = Th[2] = Th[3] = Th[4] = R(0);
    Ps[1] = Ps[2] = Ps[3] = Ps[4] = Ps[5] = R(0);
    if ((m.Q & 1) == 0) {  // phi = pi / 2
        const R w1 = recip(det[6]);
        Th[4] = w1, Ps[5] = dd[5] * (w1 * w1);
    }
    if (m.np <= kMomMax) {
#pragma unroll 1
        for (int k = 0; k < m.np; ++k) moment_step(tab + kMomRow * k, det, dd, Th, Ps);
    } else {
        moments_long<R>(m.Q, m.np, det, dd, Th, Ps);
    }
}

__device__ __forceinline__ float rsqrt_refined(float x) {
    const float y = rsqrtf(x), t = x * y;
    return fmaf(0.5f * y, fmaf(-t, y, 1.f), y);
}
__device__ __forceinline__ double rsqrt_refined(double x) { return rsqrt(x); }

// Axes of the circle normal to the unit vector T: a is the coordinate axis k of T's smallest
// component (the first of equals) made orthogonal to T, b = T x a -- the pointwise rules' axes,
// written from T's components (a_k = n, a_i = -T_k T_i / n, b = T x axis / n, n^2 = the sum of
// the other two squares)
template <typename R>
__device__ __forceinline__ void circle_axes(const R T[3], R a[3], R b[3]) {
    const R A0 = fabs(T[0]), A1 = fabs(T[1]), A2 = fabs(T[2]);
    const bool s1 = A1 < A0;
    const bool s2 = A2 < (s1 ? A1 : A0);
    const bool k2 = s2, k1 = !s2 && s1, k0 = !s2 && !s1;
    const R tk = k0 ? T[0] : (k1 ? T[1] : T[2]);
    const R u1 = k0 ? T[1] : T[0], u2 = k2 ? T[1] : T[2];  // the other two components
    const R n2 = u1 * u1 + u2 * u2;
    const R rn = rsqrt_refined(n2), u = tk * rn;
    const R n = n2 * rn;
    a[0] = k0 ? n : -u * T[0];
    a[1] = k1 ? n : -u * T[1];
    a[2] = k2 ? n : -u * T[2];
    const R r0 = T[0] * rn, r1 = T[1] * rn, r2 = T[2] * rn;
    b[0] = k0 ? R(0) : (k1 ? -r2 : r1);
    b[1] = k1 ? R(0) : (k0 ? r2 : -r0);
    b[2] = k2 ? R(0) : (k0 ? -r1 : r0);
}

// A cubic polynomial's coefficients: P[m] of c^(3-m) s^m, E[m] of c^(2-m) s^m eps
template <typename R>
struct Cubic {
    R P[4], E[3];
};
// L on a cubic polynomial, given its moments F (of y) and G (of w)
template <typename R>
__device__ __forceinline__ R apply3(const R F[4], const R G[3], const Cubic<R> &p) {
    R u = F[0] * p.P[0] + F[1] * p.P[1] + F[2] * p.P[2] + F[3] * p.P[3];
    u -= G[0] * p.E[0];
    u -= G[1] * p.E[1];
    u -= G[2] * p.E[2];
    return u;
}

// A cubic medium with axes along x, y, z: the stress rows Y (see stress_rows) of 4 pi Q h without
// h itself.  With adj_ii = al - be z_i^2 + ga z_j^2 z_k^2 and adj_ij = mcp z_i z_j (c44 + cd z_k^2)
// every row is a combination of L on monomials: lin_q = L[z_q], c1_q = L[z_q^3],
// c2_qk = L[z_q z_k^2], c3 = L[z_0 z_1 z_2], x2_q = L[z_q z_j^2 z_k^2], x3_q = L[z_i z_j z_q^3] and
// t_qk = L[z_q^3 z_k^2]; components of h that meet in a row share its terms, so the 18 rows cost 48
// multiply-adds where h and its contraction cost 92 (with Kahan sums of the pairs, whole pass of 250,000
// segments, Q = 16: 46.6 -> 44.6 ms; 3,000 segments in FP64, Q = 32: 17.7 -> 17.0 ms), and round less
// (rows of random directions, FP32, C11 = 1.684, C12 = 1.214, C44 = 0.754: 3.0e-7 by way of h, 2.5e-7).
template <typename R>
__device__ __forceinline__ void rows_cubic(const NearMedium<R> &md, const R *tab, const R T[3], R Y[3][6]) {
    R a[3], b[3];
    circle_axes<R>(T, a, b);
    R aa[3], ab[3], bb[3];  // z_i^2: aa c^2 + ab c s + bb s^2 (ab = 2 a b)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        aa[i] = a[i] * a[i];
        ab[i] = R(2) * a[i] * b[i];
        bb[i] = b[i] * b[i];
    }
    Cubic<R> z3[3];  // z_i^3
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const R a3 = R(3) * a[i], b3 = R(3) * b[i], t3 = R(3) * T[i];
        z3[i].P[0] = a[i] * aa[i], z3[i].P[1] = b3 * aa[i], z3[i].P[2] = a3 * bb[i], z3[i].P[3] = b[i] * bb[i];
        z3[i].E[0] = t3 * aa[i], z3[i].E[1] = t3 * ab[i], z3[i].E[2] = t3 * bb[i];
    }
    Cubic<R> zq[3], p3;  // z_q z_(q+1)^2 and z_0 z_1 z_2
    R x12[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int k = (q + 1) % 3;
        const R x0 = a[q] * a[k], x1 = a[q] * b[k] + b[q] * a[k], x2 = b[q] * b[k], t2 = R(2) * T[k];
        zq[q].P[0] = a[q] * aa[k], zq[q].P[1] = a[q] * ab[k] + b[q] * aa[k];
        zq[q].P[2] = a[q] * bb[k] + b[q] * ab[k], zq[q].P[3] = b[q] * bb[k];
        zq[q].E[0] = T[q] * aa[k] + t2 * x0, zq[q].E[1] = T[q] * ab[k] + t2 * x1, zq[q].E[2] = T[q] * bb[k] + t2 * x2;
        if (q == 1) x12[0] = x0, x12[1] = x1, x12[2] = x2;
    }
    {
        const R l0 = T[1] * a[2] + T[2] * a[1], l1 = T[1] * b[2] + T[2] * b[1];
        p3.P[0] = a[0] * x12[0], p3.P[1] = a[0] * x12[1] + b[0] * x12[0];
        p3.P[2] = a[0] * x12[2] + b[0] * x12[1], p3.P[3] = b[0] * x12[2];
        p3.E[0] = T[0] * x12[0] + a[0] * l0, p3.E[1] = T[0] * x12[1] + a[0] * l1 + b[0] * l0;
        p3.E[2] = T[0] * x12[2] + b[0] * l1;
    }
    // det = d0 + d1 s2 + d2 s3 as a form of degree 6 in (c, s), s2 = (1 - sum z_i^4) / 2, s3 = (z_0 z_1 z_2)^2,
    // and its derivative along T as a form of degree 5
    R det[7], dd[6];
    {
        const R r = R(-0.5) * md.d1, r43 = R(-2.0 / 3.0) * md.d1, r2 = -md.d1;
        const R q0 = r * (a[0] * z3[0].P[0] + a[1] * z3[1].P[0] + a[2] * z3[2].P[0]);
        const R q1 = r43 * (a[0] * z3[0].P[1] + a[1] * z3[1].P[1] + a[2] * z3[2].P[1]);
        const R q2 = r2 * (a[0] * z3[0].P[2] + a[1] * z3[1].P[2] + a[2] * z3[2].P[2]);
        const R q3 = r43 * (b[0] * z3[0].P[2] + b[1] * z3[1].P[2] + b[2] * z3[2].P[2]);
        const R q4 = r * (b[0] * z3[0].P[3] + b[1] * z3[1].P[3] + b[2] * z3[2].P[3]);
        const R *p = p3.P;
        const R u0 = md.d2 * p[0], u1 = md.d2 * p[1], u2 = md.d2 * p[2], u3 = md.d2 * p[3];
        const R e0 = md.e0, e3 = R(3) * md.e0;
        det[0] = (e0 + q0) + u0 * p[0];
        det[1] = q1 + R(2) * u0 * p[1];
        det[2] = (e3 + (q0 + q2)) + (R(2) * u0 * p[2] + u1 * p[1]);
        det[3] = (q1 + q3) + R(2) * (u0 * p[3] + u1 * p[2]);
        det[4] = (e3 + (q2 + q4)) + (R(2) * u1 * p[3] + u2 * p[2]);
        det[5] = q3 + R(2) * u2 * p[3];
        det[6] = (e0 + q4) + u3 * p[3];
        const R m2 = R(-2) * md.d1, v0 = R(2) * u0, v1 = R(2) * u1, v2 = R(2) * u2, v3 = R(2) * u3;
        const R g0 = m2 * (T[0] * z3[0].P[0] + T[1] * z3[1].P[0] + T[2] * z3[2].P[0]);
        const R g1 = m2 * (T[0] * z3[0].P[1] + T[1] * z3[1].P[1] + T[2] * z3[2].P[1]);
        const R g2 = m2 * (T[0] * z3[0].P[2] + T[1] * z3[1].P[2] + T[2] * z3[2].P[2]);
        const R g3 = m2 * (T[0] * z3[0].P[3] + T[1] * z3[1].P[3] + T[2] * z3[2].P[3]);
        const R *E = p3.E;
        dd[0] = g0 + v0 * E[0];
        dd[1] = g1 + (v0 * E[1] + v1 * E[0]);
        dd[2] = (g0 + g2) + (v0 * E[2] + v1 * E[1] + v2 * E[0]);
        dd[3] = (g1 + g3) + (v1 * E[2] + v2 * E[1] + v3 * E[0]);
        dd[4] = g2 + (v2 * E[2] + v3 * E[1]);
        dd[5] = g3 + v3 * E[2];
    }
    R Th[5], Ps[6];
    moments<R>(md, tab, det, dd, Th, Ps);
    // lower moments (c^2 + s^2 = 1) and L on linear and cubic monomials
    const R G[3] = {Th[0] + Th[2], Th[1] + Th[3], Th[2] + Th[4]};
    const R F[4] = {Ps[0] + Ps[2], Ps[1] + Ps[3], Ps[2] + Ps[4], Ps[3] + Ps[5]};
    const R f0 = F[0] + F[2], f1 = F[1] + F[3], g0 = G[0] + G[2];
    R lin[3], c1[3], c2[3][3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        lin[q] = a[q] * f0 + b[q] * f1 - T[q] * g0;
        c1[q] = apply3<R>(F, G, z3[q]);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int k = (q + 1) % 3, j = (q + 2) % 3;
        c2[q][k] = apply3<R>(F, G, zq[q]);          // z_q z_k^2
        c2[q][j] = lin[q] - c1[q] - c2[q][k];       // |z|^2 = 1
    }
    const R c3 = apply3<R>(F, G, p3);
    // the functionals p -> L[z_k^2 p] on cubic p; their sum over k is L
    R F2[3][4], G2[3][3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const R t2 = R(2) * T[k], ta = t2 * a[k], tb = t2 * b[k];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            R u = aa[k] * Ps[i] + ab[k] * Ps[i + 1] + bb[k] * Ps[i + 2];
            u -= ta * Th[i];
            u -= tb * Th[i + 1];
            F2[k][i] = u;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) G2[k][i] = aa[k] * Th[i] + ab[k] * Th[i + 1] + bb[k] * Th[i + 2];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) F2[2][i] = F[i] - F2[0][i] - F2[1][i];
#pragma unroll
    for (int i = 0; i < 3; ++i) G2[2][i] = G[i] - G2[0][i] - G2[1][i];
    R x2[3], x3[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int j = (q + 2) % 3;
        x2[q] = apply3<R>(F2[j], G2[j], zq[q]);
        x3[q] = q < 2 ? apply3<R>(F2[q], G2[q], p3) : c3 - x3[0] - x3[1];  // |z|^2 = 1
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R v = md.rn[0] * lin[c] + md.rn[1] * c1[c] + md.rn[2] * x2[c];
        Y[c][c] = md.rc[0] * lin[c] + md.rc[1] * c1[c] + md.rc[2] * x2[c];
        Y[c][(c + 1) % 3] = v + md.rn[3] * c2[c][(c + 1) % 3];
        Y[c][(c + 2) % 3] = v + md.rn[3] * c2[c][(c + 2) % 3];
        Y[c][3 + c] = md.re[0] * c3 + md.re[1] * x3[c];
        const R u = md.rs[0] * lin[c] + md.rs[1] * x2[c];  // shear rows with z_c as the odd factor
#pragma unroll
        for (int n = 1; n < 3; ++n) {
            const int r = (c + n) % 3, k = (c + 3 - n) % 3;
            Y[r][3 + k] = u + md.rs[2] * c2[c][r] + md.rs[3] * apply3<R>(F2[k], G2[k], z3[c]);
        }
    }
}

// An isotropic medium: with h_cpq = -3 T_c T_p T_q - ha d_cp T_q + d_cq T_p + d_pq T_c (ha = 3 - 4 nu) the
// contraction of strain_of leaves, up to an antisymmetric part that the strain does not see, the
// symmetric part of T (x) S x (k1 b - k6 (T.b) T) + k3 b (x) (S x T): 43 multiply-adds a direction and
// no rows (2,000 segments in FP64, whose near field is bound by its arithmetic: whole
// pass 5.35 -> 3.89 ms; FP32 rounding 1.7e-7 by way of the rows, 0.9e-7).
template <typename R>
__device__ __forceinline__ void strain_iso(const NearMedium<R> &md, const R T[3], R b0, R b1, R b2, R S0, R S1, R S2,
                                           R e[6]) {
    const R x0 = S1 * T[2] - S2 * T[1], x1 = S2 * T[0] - S0 * T[2], x2 = S0 * T[1] - S1 * T[0];  // S x T
    const R f = md.k6 * (T[0] * b0 + T[1] * b1 + T[2] * b2);
    const R u0 = md.k1 * (S1 * b2 - S2 * b1) - f * x0, u1 = md.k1 * (S2 * b0 - S0 * b2) - f * x1,
            u2 = md.k1 * (S0 * b1 - S1 * b0) - f * x2;
    const R w0 = md.k3 * x0, w1 = md.k3 * x1, w2 = md.k3 * x2;
    e[0] = T[0] * u0 + b0 * w0;
    e[1] = T[1] * u1 + b1 * w1;
    e[2] = T[2] * u2 + b2 * w2;
    e[3] = (T[1] * u2 + b1 * w2) + (T[2] * u1 + b2 * w1);
    e[4] = (T[0] * u2 + b0 * w2) + (T[2] * u0 + b2 * w0);
    e[5] = (T[0] * u1 + b0 * w1) + (T[1] * u0 + b1 * w0);
}

// product of two quadratic forms, A and B: coefficients of c^2, c s, s^2, then of c eps, s eps;
// out: five of degree 4, then four of degree 3 times eps
template <typename R, bool ADD>
__device__ __forceinline__ void mul_quad(const R A[5], const R B[5], R q[9]) {
    const R v[9] = {A[0] * B[0],
                    A[0] * B[1] + A[1] * B[0],
                    A[0] * B[2] + A[1] * B[1] + A[2] * B[0],
                    A[1] * B[2] + A[2] * B[1],
                    A[2] * B[2],
                    A[0] * B[3] + A[3] * B[0],
                    A[0] * B[4] + A[4] * B[0] + A[1] * B[3] + A[3] * B[1],
                    A[1] * B[4] + A[4] * B[1] + A[2] * B[3] + A[3] * B[2],
                    A[2] * B[4] + A[4] * B[2]};
#pragma unroll
    for (int i = 0; i < 9; ++i) q[i] = ADD ? v[i] : q[i] - v[i];
}

// h of any medium, times 4 pi Q: (zz) as six quadratic forms, its adjugate as six of degree 4
template <typename R>
__device__ __forceinline__ void h_general_moments(const NearMedium<R> &md, const R *tab, const R T[3], R hs[18]) {
    R a[3], b[3];
    circle_axes<R>(T, a, b);
    constexpr int PV[6] = {0, 1, 2, 1, 0, 0}, PP[6] = {0, 1, 2, 2, 2, 1};
    R q[6][9];  // adjugate
    R det[7], dd[6];
    {
        R M[6][5];
#pragma unroll
        for (int m = 0; m < 6; ++m)
#pragma unroll
            for (int i = 0; i < 5; ++i) M[m][i] = R(0);
#pragma unroll
        for (int x = 0; x < 6; ++x) {
            const int i = PV[x], l = PP[x];
            R z[5];
            if (i == l) {
                z[0] = a[i] * a[i], z[1] = R(2) * a[i] * b[i], z[2] = b[i] * b[i];
                z[3] = R(2) * T[i] * a[i], z[4] = R(2) * T[i] * b[i];
            } else {
                z[0] = a[i] * a[l], z[1] = a[i] * b[l] + b[i] * a[l], z[2] = b[i] * b[l];
                z[3] = T[i] * a[l] + T[l] * a[i], z[4] = T[i] * b[l] + T[l] * b[i];
            }
#pragma unroll
            for (int m = 0; m < 6; ++m)
#pragma unroll
                for (int e = 0; e < 5; ++e) M[m][e] += md.Z[6 * m + x] * z[e];
        }
        // pairs 00 11 22 12 02 01
        mul_quad<R, true>(M[1], M[2], q[0]);
        mul_quad<R, false>(M[3], M[3], q[0]);
        mul_quad<R, true>(M[0], M[2], q[1]);
        mul_quad<R, false>(M[4], M[4], q[1]);
        mul_quad<R, true>(M[0], M[1], q[2]);
        mul_quad<R, false>(M[5], M[5], q[2]);
        mul_quad<R, true>(M[5], M[4], q[3]);
        mul_quad<R, false>(M[0], M[3], q[3]);
        mul_quad<R, true>(M[5], M[3], q[4]);
        mul_quad<R, false>(M[4], M[1], q[4]);
        mul_quad<R, true>(M[4], M[3], q[5]);
        mul_quad<R, false>(M[5], M[2], q[5]);
#pragma unroll
        for (int i = 0; i < 7; ++i) det[i] = R(0);
#pragma unroll
        for (int i = 0; i < 6; ++i) dd[i] = R(0);
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const int m = t == 0 ? 0 : (t == 1 ? 5 : 4);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
#pragma unroll
                for (int j = 0; j < 5; ++j) det[i + j] += M[m][i] * q[m][j];
#pragma unroll
                for (int j = 0; j < 4; ++j) dd[i + j] += M[m][i] * q[m][5 + j];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 5; ++j) dd[i + j] += M[m][3 + i] * q[m][j];
        }
    }
    R Th[5], Ps[6];
    moments<R>(md, tab, det, dd, Th, Ps);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        R F[5], G[4];  // p -> L[z_d p] on p of degree 4
#pragma unroll
        for (int i = 0; i < 5; ++i) F[i] = a[d] * Ps[i] + b[d] * Ps[i + 1] - T[d] * Th[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) G[i] = a[d] * Th[i] + b[d] * Th[i + 1];
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            R s = F[0] * q[m][0] + F[1] * q[m][1] + F[2] * q[m][2] + F[3] * q[m][3] + F[4] * q[m][4];
            s -= G[0] * q[m][5] + G[1] * q[m][6] + G[2] * q[m][7] + G[3] * q[m][8];
            hs[3 * m + d] = s;
        }
    }
}

// Points of the pointwise general rule, two by two: (cos phi, cos phi', sin phi, sin phi'); the last of an
// odd number stands twice
constexpr int kPointMax = 1024;  // points kept in shared memory, else computed where used
__device__ __noinline__ inline float4 circle_points2(int k, int Q) {
    const int k0 = 2 * k, k1 = min(2 * k + 1, Q - 1);
    double s0, c0, s1, c1;
    sincospi(double(k0) / double(Q), &s0, &c0);
    sincospi(double(k1) / double(Q), &s1, &c1);
    return make_float4(float(c0), float(c1), float(s0), float(s1));
}
__device__ __forceinline__ void point_table(int Q, float *tab) {
    if (Q > kPointMax) return;
    for (int k = threadIdx.x; 2 * k < Q; k += blockDim.x) reinterpret_cast<float4 *>(tab)[k] = circle_points2(k, Q);
}

// h of any medium, times 4 pi Q, point by point (FP32), two points a step in packed arithmetic.
// (zz) comes from z itself, 36 multiply-adds, its derivative along T as S = sc cos phi + ss sin phi, and
//     F_vp = (adj_vp (adj : S) / det - dadj_vp) / det
// needs no matrix product: 66 instructions a point (132 multiply-adds; from the 81-entry C: ~450).
// (zz) as m + u cos 2phi + v sin 2phi takes 24 multiply-adds less a point, but rounds three coefficients
// into every point alike, which the sum over the points does not average out.  RMS error of the mixed
// pass's K, rule from C / harmonics / this / moments, in 1e-7: turned cubic, A = 3.2, 3.9 / 4.7 / 3.4 /
// 3.8, A = 0.17, 16.5 / 18 / 12 / 18; aligned, A = 0.48, 5.2 / 5.7 / 4.0 / 4.2; triclinic 2.8 / 3.0 / 2.3 /
// 2.5.  6,101 segments in a turned crystal, whole pass: 3.22 ms with harmonics, 3.35 here; the near
// field of 100,000 192 and 202 (88 in moment form, kept for the plain pairs beside the learned h).
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }
// a b - c d
__device__ __forceinline__ float2 det2(float2 a, float2 b, float2 c, float2 d) { return fma2(a, b, mul2(neg2(c), d)); }
__device__ __forceinline__ void h_general_points(const NearMedium<float> &md, const float *tab, const float T[3],
                                                 float hs[18]) {
    float a[3], b[3];
    circle_axes<float>(T, a, b);
    constexpr int PV[6] = {0, 1, 2, 1, 0, 0}, PP[6] = {0, 1, 2, 2, 2, 1};
    float sc[6], ss[6];
#pragma unroll
    for (int x = 0; x < 6; ++x) {
        const int i = PV[x], l = PP[x];
        const float zc = i == l ? 2.f * T[i] * a[i] : T[i] * a[l] + T[l] * a[i];
        const float zs = i == l ? 2.f * T[i] * b[i] : T[i] * b[l] + T[l] * b[i];
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            const float Z = md.Z[6 * m + x];
            sc[m] = x == 0 ? Z * zc : fmaf(Z, zc, sc[m]);
            ss[m] = x == 0 ? Z * zs : fmaf(Z, zs, ss[m]);
        }
    }
    float2 A[6], B[6], G[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) A[i] = B[i] = G[i] = dup(0.f);
    const float4 *pt = reinterpret_cast<const float4 *>(tab);
#pragma unroll 1
    for (int k = 0; 2 * k < md.Q; ++k) {
        const float4 t = md.Q <= kPointMax ? pt[k] : circle_points2(k, md.Q);
        const float2 c = make_float2(t.x, t.y), s = make_float2(t.z, t.w);
        float2 z[3], M[6], S[6];
#pragma unroll
        for (int i = 0; i < 3; ++i) z[i] = fma2(c, dup(a[i]), mul2(s, dup(b[i])));
#pragma unroll
        for (int x = 0; x < 6; ++x) {
            const int i = PV[x], l = PP[x];
            const float2 zz = mul2(z[i], z[l]);
#pragma unroll
            for (int m = 0; m < 6; ++m) {
                const float2 Z = md.Z2[6 * m + x];
                M[m] = x == 0 ? mul2(Z, zz) : fma2(Z, zz, M[m]);
            }
        }
#pragma unroll
        for (int m = 0; m < 6; ++m) S[m] = fma2(s, dup(ss[m]), mul2(c, dup(sc[m])));
        const float2 adj[6] = {det2(M[1], M[2], M[3], M[3]), det2(M[0], M[2], M[4], M[4]), det2(M[0], M[1], M[5], M[5]),
                               det2(M[5], M[4], M[0], M[3]), det2(M[5], M[3], M[4], M[1]), det2(M[4], M[3], M[5], M[2])};
        const float2 det = fma2(M[0], adj[0], fma2(M[5], adj[5], mul2(M[4], adj[4])));
        float2 w = make_float2(recip(det.x), recip(det.y));
        if (2 * k + 1 >= md.Q) w.y = 0.f;  // the point that stands twice
        const float2 S3 = mul2(S[3], dup(2.f)), S4 = mul2(S[4], dup(2.f)), S5 = mul2(S[5], dup(2.f));
        const float2 da[6] = {fma2(neg2(M[3]), S3, fma2(M[1], S[2], mul2(S[1], M[2]))),
                              fma2(neg2(M[4]), S4, fma2(M[0], S[2], mul2(S[0], M[2]))),
                              fma2(neg2(M[5]), S5, fma2(M[0], S[1], mul2(S[0], M[1]))),
                              fma2(neg2(M[0]), S[3], fma2(neg2(S[0]), M[3], fma2(M[5], S[4], mul2(S[5], M[4])))),
                              fma2(neg2(M[4]), S[1], fma2(neg2(S[4]), M[1], fma2(M[5], S[3], mul2(S[5], M[3])))),
                              fma2(neg2(M[5]), S[2], fma2(neg2(S[5]), M[2], fma2(M[4], S[3], mul2(S[4], M[3]))))};
        const float2 tau = mul2(w, fma2(adj[0], S[0], fma2(adj[1], S[1], fma2(adj[2], S[2],
                                   fma2(adj[3], S3, fma2(adj[4], S4, mul2(adj[5], S5)))))));
        const float2 cw = mul2(c, w), sw = mul2(s, w);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const float2 F = fma2(adj[i], tau, neg2(da[i]));
            A[i] = fma2(cw, F, A[i]);
            B[i] = fma2(sw, F, B[i]);
            G[i] = fma2(w, adj[i], G[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int q = 0; q < 3; ++q)
            hs[3 * i + q] = a[q] * (A[i].x + A[i].y) + b[q] * (B[i].x + B[i].y) - T[q] * (G[i].x + G[i].y);
}

// The contraction of Sec. 2, Eq. "kernel" with a point's strength q = b' x S, without the
// 6 x 18 tensor of the point: Y_c = C : h_c (the stress of the gradient h_cpq over p, q, six
// values for each c) serves both directions of a pair, X_cn = sum_w b'_w Y_c(wn), and the
// distortion S x X_c is added to a strain in Voigt order (xx yy zz, 2yz 2xz 2xy); the stress is
// C times the summed strain, applied once per target.  Per direction 48 multiply-adds and six
// values per source instead of 108 and 108.
template <typename R, bool GENERAL>
__device__ __forceinline__ void stress_rows(const NearMedium<R> &md, const R hs[18], R Y[3][6]) {
    constexpr int PIX[3][3] = {{0, 5, 4}, {5, 1, 3}, {4, 3, 2}};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R g0 = hs[3 * PIX[c][0]], g1 = hs[3 * PIX[c][1] + 1], g2 = hs[3 * PIX[c][2] + 2];
        const R g3 = hs[3 * PIX[c][1] + 2] + hs[3 * PIX[c][2] + 1], g4 = hs[3 * PIX[c][0] + 2] + hs[3 * PIX[c][2]],
                g5 = hs[3 * PIX[c][0] + 1] + hs[3 * PIX[c][1]];
        if (GENERAL) {
#pragma unroll
            for (int m = 0; m < 6; ++m)
                Y[c][m] = md.C[6 * m] * g0 + md.C[6 * m + 1] * g1 + md.C[6 * m + 2] * g2 + md.C[6 * m + 3] * g3 +
                          md.C[6 * m + 4] * g4 + md.C[6 * m + 5] * g5;
        } else {
            const R tr = md.y12 * (g0 + g1 + g2);
            Y[c][0] = tr + md.ydiag * g0, Y[c][1] = tr + md.ydiag * g1, Y[c][2] = tr + md.ydiag * g2;
            Y[c][3] = md.y44 * g3, Y[c][4] = md.y44 * g4, Y[c][5] = md.y44 * g5;
        }
    }
}

template <typename R>
__device__ __forceinline__ void strain_of(const R Y[3][6], R b0, R b1, R b2, R S0, R S1, R S2, R e[6]) {
    R X[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        X[c][0] = b0 * Y[c][0] + b1 * Y[c][5] + b2 * Y[c][4];
        X[c][1] = b0 * Y[c][5] + b1 * Y[c][1] + b2 * Y[c][3];
        X[c][2] = b0 * Y[c][4] + b1 * Y[c][3] + b2 * Y[c][2];
    }
    e[0] = S1 * X[0][2] - S2 * X[0][1];
    e[1] = S2 * X[1][0] - S0 * X[1][2];
    e[2] = S0 * X[2][1] - S1 * X[2][0];
    e[3] = (S0 * X[1][1] - S1 * X[1][0]) + (S2 * X[2][0] - S0 * X[2][2]);
    e[4] = (S0 * X[0][1] - S1 * X[0][0]) + (S1 * X[2][2] - S2 * X[2][1]);
    e[5] = (S2 * X[0][0] - S0 * X[0][2]) + (S1 * X[1][2] - S2 * X[1][1]);
}
