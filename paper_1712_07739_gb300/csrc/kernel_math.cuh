// Device arithmetic of the dislocation kernel, shared by the setup and the
// near-field kernels of this library.
//
// The kernel of Sec. 2, Eq. "kernel" is K_abwr = A_{ab,wr,vpq} dG_vp/dx_q
// with dG_vp/dx_q = h_vpq(T) / R^2.  h is symmetric in (v, p), so only 18
// components are kept, in the order k = 3 * pair + q with pairs
// (0,0) (1,1) (2,2) (1,2) (0,2) (0,1).
#pragma once
#include <cmath>

#include "internal.cuh"

// Isotropic medium: derivative of the Kelvin Green's function
// G_vp = [(3 - 4 nu) delta_vp + T_v T_p] / (16 pi mu (1 - nu) R), which is
// Sec. 2, Eq. "k_iso" with R,ii = 2/R and R,vp = (delta_vp - T_v T_p)/R:
// h_vpq = hc [ -ha delta_vp T_q + delta_vq T_p + delta_pq T_v - 3 T_v T_p T_q ].
template <typename R>
__device__ __forceinline__ void h_iso_sym(R hc, R ha, const R T[3], R hs[18]) {
    constexpr int PV[6] = {0, 1, 2, 1, 0, 0};
    constexpr int PP[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
    for (int pr = 0; pr < 6; ++pr) {
        const int v = PV[pr], p = PP[pr];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            R s = R(-3) * T[v] * T[p] * T[q];
            if (v == p) s -= ha * T[q];
            if (v == q) s += T[p];
            if (p == q) s += T[v];
            hs[3 * pr + q] = hc * s;
        }
    }
}

// (a b)_jk = a_i C_ijkl b_l
template <typename R, typename CT>
__device__ __forceinline__ void cmat(const CT *C, const R a[3], const R b[3], R M[9]) {
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            R s = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int l = 0; l < 3; ++l) s += a[i] * R(C[((i * 3 + j) * 3 + k) * 3 + l]) * b[l];
            M[j * 3 + k] = s;
        }
}

// Any medium: h_vpq(T) = 1/(8 pi^2) oint [ -T_q (zz)^-1_vp + z_q F_vp ] dphi
// over the unit circle z . T = 0, F = (zz)^-1 [(zT) + (Tz)] (zz)^-1.
// The integrand has period pi, so the loop is the Q-point trapezoid rule on
// [0, pi) doubled.  C is read through the generic 81-entry tensor.
template <typename R, typename CT>
__device__ __forceinline__ void h_circle_sym(const CT *C, int Q, const R Tin[3], R hs[18]) {
    R T[3] = {Tin[0], Tin[1], Tin[2]};
    // e1: T with its smallest component replaced, orthogonalised; e2 = T x e1
    int k0 = 0;
    if (fabs(T[1]) < fabs(T[k0])) k0 = 1;
    if (fabs(T[2]) < fabs(T[k0])) k0 = 2;
    R e1[3] = {R(0), R(0), R(0)};
    e1[k0] = R(1);
    R d = e1[0] * T[0] + e1[1] * T[1] + e1[2] * T[2];
    for (int i = 0; i < 3; ++i) e1[i] -= d * T[i];
    R n = R(1) / sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]);
    for (int i = 0; i < 3; ++i) e1[i] *= n;
    R e2[3] = {T[1] * e1[2] - T[2] * e1[1], T[2] * e1[0] - T[0] * e1[2], T[0] * e1[1] - T[1] * e1[0]};
    R acc[18];
#pragma unroll
    for (int i = 0; i < 18; ++i) acc[i] = 0;
    for (int k = 0; k < Q; ++k) {
        R s, c;
        sincospi(double(k) / double(Q), &s, &c);
        R z[3];
        for (int i = 0; i < 3; ++i) z[i] = c * e1[i] + s * e2[i];
        R M[9], ZT[9];
        cmat<R, CT>(C, z, z, M);
        cmat<R, CT>(C, z, T, ZT);
        // inverse of the symmetric positive-definite M (adjugate / determinant)
        R i00 = M[4] * M[8] - M[5] * M[7];
        R i01 = M[2] * M[7] - M[1] * M[8];
        R i02 = M[1] * M[5] - M[2] * M[4];
        R i11 = M[0] * M[8] - M[2] * M[6];
        R i12 = M[2] * M[3] - M[0] * M[5];
        R i22 = M[0] * M[4] - M[1] * M[3];
        R idet = R(1) / (M[0] * i00 + M[1] * (M[5] * M[6] - M[3] * M[8]) + M[2] * (M[3] * M[7] - M[4] * M[6]));
        R Mi[9] = {i00 * idet, i01 * idet, i02 * idet, i01 * idet, i11 * idet,
                   i12 * idet, i02 * idet, i12 * idet, i22 * idet};
        R S[9];
        for (int j = 0; j < 3; ++j)
            for (int l = 0; l < 3; ++l) S[j * 3 + l] = ZT[j * 3 + l] + ZT[l * 3 + j];
        R tmp[9], F[9];
        for (int j = 0; j < 3; ++j)
            for (int l = 0; l < 3; ++l)
                tmp[j * 3 + l] = Mi[j * 3] * S[l] + Mi[j * 3 + 1] * S[3 + l] + Mi[j * 3 + 2] * S[6 + l];
        for (int j = 0; j < 3; ++j)
            for (int l = 0; l < 3; ++l)
                F[j * 3 + l] = tmp[j * 3] * Mi[l] + tmp[j * 3 + 1] * Mi[3 + l] + tmp[j * 3 + 2] * Mi[6 + l];
        constexpr int PV[6] = {0, 1, 2, 1, 0, 0};
        constexpr int PP[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
        for (int pr = 0; pr < 6; ++pr) {
            const int v = PV[pr], p = PP[pr];
#pragma unroll
            for (int q = 0; q < 3; ++q) acc[3 * pr + q] += -T[q] * Mi[v * 3 + p] + z[q] * F[v * 3 + p];
        }
    }
    // 2 (pi / Q) / (8 pi^2) = 1 / (4 pi Q)
    const R f = R(1.0 / (4.0 * 3.14159265358979323846 * double(Q)));
#pragma unroll
    for (int i = 0; i < 18; ++i) hs[i] = acc[i] * f;
}

// Cubic medium with crystal axes along x, y, z:
// C_ijkl = C12 d_ij d_kl + C44 (d_ik d_jl + d_il d_jk) + D d_ijkl, D = C11 - C12 - 2 C44,
// so (zz)_jk = (C12 + C44) z_j z_k + (C44 |z|^2 + D z_j^2) d_jk and, for z . T = 0,
// (zT) + (Tz) = (C12 + C44) (z_j T_k + z_k T_j) + 2 D z_j T_j d_jk.
// Same integral as h_circle_sym, about a third of the arithmetic.
template <typename R>
__device__ __forceinline__ void h_circle_cubic(R c12, R c44, R D, int Q, const R Tin[3], R hs[18]) {
    R T[3] = {Tin[0], Tin[1], Tin[2]};
    int k0 = 0;
    if (fabs(T[1]) < fabs(T[k0])) k0 = 1;
    if (fabs(T[2]) < fabs(T[k0])) k0 = 2;
    R e1[3] = {R(0), R(0), R(0)};
    e1[k0] = R(1);
    R dd = e1[0] * T[0] + e1[1] * T[1] + e1[2] * T[2];
    for (int i = 0; i < 3; ++i) e1[i] -= dd * T[i];
    R nrm = R(1) / sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]);
    for (int i = 0; i < 3; ++i) e1[i] *= nrm;
    R e2[3] = {T[1] * e1[2] - T[2] * e1[1], T[2] * e1[0] - T[0] * e1[2], T[0] * e1[1] - T[1] * e1[0]};
    const R cp = c12 + c44;
    R acc[18];
#pragma unroll
    for (int i = 0; i < 18; ++i) acc[i] = 0;
    for (int k = 0; k < Q; ++k) {
        R sn, cs;
        sincospi(double(k) / double(Q), &sn, &cs);
        R z[3];
        for (int i = 0; i < 3; ++i) z[i] = cs * e1[i] + sn * e2[i];
        // M = (zz) (symmetric; |z| = 1)
        const R m00 = cp * z[0] * z[0] + c44 + D * z[0] * z[0];
        const R m11 = cp * z[1] * z[1] + c44 + D * z[1] * z[1];
        const R m22 = cp * z[2] * z[2] + c44 + D * z[2] * z[2];
        const R m01 = cp * z[0] * z[1], m02 = cp * z[0] * z[2], m12 = cp * z[1] * z[2];
        // inverse by cofactors
        const R i00 = m11 * m22 - m12 * m12, i01 = m02 * m12 - m01 * m22, i02 = m01 * m12 - m02 * m11;
        const R i11 = m00 * m22 - m02 * m02, i12 = m01 * m02 - m00 * m12, i22 = m00 * m11 - m01 * m01;
        const R idet = R(1) / (m00 * i00 + m01 * i01 + m02 * i02);
        const R Mi[9] = {i00 * idet, i01 * idet, i02 * idet, i01 * idet, i11 * idet,
                         i12 * idet, i02 * idet, i12 * idet, i22 * idet};
        // S = (zT) + (Tz)
        R S[9];
        for (int j = 0; j < 3; ++j)
            for (int l = 0; l < 3; ++l) S[j * 3 + l] = cp * (z[j] * T[l] + z[l] * T[j]);
        for (int j = 0; j < 3; ++j) S[j * 3 + j] += R(2) * D * z[j] * T[j];
        R tmp[9], F[9];
        for (int j = 0; j < 3; ++j)
            for (int l = 0; l < 3; ++l)
                tmp[j * 3 + l] = Mi[j * 3] * S[l] + Mi[j * 3 + 1] * S[3 + l] + Mi[j * 3 + 2] * S[6 + l];
        for (int j = 0; j < 3; ++j)
            for (int l = j; l < 3; ++l)
                F[j * 3 + l] = tmp[j * 3] * Mi[l] + tmp[j * 3 + 1] * Mi[3 + l] + tmp[j * 3 + 2] * Mi[6 + l];
        constexpr int PV[6] = {0, 1, 2, 1, 0, 0};
        constexpr int PP[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
        for (int pr = 0; pr < 6; ++pr) {
            const int v = PV[pr], p = PP[pr];
            const int vl = v < p ? v : p, ph = v < p ? p : v;
#pragma unroll
            for (int q = 0; q < 3; ++q) acc[3 * pr + q] += -T[q] * Mi[v * 3 + p] + z[q] * F[vl * 3 + ph];
        }
    }
    const R f = R(1.0 / (4.0 * 3.14159265358979323846 * double(Q)));
#pragma unroll
    for (int i = 0; i < 18; ++i) hs[i] = acc[i] * f;
}

// packed FP32x2 arithmetic (one instruction for two values)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// Lagrange basis ell_a(t) = prod_{b != a} (t - t_b) / (t_a - t_b) on the p
// nodes of [0, 1]: nodes = GBFMM_NODES_EQUISPACED, t_a = a / (p - 1) (Sec. 4.1
// footnote); nodes = GBFMM_NODES_CHEBYSHEV, the zeros of the Chebyshev
// polynomial T_p mapped to [0, 1], t_a = (1 - cos((2a + 1) pi / (2p))) / 2
// (the nodes of the Chebyshev FMM, Sec. 3).
__device__ __forceinline__ double cheb_node(int a, int p) {
    return 0.5 * (1.0 - cospi(double(2 * a + 1) / double(2 * p)));
}

// The nodes and the inverse denominators of the basis, made on the host in FP64 and passed by
// value (kernel parameters): one product of p factors per value.
template <typename R>
struct NodeTab {
    R t[GB_MAXP], w[GB_MAXP];
};
template <typename R>
inline NodeTab<R> make_nodes(int p, int nodes) {
    NodeTab<R> n{};
    double t[GB_MAXP];
    for (int a = 0; a < p; ++a)
        t[a] = nodes == GBFMM_NODES_CHEBYSHEV ? 0.5 * (1.0 - std::cos(M_PI * double(2 * a + 1) / double(2 * p)))
                                              : double(a) / double(p - 1);
    for (int a = 0; a < p; ++a) {
        double d = 1.0;
        for (int b = 0; b < p; ++b)
            if (b != a) d *= t[a] - t[b];
        n.t[a] = R(t[a]);
        n.w[a] = R(1.0 / d);
    }
    return n;
}
template <typename R>
__device__ __forceinline__ R lagrange_at(const NodeTab<R> &n, int p, int a, R t) {
    R v = n.w[a];
    for (int b = 0; b < p; ++b)
        if (b != a) v *= t - n.t[b];
    return v;
}

// The kernel of Sec. 2, Eq. "kernel" at separation d (FP64, 54 values
// K[ab][wr]): K = sum_k Asym[ab wr][k] h_k(d / |d|) / |d|^2, zero at d = 0.
__device__ __forceinline__ void kernel_at(const DevMaterial *mat, const double *Asym, const double d[3],
                                          double out[54]) {
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    if (r2 == 0.0) {
        for (int i = 0; i < 54; ++i) out[i] = 0.0;
        return;
    }
    const double ir = 1.0 / sqrt(r2);
    const double T[3] = {d[0] * ir, d[1] * ir, d[2] * ir};
    double hs[18];
    if (mat->mode == GBFMM_H_ISO)
        h_iso_sym<double>(mat->hc, mat->ha, T, hs);
    else if (mat->cubic)
        h_circle_cubic<double>(mat->c12, mat->c44, mat->cd, mat->Q, T, hs);
    else
        h_circle_sym<double, double>(mat->C, mat->Q, T, hs);
    const double ir2 = 1.0 / r2;
    for (int i = 0; i < 54; ++i) {
        double acc = 0.0;
        for (int k = 0; k < 18; ++k) acc += Asym[i * 18 + k] * hs[k];
        out[i] = acc * ir2;
    }
}
