// Interpolation stages of Algorithm 2 around the M2L:
//   P2M  W_m = sum_{y_j in leaf} L_p(ybar_m, y_j) q_j           (Eq. "far-field", source side)
//   M2M  W_m' = sum_children sum_m L_p(ybar_m', ybar_m) W_m     (parent basis at the child nodes)
//   L2L  s(xbar_l') += sum_l L_p(xbar_l', xbar_l) s(xbar_l)     (parent local values at the child nodes)
// on p^3 nodes per cell, m = (mz p + my) p + mx, 9 strength or 6 stress components per node.
// Every kernel is compiled for each order p = 2 .. 8: the node indices are divisions by constants
// and the loops over nodes unroll (with p a run-time value the index arithmetic was the time:
// 1M segments, p = 7, FP32: P2M 3.5, M2M 4.8, L2L 4.4 + 1.5 ms).
#include <cmath>

#include "internal.cuh"
#include "kernel_math.cuh"

namespace {

__device__ __forceinline__ void cell_xyz(int64_t lin, int n, int &x, int &y, int &z) {
    x = int(lin % n);
    y = int((lin / n) % n);
    z = int(lin / (int64_t(n) * n));
}

// M[c][A][a] = ell_A((c + t_a) / 2): the parent's basis function A at node a of child c
template <typename R>
struct Transfer {
    R M[2][GB_MAXP][GB_MAXP];
};

template <typename R>
Transfer<R> make_transfer(int p, int nodes) {
    const NodeTab<double> n = make_nodes<double>(p, nodes);
    Transfer<R> t{};
    for (int c = 0; c < 2; ++c)
        for (int A = 0; A < p; ++A)
            for (int a = 0; a < p; ++a) {
                const double x = (c + n.t[a]) / 2.0;
                double v = 1.0;
                for (int b = 0; b < p; ++b)
                    if (b != A) v *= (x - n.t[b]) / (n.t[A] - n.t[b]);
                t.M[c][A][a] = R(v);
            }
    return t;
}

// ---------------------------------------------------------------- P2M
// One block per cell.  A thread owns one (y, z) row of nodes -- p nodes x 9 components in
// registers, so a staged point costs it 9 p + 10 multiply-adds for two basis values, the x basis
// and nine strengths -- and one of the block's 256 / 32 (p <= 5) or 256 / 64 groups, which take
// every G-th point; the groups are added in order at the end.  The local coordinate of a point is
// formed in FP64; the basis and sums in R.
constexpr int kP2MThreads = 256, kP2MPoints = 64;
template <int P, typename R>
constexpr size_t p2m_smem() { return (kP2MPoints * (3 * GB_MAXP + 12) + P * P * P * 9) * sizeof(R); }

template <int P, typename R>
__device__ void p2m_range(const NodeTab<R> &nt, int b, int e, const double c0[3], double ih,
                          const double *__restrict__ y, const double *__restrict__ q, R *__restrict__ Wc) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    R *sb = reinterpret_cast<R *>(sm_raw);         // [points][3][8]
    R *sq = sb + kP2MPoints * 3 * GB_MAXP;         // [points][12]
    R *sW = sq + kP2MPoints * 12;                  // [9 p^3]
    constexpr int PP = P * P <= 32 ? 32 : 64, G = kP2MThreads / PP, NV = P * P * P * 9;
    const int g = threadIdx.x / PP, r = threadIdx.x % PP, my = r % P, mz = r / P;
    const bool on = r < P * P;
    R acc[P][9];
#pragma unroll
    for (int x = 0; x < P; ++x)
#pragma unroll
        for (int i = 0; i < 9; ++i) acc[x][i] = R(0);
    for (int j0 = b; j0 < e; j0 += kP2MPoints) {
        const int nj = min(kP2MPoints, e - j0);
        __syncthreads();
        for (int t = threadIdx.x; t < nj * 3 * P; t += kP2MThreads) {
            const int j = t / (3 * P), d = (t / P) % 3, a = t % P;
            const double c = d == 0 ? c0[0] : d == 1 ? c0[1] : c0[2];
            sb[(j * 3 + d) * GB_MAXP + a] = lagrange_at<R>(nt, P, a, R((y[3 * int64_t(j0 + j) + d] - c) * ih));
        }
        for (int t = threadIdx.x; t < nj * 9; t += kP2MThreads) sq[(t / 9) * 12 + t % 9] = R(q[9 * int64_t(j0) + t]);
        __syncthreads();
        if (on)
            for (int j = g; j < nj; j += G) {
                const R *bj = sb + j * 3 * GB_MAXP;
                const R w = bj[GB_MAXP + my] * bj[2 * GB_MAXP + mz];
                R tq[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) tq[i] = w * sq[j * 12 + i];
#pragma unroll
                for (int x = 0; x < P; ++x) {
                    const R bx = bj[x];
#pragma unroll
                    for (int i = 0; i < 9; ++i) acc[x][i] += bx * tq[i];
                }
            }
    }
    for (int k = 0; k < G; ++k) {
        __syncthreads();
        if (on && g == k)
#pragma unroll
            for (int x = 0; x < P; ++x)
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    R &w = sW[(r * P + x) * 9 + i];
                    w = k == 0 ? acc[x][i] : w + acc[x][i];
                }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < NV; t += kP2MThreads) Wc[t] = sW[t];
}

template <int P, typename R>
__global__ void __launch_bounds__(kP2MThreads) k_p2m(const __grid_constant__ NodeTab<R> nt, int L,
                                                     const TreeBox *__restrict__ box, const int *__restrict__ start,
                                                     const double *__restrict__ y, const double *__restrict__ q,
                                                     R *__restrict__ W) {
    const int64_t leaf = blockIdx.x;
    const int nl = 1 << (L - 1);
    constexpr int NV = P * P * P * 9;
    R *Wc = W + (cell_base_d(L - 1) + leaf) * int64_t(NV);
    const int b = start[leaf], e = start[leaf + 1];
    if (b == e) {
        for (int i = threadIdx.x; i < NV; i += kP2MThreads) Wc[i] = R(0);
        return;
    }
    int cx, cy, cz;
    cell_xyz(leaf, nl, cx, cy, cz);
    const double h = box->H / nl, ih = double(nl) / box->H;
    const double c0[3] = {box->origin[0] + cx * h, box->origin[1] + cy * h, box->origin[2] + cz * h};
    p2m_range<P, R>(nt, b, e, c0, ih, y, q, Wc);
}

// adaptive tree: P2M of the children of split leaves, one block per child cell 8 r + c
// (compact rows; empty and absent children get zeros)
template <int P, typename R>
__global__ void __launch_bounds__(kP2MThreads) k_p2m_fine(const __grid_constant__ NodeTab<R> nt, int L,
                                                          const TreeBox *__restrict__ box,
                                                          const int *__restrict__ n_ref,
                                                          const int *__restrict__ ref_leaf,
                                                          const int *__restrict__ child_start,
                                                          const double *__restrict__ y, const double *__restrict__ q,
                                                          R *__restrict__ W7) {
    const int64_t f = blockIdx.x;
    const int r = int(f >> 3), c = int(f & 7);
    constexpr int NV = P * P * P * 9;
    R *Wc = W7 + f * int64_t(NV);
    int b = 0, e = 0;
    if (r < *n_ref) {
        b = child_start[9 * r + c];
        e = child_start[9 * r + c + 1];
    }
    if (b == e) {
        for (int i = threadIdx.x; i < NV; i += kP2MThreads) Wc[i] = R(0);
        return;
    }
    const int nl = 1 << (L - 1);
    int cx, cy, cz;
    cell_xyz(ref_leaf[r], nl, cx, cy, cz);
    const double h = box->H / (2 * nl), ih = double(2 * nl) / box->H;
    const double c0[3] = {box->origin[0] + (2 * cx + (c & 1)) * h, box->origin[1] + (2 * cy + ((c >> 1) & 1)) * h,
                          box->origin[2] + (2 * cz + (c >> 2)) * h};
    p2m_range<P, R>(nt, b, e, c0, ih, y, q, Wc);
}

// ---------------------------------------------------------------- M2M
// Parent weights at `level` from its 8 children at level + 1, the children merged one axis at a
// time: for each child row (oy, oz) the x transfer sums over both x children (2 p terms), then the
// y transfer over both y halves, then the z transfer over both z halves -- 14 p multiply-adds per
// parent value instead of 24 p for eight separate tensor-product transfers.  Shared memory: 4 x 9
// p^3 values (x-merged rows of one z half, x- and y-merged halves).
template <int P, typename R>
__global__ void __launch_bounds__(256) k_m2m(int level, const __grid_constant__ Transfer<R> tr,
                                             const int *__restrict__ occ, R *__restrict__ W) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    R *tx = reinterpret_cast<R *>(sm_raw);
    __shared__ R Ms[2][GB_MAXP][GB_MAXP];
    __shared__ int64_t s_ch[8];
    constexpr int NV = P * P * P * 9;
    R *u = tx + 2 * NV;
    const int n = 1 << level, nc = 2 * n;
    const int64_t cell = blockIdx.x;
    R *Wp = W + (cell_base_d(level) + cell) * int64_t(NV);
    if (occ[cell_base_d(level) + cell] == 0) {
        for (int i = threadIdx.x; i < NV; i += 256) Wp[i] = R(0);
        return;
    }
    int x, y, z;
    cell_xyz(cell, n, x, y, z);
    for (int i = threadIdx.x; i < 2 * GB_MAXP * GB_MAXP; i += 256) (&Ms[0][0][0])[i] = (&tr.M[0][0][0])[i];
    if (threadIdx.x < 8) {
        const int ox = threadIdx.x & 1, oy = (threadIdx.x >> 1) & 1, oz = threadIdx.x >> 2;
        const int64_t ch = cell_base_d(level + 1) + (int64_t(2 * z + oz) * nc + (2 * y + oy)) * nc + (2 * x + ox);
        s_ch[threadIdx.x] = occ[ch] > 0 ? ch * int64_t(NV) : int64_t(-1);
    }
    __syncthreads();
    for (int oz = 0; oz < 2; ++oz) {
        // x: tx[oy][((c p + b) p + A) 9 + k] = sum_ox sum_a M[ox][A][a] W_(ox,oy,oz)[((c p + b) p + a) 9 + k]
        for (int t = threadIdx.x; t < 2 * NV; t += 256) {
            const int oy = t / NV, r = t - oy * NV;
            const int k = r % 9, node = r / 9, A = node % P, bc = node / P;
            R s = R(0);
#pragma unroll
            for (int ox = 0; ox < 2; ++ox) {
                const int64_t base = s_ch[ox + 2 * oy + 4 * oz];
                if (base < 0) continue;
                const R *Wc = W + base + bc * (P * 9) + k;
#pragma unroll
                for (int a = 0; a < P; ++a) s += Ms[ox][A][a] * Wc[9 * a];
            }
            tx[t] = s;
        }
        __syncthreads();
        // y: u[oz][((c p + B) p + A) 9 + k] = sum_oy sum_b M[oy][B][b] tx[oy][((c p + b) p + A) 9 + k]
        for (int r = threadIdx.x; r < NV; r += 256) {
            const int kA = r % (9 * P), B = (r / (9 * P)) % P, c = r / (9 * P * P);
            R s = R(0);
#pragma unroll
            for (int oy = 0; oy < 2; ++oy)
#pragma unroll
                for (int b = 0; b < P; ++b) s += Ms[oy][B][b] * tx[oy * NV + (c * P + b) * (P * 9) + kA];
            u[oz * NV + r] = s;
        }
        __syncthreads();
    }
    // z: W[((C p + B) p + A) 9 + k] = sum_oz sum_c M[oz][C][c] u[oz][((c p + B) p + A) 9 + k]
    for (int r = threadIdx.x; r < NV; r += 256) {
        const int kAB = r % (9 * P * P), C = r / (9 * P * P);
        R s = R(0);
#pragma unroll
        for (int oz = 0; oz < 2; ++oz)
#pragma unroll
            for (int c = 0; c < P; ++c) s += Ms[oz][C][c] * u[oz * NV + c * (P * P * 9) + kAB];
        Wp[r] = s;
    }
}

// ---------------------------------------------------------------- L2L
// Child locals at `level` += their parent's, interpolated, one block per parent at level - 1
// producing all eight children axis by axis: the parent's values are read once, the x transfer
// gives both x halves, the y transfer the four (ox, oy) quarters, the z transfer the eight
// children -- 14 p multiply-adds per child value on average instead of 24 p.  Shared memory: 7 x 6
// p^3 values.
template <int P, typename R>
__global__ void __launch_bounds__(256) k_l2l(int level, const __grid_constant__ Transfer<R> tr,
                                             const int *__restrict__ tocc, R *__restrict__ S) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    R *in = reinterpret_cast<R *>(sm_raw);
    __shared__ R Ms[2][GB_MAXP][GB_MAXP];
    __shared__ int64_t s_ch[8];
    constexpr int NV = P * P * P * 6;
    R *tx = in + NV, *ty = tx + 2 * NV;
    const int np = 1 << (level - 1), n = 2 * np;
    const int64_t par = blockIdx.x;
    if (tocc[cell_base_d(level - 1) + par] == 0) return;
    int x, y, z;
    cell_xyz(par, np, x, y, z);
    if (threadIdx.x < 8) {
        const int ox = threadIdx.x & 1, oy = (threadIdx.x >> 1) & 1, oz = threadIdx.x >> 2;
        const int64_t ch = cell_base_d(level) + (int64_t(2 * z + oz) * n + (2 * y + oy)) * n + (2 * x + ox);
        s_ch[threadIdx.x] = tocc[ch] > 0 ? ch * int64_t(NV) : int64_t(-1);
    }
    for (int i = threadIdx.x; i < 2 * GB_MAXP * GB_MAXP; i += 256) (&Ms[0][0][0])[i] = (&tr.M[0][0][0])[i];
    const R *Sp = S + (cell_base_d(level - 1) + par) * int64_t(NV);
    for (int i = threadIdx.x; i < NV; i += 256) in[i] = Sp[i];
    __syncthreads();
    // x: tx[ox][((c p + b) p + A) 6 + k] = sum_a M[ox][a][A] in[((c p + b) p + a) 6 + k]
    for (int t = threadIdx.x; t < 2 * NV; t += 256) {
        const int ox = t / NV, r = t - ox * NV;
        const int k = r % 6, node = r / 6, A = node % P, bc = node / P;
        R s = R(0);
#pragma unroll
        for (int a = 0; a < P; ++a) s += Ms[ox][a][A] * in[(bc * P + a) * 6 + k];
        tx[t] = s;
    }
    __syncthreads();
    // y: ty[ox + 2 oy][((c p + B) p + A) 6 + k] = sum_b M[oy][b][B] tx[ox][((c p + b) p + A) 6 + k]
    for (int t = threadIdx.x; t < 4 * NV; t += 256) {
        const int q = t / NV, r = t - q * NV, ox = q & 1, oy = q >> 1;
        const int kA = r % (6 * P), B = (r / (6 * P)) % P, c = r / (6 * P * P);
        R s = R(0);
#pragma unroll
        for (int b = 0; b < P; ++b) s += Ms[oy][b][B] * tx[ox * NV + (c * P + b) * (P * 6) + kA];
        ty[t] = s;
    }
    __syncthreads();
    // z: child (ox, oy, oz) += sum_c M[oz][c][C] ty[ox + 2 oy][((c p + B) p + A) 6 + k]
    for (int t = threadIdx.x; t < 8 * NV; t += 256) {
        const int ci = t / NV, r = t - ci * NV, oz = ci >> 2;
        const int64_t base = s_ch[ci];
        if (base < 0) continue;
        const int kAB = r % (6 * P * P), C = r / (6 * P * P);
        const R *tq = ty + (ci & 3) * NV;
        R s = R(0);
#pragma unroll
        for (int c = 0; c < P; ++c) s += Ms[oz][c][C] * tq[c * (P * P * 6) + kAB];
        S[base + r] += s;
    }
}

// adaptive tree: children's local values += their split parent's, interpolated, one block per
// child cell 8 r + c that holds points
template <int P, typename R>
__global__ void __launch_bounds__(256) k_l2l_fine(int L, const __grid_constant__ Transfer<R> tr,
                                                  const int *__restrict__ n_ref, const int *__restrict__ ref_leaf,
                                                  const int *__restrict__ child_start, const R *__restrict__ S,
                                                  R *__restrict__ S7) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    R *in = reinterpret_cast<R *>(sm_raw);
    __shared__ R Ms[2][GB_MAXP][GB_MAXP];
    const int64_t f = blockIdx.x;
    const int r = int(f >> 3), ch = int(f & 7);
    if (r >= *n_ref || child_start[9 * r + ch + 1] == child_start[9 * r + ch]) return;
    constexpr int NV = P * P * P * 6;
    R *t1 = in + NV;
    for (int i = threadIdx.x; i < 2 * GB_MAXP * GB_MAXP; i += 256) (&Ms[0][0][0])[i] = (&tr.M[0][0][0])[i];
    const R *Sp = S + (cell_base_d(L - 1) + ref_leaf[r]) * int64_t(NV);
    for (int i = threadIdx.x; i < NV; i += 256) in[i] = Sp[i];
    __syncthreads();
    const R(*Mx)[GB_MAXP] = Ms[ch & 1], (*My)[GB_MAXP] = Ms[(ch >> 1) & 1], (*Mz)[GB_MAXP] = Ms[ch >> 2];
    for (int t = threadIdx.x; t < NV; t += 256) {
        const int k = t % 6, node = t / 6, A = node % P, bc = node / P;
        R s = R(0);
#pragma unroll
        for (int a = 0; a < P; ++a) s += Mx[a][A] * in[(bc * P + a) * 6 + k];
        t1[t] = s;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < NV; t += 256) {
        const int kA = t % (6 * P), B = (t / (6 * P)) % P, c = t / (6 * P * P);
        R s = R(0);
#pragma unroll
        for (int b = 0; b < P; ++b) s += My[b][B] * t1[(c * P + b) * (P * 6) + kA];
        in[t] = s;
    }
    __syncthreads();
    R *out = S7 + f * int64_t(NV);
    for (int t = threadIdx.x; t < NV; t += 256) {
        const int kAB = t % (6 * P * P), C = t / (6 * P * P);
        R s = R(0);
#pragma unroll
        for (int c = 0; c < P; ++c) s += Mz[c][C] * in[c * (P * P * 6) + kAB];
        out[t] += s;
    }
}

template <int P, typename R>
int upward_p(gbfmm_ctx *ctx, const int *occ, R *W, int64_t n_fine) {
    const int L = ctx->L;
    cudaStream_t st = ctx->stream;
    const NodeTab<R> nt = make_nodes<R>(P, ctx->opt.nodes);
    const Transfer<R> tr = make_transfer<R>(P, ctx->opt.nodes);
    const size_t sm = p2m_smem<P, R>(), smm = size_t(4) * P * P * P * 9 * sizeof(R);
    CK(cudaFuncSetAttribute(k_p2m<P, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm)));
    CK(cudaFuncSetAttribute(k_m2m<P, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smm)));
    ++ctx->launches;
    k_p2m<P, R><<<unsigned(ctx->n_leaves), kP2MThreads, sm, st>>>(nt, L, ctx->d_box, ctx->d_leaf_start, ctx->d_y,
                                                                  ctx->d_q, W);
    for (int lev = L - 2; lev >= 2; --lev) {
        ++ctx->launches;
        k_m2m<P, R><<<unsigned(int64_t(1) << (3 * lev)), 256, smm, st>>>(lev, tr, occ, W);
    }
    if constexpr (sizeof(R) == 4)
        if (n_fine > 0) {
            // the children of split leaves
            const auto &RF = ctx->rf;
            CK(cudaFuncSetAttribute(k_p2m_fine<P, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm)));
            ++ctx->launches;
            k_p2m_fine<P, R><<<unsigned(n_fine), kP2MThreads, sm, st>>>(nt, L, ctx->d_box, RF.ref_start + ctx->n_leaves,
                                                                        RF.ref_leaf, RF.child_start, ctx->d_y, ctx->d_q,
                                                                        RF.W7);
        }
    CK(cudaGetLastError());
    return GBFMM_OK;
}

template <int P, typename R>
int downward_p(gbfmm_ctx *ctx, const int *tocc, R *S, int64_t n_fine) {
    const int L = ctx->L;
    cudaStream_t st = ctx->stream;
    const Transfer<R> tr = make_transfer<R>(P, ctx->opt.nodes);
    const size_t sm = size_t(7) * P * P * P * 6 * sizeof(R);
    CK(cudaFuncSetAttribute(k_l2l<P, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm)));
    for (int lev = 3; lev <= L - 1; ++lev) {
        ++ctx->launches;
        k_l2l<P, R><<<unsigned(int64_t(1) << (3 * (lev - 1))), 256, sm, st>>>(lev, tr, tocc, S);
    }
    if constexpr (sizeof(R) == 4)
        if (n_fine > 0) {
            const auto &RF = ctx->rf;
            ++ctx->launches;
            k_l2l_fine<P, R><<<unsigned(n_fine), 256, size_t(2) * P * P * P * 6 * sizeof(R), st>>>(
                L, tr, RF.ref_start + ctx->n_leaves, RF.ref_leaf, RF.child_start, S, RF.S7);
        }
    CK(cudaGetLastError());
    return GBFMM_OK;
}

}  // namespace

// P2M and M2M into W (levels L-1 .. 2); n_fine > 0: the children of split leaves too (FP32)
template <typename R>
int upward(gbfmm_ctx *ctx, const int *occ, R *W, int64_t n_fine) {
    switch (ctx->opt.p) {
        case 2: return upward_p<2, R>(ctx, occ, W, n_fine);
        case 3: return upward_p<3, R>(ctx, occ, W, n_fine);
        case 4: return upward_p<4, R>(ctx, occ, W, n_fine);
        case 5: return upward_p<5, R>(ctx, occ, W, n_fine);
        case 6: return upward_p<6, R>(ctx, occ, W, n_fine);
        case 7: return upward_p<7, R>(ctx, occ, W, n_fine);
        default: return upward_p<8, R>(ctx, occ, W, n_fine);
    }
}
template int upward<float>(gbfmm_ctx *, const int *, float *, int64_t);
template int upward<double>(gbfmm_ctx *, const int *, double *, int64_t);

// L2L of levels 3 .. L-1; n_fine > 0: into the children of split leaves too (FP32)
template <typename R>
int downward(gbfmm_ctx *ctx, const int *tocc, R *S, int64_t n_fine) {
    switch (ctx->opt.p) {
        case 2: return downward_p<2, R>(ctx, tocc, S, n_fine);
        case 3: return downward_p<3, R>(ctx, tocc, S, n_fine);
        case 4: return downward_p<4, R>(ctx, tocc, S, n_fine);
        case 5: return downward_p<5, R>(ctx, tocc, S, n_fine);
        case 6: return downward_p<6, R>(ctx, tocc, S, n_fine);
        case 7: return downward_p<7, R>(ctx, tocc, S, n_fine);
        default: return downward_p<8, R>(ctx, tocc, S, n_fine);
    }
}
template int downward<float>(gbfmm_ctx *, const int *, float *, int64_t);
template int downward<double>(gbfmm_ctx *, const int *, double *, int64_t);
