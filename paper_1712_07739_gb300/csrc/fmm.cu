// The Lagrange FMM pass (Sec. 4, Algorithm 2), FP64 path:
//   P2M  W_m = sum_{y_j in leaf} L_p(ybar_m, y_j) q_j          (Eq. "far-field", source side)
//   M2M  W_m' = sum_children sum_m L_p(ybar_m', ybar_m) W_m    (parent basis at the child nodes)
//   M2L  s(xbar_l) = sum_{A in I(B)} sum_m K(xbar_l - ybar_m) W_m   (Eq. "m2l")
//   L2L  s(xbar_l') += sum_l L_p(xbar_l', xbar_l) s(xbar_l)    (parent local values at the child nodes)
//   L2P  s(x_i) = sum_l L_p(xbar_l, x_i) s(xbar_l) + near field over N(leaf)
// Nodes of a cell of edge h at corner c are c + h t_a, t_a = a/(p-1)
// (Sec. 4.1); node index m = (mz p + my) p + mx.
#include <algorithm>
#include <cmath>
#include <string>

#include "internal.cuh"
#include "kernel_math.cuh"

namespace {

inline unsigned nblk(int64_t n, int b) { return unsigned((n + b - 1) / b); }

__device__ __forceinline__ void cell_xyz(int64_t lin, int n, int &x, int &y, int &z) {
    x = int(lin % n);
    y = int((lin / n) % n);
    z = int(lin / (int64_t(n) * n));
}

// ---------------------------------------------------------------- occupancy
__global__ void k_occ_leaves(int64_t nl, const int *__restrict__ start, int64_t base, int *__restrict__ occ) {
    int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= nl) return;
    occ[base + i] = start[i + 1] - start[i];
}

// levels `top` .. 0 from level top + 1, one block (level 5 and up have blocks enough of their own)
__global__ void __launch_bounds__(1024) k_occ_top(int top, int *__restrict__ occ) {
    for (int level = top; level >= 0; --level) {
        const int n = 1 << level, nc = 2 * n;
        const int64_t cb = cell_base_d(level + 1), base = cell_base_d(level);
        for (int i = threadIdx.x; i < n * n * n; i += blockDim.x) {
            int x, y, z, s = 0;
            cell_xyz(i, n, x, y, z);
            for (int c = 0; c < 8; ++c)
                s += occ[cb + (int64_t(2 * z + (c >> 2)) * nc + (2 * y + ((c >> 1) & 1))) * nc + (2 * x + (c & 1))];
            occ[base + i] = s;
        }
        __syncthreads();
    }
}

__global__ void k_occ_up(int level, int *__restrict__ occ) {
    int n = 1 << level;
    int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= int64_t(n) * n * n) return;
    int x, y, z;
    cell_xyz(i, n, x, y, z);
    int nc = 2 * n;
    int64_t cb = cell_base_d(level + 1);
    int s = 0;
    for (int c = 0; c < 8; ++c) {
        int cx = 2 * x + (c & 1), cy = 2 * y + ((c >> 1) & 1), cz = 2 * z + (c >> 2);
        s += occ[cb + (int64_t(cz) * nc + cy) * nc + cx];
    }
    occ[cell_base_d(level) + i] = s;
}

// adaptive tree: occupancy of the children of split leaves at level L (one below the
// leaves), into occL (the level's part of the occupancy array, zeroed before); the work
// counts read it to count the children's M2L pairs
__global__ void k_fine_occ(int64_t n_fine, int L, const int *__restrict__ n_ref, const int *__restrict__ ref_leaf,
                           const int *__restrict__ child_start, int *__restrict__ occL) {
    const int64_t f = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (f >= n_fine) return;
    const int r = int(f >> 3), c = int(f & 7);
    if (r >= *n_ref) return;
    const int cnt = child_start[9 * r + c + 1] - child_start[9 * r + c];
    if (cnt == 0) return;
    const int nl = 1 << (L - 1), nf = 2 * nl;
    int x, y, z;
    cell_xyz(ref_leaf[r], nl, x, y, z);
    const int64_t lin = (int64_t(2 * z + (c >> 2)) * nf + (2 * y + ((c >> 1) & 1))) * nf + (2 * x + (c & 1));
    occL[lin] = cnt;
}

// ---------------------------------------------------------------- M2L (FP64)
// One block per target cell of levels 2..L-1; thread l owns node l's 6
// components.  Sources: the interaction list I(B) = children of the
// parent's neighbours that are not neighbours of B.  Node kernels come
// from the lattice table: K(xbar_l - ybar_m) at level `lev` is
// Klat[o (p-1) + l - m] * (2^lev / H)^2.
__global__ void k_m2l_f64(int p, int L, int lat_n, const TreeBox *__restrict__ box, const double *__restrict__ Klat,
                          const int *__restrict__ occ, const int *__restrict__ tocc, const double *__restrict__ W,
                          double *__restrict__ S) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    double *sW = reinterpret_cast<double *>(sm_raw);
    const int P3 = p * p * p;
    int64_t g = cell_base_d(2) + blockIdx.x;
    int lev = 2;
    while (lev + 1 < L && g >= cell_base_d(lev + 1)) ++lev;
    const int64_t cell = g - cell_base_d(lev);
    if (tocc[g] == 0) return;
    const int n = 1 << lev;
    int bx, by, bz;
    cell_xyz(cell, n, bx, by, bz);
    const int l = threadIdx.x;
    const bool own = l < P3;
    const int lx = l % p, ly = (l / p) % p, lz = l / (p * p);
    const int R0 = (lat_n - 1) / 2;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int nb = 0; nb < 27; ++nb) {
        const int px = bx / 2 + nb % 3 - 1, py = by / 2 + (nb / 3) % 3 - 1, pz = bz / 2 + nb / 9 - 1;
        for (int c = 0; c < 8; ++c) {
            const int ax = 2 * px + (c & 1), ay = 2 * py + ((c >> 1) & 1), az = 2 * pz + (c >> 2);
            if (ax < 0 || ay < 0 || az < 0 || ax >= n || ay >= n || az >= n) continue;
            const int ox = bx - ax, oy = by - ay, oz = bz - az;
            if (abs(ox) <= 1 && abs(oy) <= 1 && abs(oz) <= 1) continue;
            const int64_t A = cell_base_d(lev) + (int64_t(az) * n + ay) * n + ax;
            if (occ[A] == 0) continue;
            __syncthreads();
            for (int i = threadIdx.x; i < P3 * 9; i += blockDim.x) sW[i] = W[A * P3 * 9 + i];
            __syncthreads();
            if (!own) continue;
            const int Dx0 = ox * (p - 1) + lx + R0, Dy0 = oy * (p - 1) + ly + R0, Dz0 = oz * (p - 1) + lz + R0;
            for (int m = 0; m < P3; ++m) {
                const int mx = m % p, my = (m / p) % p, mz = m / (p * p);
                const double *K = Klat + ((int64_t(Dz0 - mz) * lat_n + (Dy0 - my)) * lat_n + (Dx0 - mx)) * 54;
                const double *w = sW + m * 9;
                for (int ab = 0; ab < 6; ++ab) {
                    double s = 0.0;
                    for (int wr = 0; wr < 9; ++wr) s += K[ab * 9 + wr] * w[wr];
                    acc[ab] += s;
                }
            }
        }
    }
    if (own) {
        const double sc = double(n) / box->H;
        double *Sc = S + g * int64_t(P3) * 6 + l * 6;
        for (int ab = 0; ab < 6; ++ab) Sc[ab] = acc[ab] * sc * sc;
    }
}

// ---------------------------------------------------------------- forces
struct ForceParams {
    double xi[GB_MAXG], w[GB_MAXG];
    int n;
};

__global__ void k_forces(int64_t n_segs, ForceParams fp, const double *__restrict__ nodes,
                         const int64_t *__restrict__ segs, const double *__restrict__ b, const int *__restrict__ pos,
                         const double *__restrict__ sig, double *__restrict__ f_nodes, double *__restrict__ f_seg,
                         double *__restrict__ sig_out) {
    int64_t s = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (s >= n_segs) return;
    const int64_t n0 = segs[2 * s], n1 = segs[2 * s + 1];
    double S[3], bb[3];
    for (int i = 0; i < 3; ++i) {
        S[i] = nodes[3 * n1 + i] - nodes[3 * n0 + i];
        bb[i] = b[3 * s + i];
    }
    double f1[3] = {0, 0, 0}, f2[3] = {0, 0, 0};
    for (int g = 0; g < fp.n; ++g) {
        const int i = pos[s * fp.n + g];
        const double *sg = sig + 6 * int64_t(i);
        if (sig_out)
            for (int a = 0; a < 6; ++a) sig_out[6 * (s * fp.n + g) + a] = sg[a];
        // (sigma b)_i with sigma in Voigt order xx yy zz yz xz xy
        const double sb[3] = {sg[0] * bb[0] + sg[5] * bb[1] + sg[4] * bb[2],
                              sg[5] * bb[0] + sg[1] * bb[1] + sg[3] * bb[2],
                              sg[4] * bb[0] + sg[3] * bb[1] + sg[2] * bb[2]};
        const double pk[3] = {sb[1] * S[2] - sb[2] * S[1], sb[2] * S[0] - sb[0] * S[2], sb[0] * S[1] - sb[1] * S[0]};
        const double w1 = 0.5 * fp.w[g] * 0.5 * (1.0 - fp.xi[g]);
        const double w2 = 0.5 * fp.w[g] * 0.5 * (1.0 + fp.xi[g]);
        for (int d = 0; d < 3; ++d) {
            f1[d] += w1 * pk[d];
            f2[d] += w2 * pk[d];
        }
    }
    for (int d = 0; d < 3; ++d) {
        atomicAdd(&f_nodes[3 * n0 + d], f1[d]);
        atomicAdd(&f_nodes[3 * n1 + d], f2[d]);
    }
    if (f_seg)
        for (int d = 0; d < 3; ++d) {
            f_seg[6 * s + d] = f1[d];
            f_seg[6 * s + 3 + d] = f2[d];
        }
}

__global__ void k_scatter_targets(int64_t n, const int *__restrict__ pos, const double *__restrict__ src,
                                  double *__restrict__ dst) {
    int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (k >= n) return;
    const double *s = src + 6 * int64_t(pos[k]);
    for (int a = 0; a < 6; ++a) dst[6 * k + a] = s[a];
}

}  // namespace

// points per cell at every level, from the leaf ranges
void compute_occ(gbfmm_ctx *ctx, const int *start, int *occ) {
    const int L = ctx->L;
    const int64_t nl = ctx->n_leaves;
    ++ctx->launches;
    k_occ_leaves<<<nblk(nl, 256), 256, 0, ctx->stream>>>(nl, start, cell_base(L - 1), occ);
    for (int lev = L - 2; lev > 3; --lev) {
        ++ctx->launches;
        k_occ_up<<<nblk(int64_t(1) << (3 * lev), 256), 256, 0, ctx->stream>>>(lev, occ);
    }
    ++ctx->launches;
    k_occ_top<<<1, 1024, 0, ctx->stream>>>(std::min(L - 2, 3), occ);
}

namespace {
// near pairs per target point: sources in the 27 neighbour leaves minus the
// points of its own segment that lie there
// (adaptive tree: a point of a split leaf meets, in another split leaf, the points of the
// children adjacent to its own child only)
__device__ inline bool fine_adjacent(int ox, int oy, int oz, int ca, int cb) {
    return abs(2 * ox + (cb & 1) - (ca & 1)) <= 1 && abs(2 * oy + ((cb >> 1) & 1) - ((ca >> 1) & 1)) <= 1 &&
           abs(2 * oz + (cb >> 2) - (ca >> 2)) <= 1;
}
__global__ void k_count_near(int64_t N, int L, int n_g, const int *__restrict__ start, const int *__restrict__ pleaf,
                             const int64_t *__restrict__ sid, const int *__restrict__ pos,
                             const int *__restrict__ ref_start, const int *__restrict__ child_start,
                             const int *__restrict__ pfine, unsigned long long *__restrict__ out) {
    int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    unsigned long long c = 0;
    if (i < N) {
        const int nl = 1 << (L - 1);
        int bx, by, bz;
        const int Bl = pleaf[i];
        cell_xyz(Bl, nl, bx, by, bz);
        const int fi = pfine ? pfine[i] : -1;
        for (int nb = 0; nb < 27; ++nb) {
            int ax = bx + nb % 3 - 1, ay = by + (nb / 3) % 3 - 1, az = bz + nb / 9 - 1;
            if (ax < 0 || ay < 0 || az < 0 || ax >= nl || ay >= nl || az >= nl) continue;
            int64_t A = (int64_t(az) * nl + ay) * nl + ax;
            if (fi >= 0 && A != Bl && ref_start[A + 1] > ref_start[A]) {
                const int rA = ref_start[A];
                for (int cb = 0; cb < 8; ++cb)
                    if (fine_adjacent(ax - bx, ay - by, az - bz, fi & 7, cb))
                        c += child_start[9 * rA + cb + 1] - child_start[9 * rA + cb];
            } else {
                c += start[A + 1] - start[A];
            }
        }
        const int64_t s = sid[i];
        for (int g = 0; g < n_g; ++g) {
            const int j = pos[s * n_g + g];
            int ox, oy, oz;
            cell_xyz(pleaf[j], nl, ox, oy, oz);
            if (abs(ox - bx) > 1 || abs(oy - by) > 1 || abs(oz - bz) > 1) continue;
            const int fj = pfine ? pfine[j] : -1;
            if (fi >= 0 && fj >= 0 && pleaf[j] != Bl && !fine_adjacent(ox - bx, oy - by, oz - bz, fi & 7, fj & 7))
                continue;  // not a near pair of the adaptive tree
            --c;
        }
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

// levels 2 .. Lm - 1 (Lm = L + 1 adds the adaptive tree's children)
__global__ void k_count_m2l(int L, int Lm, const int *__restrict__ occ, unsigned long long *__restrict__ out) {
    int64_t g = cell_base_d(2) + blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    unsigned long long c = 0, leaves = 0;
    if (g < cell_base_d(Lm)) {
        int lev = 2;
        while (lev + 1 < Lm && g >= cell_base_d(lev + 1)) ++lev;
        const int n = 1 << lev;
        int bx, by, bz;
        cell_xyz(g - cell_base_d(lev), n, bx, by, bz);
        if (occ[g] > 0) {
            if (lev == L - 1) leaves = 1;
            for (int nb = 0; nb < 27; ++nb) {
                const int px = bx / 2 + nb % 3 - 1, py = by / 2 + (nb / 3) % 3 - 1, pz = bz / 2 + nb / 9 - 1;
                for (int ch = 0; ch < 8; ++ch) {
                    const int ax = 2 * px + (ch & 1), ay = 2 * py + ((ch >> 1) & 1), az = 2 * pz + (ch >> 2);
                    if (ax < 0 || ay < 0 || az < 0 || ax >= n || ay >= n || az >= n) continue;
                    if (abs(bx - ax) <= 1 && abs(by - ay) <= 1 && abs(bz - az) <= 1) continue;
                    if (occ[cell_base_d(lev) + (int64_t(az) * n + ay) * n + ax] > 0) ++c;
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_down_sync(0xffffffffu, c, o);
        leaves += __shfl_down_sync(0xffffffffu, leaves, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (c) atomicAdd(out + 1, c);
        if (leaves) atomicAdd(out + 2, leaves);
    }
}
}  // namespace

int work_counts(gbfmm_ctx *ctx, int64_t *res) {
    cudaStream_t st = ctx->stream;
    unsigned long long *d = nullptr;
    CK(cudaMallocAsync(&d, 4 * sizeof(unsigned long long), st));
    CK(cudaMemsetAsync(d, 0, 4 * sizeof(unsigned long long), st));
    int *occ = ctx->d_tmp_i;
    const int L = ctx->L;
    compute_occ(ctx, ctx->d_leaf_start, occ);
    const auto &RF = ctx->rf;
    const bool fine = RF.on && L >= 3 && RF.fine_rows() > 0;
    if (fine) {  // the children of split leaves at level L
        const int64_t n_fine = RF.fine_rows();
        CK(cudaMemsetAsync(occ + cell_base(L), 0, (cell_base(L + 1) - cell_base(L)) * sizeof(int), st));
        ++ctx->launches;
        k_fine_occ<<<nblk(n_fine, 256), 256, 0, st>>>(n_fine, L, RF.ref_start + ctx->n_leaves, RF.ref_leaf,
                                                      RF.child_start, occ + cell_base(L));
    }
    ++ctx->launches;
    k_count_near<<<nblk(ctx->N, 256), 256, 0, st>>>(ctx->N, L, ctx->opt.n_gauss, ctx->d_leaf_start, ctx->d_pleaf,
                                                     ctx->d_sid, ctx->d_pos, fine ? RF.ref_start : nullptr,
                                                     RF.child_start, fine ? RF.pfine : nullptr, d);
    ++ctx->launches;
    const int Lm = fine ? L + 1 : L;
    k_count_m2l<<<nblk(cell_base(Lm) - cell_base(2), 256), 256, 0, st>>>(L, Lm, occ, d);
    unsigned long long h[4];
    CK(cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, st));
    CK(cudaFreeAsync(d, st));
    CK(cudaStreamSynchronize(st));
    res[0] = int64_t(h[0]);
    res[1] = int64_t(h[1]);
    res[2] = int64_t(h[2]);
    res[3] = ctx->N;
    return GBFMM_OK;
}

template <typename R>
int upward(gbfmm_ctx *ctx, const int *occ, R *W, int64_t n_fine);  // transfer.cu
template <typename R>
int downward(gbfmm_ctx *ctx, const int *tocc, R *S, int64_t n_fine);

void timer_mark(gbfmm_ctx *ctx) {
    if (!ctx->timer.on || ctx->timer.n >= 16) return;
    cudaEventRecord(ctx->timer.ev[ctx->timer.n++], ctx->stream);
}

int near_prepare(gbfmm_ctx *ctx);                                             // near.cu
int near_alloc(gbfmm_ctx *ctx);                                               // near.cu
int near_run(gbfmm_ctx *ctx, bool free_targets, int64_t n_t, double *sig);   // near.cu

// Runs the pass.  free_targets: targets are the sorted free points of
// targets_sort (no segment exclusion), else the sorted Gauss points.
int fmm_pass(gbfmm_ctx *ctx, bool free_targets, int64_t n_t) {
    cudaStream_t st = ctx->stream;
    const int p = ctx->opt.p, L = ctx->L, P3 = p * p * p;
    int *occ = ctx->d_tmp_i;                 // [n_cells] sources per cell
    int *tocc = free_targets ? occ + ctx->n_cells : occ;

    timer_mark(ctx);
    if (int rc = near_prepare(ctx)) return rc;
    compute_occ(ctx, ctx->d_leaf_start, occ);
    if (free_targets) compute_occ(ctx, ctx->d_t_start, tocc);
    CK(cudaGetLastError());
    timer_mark(ctx);
    if (int rc = upward<double>(ctx, occ, ctx->d_W, 0)) return rc;
    timer_mark(ctx);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CK(cudaStreamIsCapturing(st, &cap));
    if (L >= 3 && ctx->opt.m2l_fft && cap == cudaStreamCaptureStatusNone) {
        if (int rc = m2l_fft_run(ctx, occ, tocc)) return rc;
    } else if (L >= 3) {
        const int64_t ncell = ctx->n_cells - cell_base(2);
        const int bd = ((P3 + 31) / 32) * 32;
        ++ctx->launches;
        k_m2l_f64<<<unsigned(ncell), bd, P3 * 9 * sizeof(double), st>>>(p, L, ctx->lat_n, ctx->d_box, ctx->d_Klat,
                                                                         occ, tocc, ctx->d_W, ctx->d_S);
        CK(cudaGetLastError());
    }
    timer_mark(ctx);
    if (int rc = downward<double>(ctx, tocc, ctx->d_S, 0)) return rc;
    timer_mark(ctx);
    if (int rc = near_run(ctx, free_targets, n_t, free_targets ? ctx->d_t_sig : ctx->d_sig)) return rc;
    timer_mark(ctx);
    return GBFMM_OK;
}

int forces_from_stress(gbfmm_ctx *ctx, double *f_nodes, double *f_seg, double *sigma_pts) {
    ForceParams fp{};
    fp.n = ctx->opt.n_gauss;
    for (int i = 0; i < fp.n; ++i) {
        fp.xi[i] = ctx->gauss_xi[i];
        fp.w[i] = ctx->gauss_w[i];
    }
    CK(cudaMemsetAsync(f_nodes, 0, ctx->n_nodes * 3 * sizeof(double), ctx->stream));
    ++ctx->launches;
    k_forces<<<nblk(ctx->n_segs, 128), 128, 0, ctx->stream>>>(ctx->n_segs, fp, ctx->node_xyz, ctx->seg_nodes,
                                                               ctx->burgers, ctx->d_pos, ctx->d_sig, f_nodes, f_seg,
                                                               sigma_pts);
    CK(cudaGetLastError());
    timer_mark(ctx);
    return GBFMM_OK;
}

int targets_scatter(gbfmm_ctx *ctx, int64_t n_t, double *sigma) {
    ++ctx->launches;
    k_scatter_targets<<<nblk(n_t, 256), 256, 0, ctx->stream>>>(n_t, ctx->d_t_pos, ctx->d_t_sig, sigma);
    CK(cudaGetLastError());
    return GBFMM_OK;
}

int fmm_kernel_attrs(gbfmm_ctx *ctx) {
    const int P3 = ctx->opt.p * ctx->opt.p * ctx->opt.p;
    CK(cudaFuncSetAttribute(k_m2l_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, int(P3 * 9 * sizeof(double))));
    return GBFMM_OK;
}

int mixed_alloc(gbfmm_ctx *ctx) {
    const int64_t nc = ctx->n_cells;
    const int P3 = ctx->opt.p * ctx->opt.p * ctx->opt.p;
    if (int rc = grow_dev(ctx, ctx->mx_cap_cells, nc,
                          {{(void **)&ctx->d_Wf, nc * P3 * 9 * sizeof(float)},
                           {(void **)&ctx->d_Sf, nc * P3 * 6 * sizeof(float)}},
                          "mixed-pass cells"))
        return rc;
    if (int rc = near_alloc(ctx)) return rc;
    if (!ctx->tc.ready_ops) {
        int rc = m2l_tc_setup(ctx);
        if (rc) return rc;
    }
    return m2l_tc_prepare(ctx);
}

int mixed_pass(gbfmm_ctx *ctx, bool free_targets, int64_t n_t) {
    if (!ctx->tc.ready_ops) {  // the medium changed after the build
        if (int rc = m2l_tc_setup(ctx)) return rc;
        if (int rc = m2l_tc_prepare(ctx)) return rc;
    }
    const bool t64 = ctx->opt.precision == GBFMM_MIXED_F64T;  // FP64 P2M, M2M, L2L, L2P
    const int L = ctx->L;
    int *occ = ctx->d_tmp_i;
    int *tocc = free_targets ? occ + ctx->n_cells : occ;
    // adaptive tree: the children of split leaves take part in nodal-force passes (free
    // targets keep the uniform tree, whose near field covers whole leaves)
    auto &RF = ctx->rf;
    const int64_t n_fine = RF.fine_rows();
    const bool fine = RF.on && !free_targets && L >= 3 && n_fine > 0;
    timer_mark(ctx);
    if (int rc = near_prepare(ctx)) return rc;
    compute_occ(ctx, ctx->d_leaf_start, occ);
    if (free_targets) compute_occ(ctx, ctx->d_t_start, tocc);
    CK(cudaGetLastError());
    timer_mark(ctx);
    if (int rc = t64 ? upward<double>(ctx, occ, ctx->d_W, 0) : upward<float>(ctx, occ, ctx->d_Wf, fine ? n_fine : 0))
        return rc;
    timer_mark(ctx);
    if (L >= 3) {
        int rc = m2l_tc_run(ctx, ctx->d_Wf, t64 ? ctx->d_W : nullptr, occ, tocc, ctx->d_Sf, t64 ? ctx->d_S : nullptr,
                            fine, n_t);
        if (rc) return rc;
    }
    timer_mark(ctx);
    // (the children's local values, the level-L M2L, were written by m2l_tc_run)
    if (int rc = t64 ? downward<double>(ctx, tocc, ctx->d_S, 0) : downward<float>(ctx, tocc, ctx->d_Sf, fine ? n_fine : 0))
        return rc;
    timer_mark(ctx);
    if (int rc = near_run(ctx, free_targets, n_t, free_targets ? ctx->d_t_sig : ctx->d_sig)) return rc;
    timer_mark(ctx);
    return GBFMM_OK;
}
