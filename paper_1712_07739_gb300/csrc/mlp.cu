// Learned angular factor: a small network T -> h_vpq(T) (the 27 components
// of R^2 dG_vp/dx_q, Sec. 2), trained on the GPU against the plain
// unit-circle evaluator and used in place of it where its error is small.
//
// Network (BF16 weights, FP32 accumulation): x = s T with s = +-1 putting T in
// the upper half-space (h is odd, so h(T) = s h(x) holds exactly), then
// 3 -> 128 -> 128 -> 128 -> 27 with SiLU activations; the output is in units
// of a per-component scale (RMS of the training labels).  Parameters are one
// flat FP32 master vector (W1 [128x3], b1, W2 [128x128], b2, W3, b3,
// W4 [32x128] (rows 27..31 stay zero), b4 [32]) with a BF16 copy for compute.
//
// Evaluation is one kernel: a warp takes 16 directions through all four layers in registers, the
// weights in shared memory (mlp_warp.cuh), so a direction moves 12 bytes in and 108 out instead of
// its 384 activations.  Training: Adam on the mean-squared error in scaled units; a step's forward
// and backward chain is the same kernel form, the weight gradients (sums over the batch) one split
// product and one ordered sum.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "internal.cuh"
#include "kernel_math.cuh"
#include "mlp_warp.cuh"

namespace {

typedef __nv_bfloat16 bf16;

using mlpw::NPAR;
using mlpw::OFF_B1;
using mlpw::OFF_B2;
using mlpw::OFF_B3;
using mlpw::OFF_B4;
using mlpw::OFF_W1;
using mlpw::OFF_W2;
using mlpw::OFF_W3;
using mlpw::OFF_W4;

inline unsigned nblk(int64_t n, int b) { return unsigned(std::min<int64_t>((n + b - 1) / b, 1 << 22)); }

// Bound by the weight fragments' way out of shared memory (its pipe 83 % busy, the tensor pipe 37 %):
// sixteen directions per warp at 128 registers, two blocks of eight warps per SM.  32 directions per
// warp would halve the fragment loads but leave 8 to 12 warps an SM, too few to cover the chain
// (254 us).  1,000,003 directions: 224 us, 2,561 us as seven kernels per 262,144 directions with the
// activations in memory.  Blocks stride over the tiles: the weights load once per block.
constexpr int kEvalWarps = 8;
struct EvalSmem {
    mlpw::Weights w;
    float out[kEvalWarps][16 * 27];
};
__global__ void __launch_bounds__(32 * kEvalWarps, 2)
    k_mlp_eval(int64_t n, const float *__restrict__ dirs, const bf16 *__restrict__ th, const float *__restrict__ th32,
               const float *__restrict__ scale, float *__restrict__ h) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    EvalSmem &sm = *reinterpret_cast<EvalSmem *>(sm_raw);
    mlpw::load(sm.w, th, th32, scale);
    __syncthreads();
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, g = lane >> 2, t = lane & 3;
    const int64_t tiles = (n + 15) / 16;
    // neighbouring tiles to different blocks: a small call spreads over the SMs
    for (int64_t tile = int64_t(warp) * gridDim.x + blockIdx.x; tile < tiles; tile += int64_t(gridDim.x) * kEvalWarps) {
        float d[2][3], s[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int64_t b = min(tile * 16 + g + 8 * r, n - 1);  // rows past the end repeat the last
            const float x = __ldg(dirs + 3 * b), y = __ldg(dirs + 3 * b + 1), z = __ldg(dirs + 3 * b + 2);
            s[r] = mlpw::half_space_sign(x, y, z);
            d[r][0] = s[r] * x, d[r][1] = s[r] * y, d[r][2] = s[r] * z;
        }
        uint32_t a[8][4];
        float z[16][4];
        mlpw::first(sm.w, d[0], d[1], z, t);
        mlpw::silu_all(z);
        mlpw::pack_a<8>(a, z);
        mlpw::layer<16, 8, false>(sm.w.W2, a, z, lane);
        mlpw::add_bias<16>(sm.w.b2, z, t);
        mlpw::silu_all(z);
        mlpw::pack_a<8>(a, z);
        mlpw::layer<16, 8, false>(sm.w.W3, a, z, lane);
        mlpw::add_bias<16>(sm.w.b3, z, t);
        mlpw::silu_all(z);
        mlpw::pack_a<8>(a, z);
        mlpw::layer<4, 8, false>(sm.w.W4, a, z, lane);
        mlpw::add_bias<4>(sm.w.b4, z, t);
        // scaled output -> h (sign of the half-space restored), rows put together in shared memory
        float *out = sm.out[warp];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 8 * nt + 2 * t + (j & 1);
                if (c < 27) out[(g + 8 * (j >> 1)) * 27 + c] = s[j >> 1] * sm.w.scale[c] * z[nt][j];
            }
        __syncwarp();
        const int rows = int(min(int64_t(16), n - tile * 16));
        for (int i = lane; i < rows * 27; i += 32) h[tile * 16 * 27 + i] = out[i];
        __syncwarp();
    }
}

// Forward and backward chain of one batch.  A warp takes 16 samples through the network and back
// in registers (the transposed products read the same weights by transposing loads) and leaves
// what the weight gradients read: inputs x, activations a1 .. a3 and the gradients of the
// pre-activations g1 .. g3, go, in BF16 rows, g1 also in FP32.  The pre-activations go through
// memory in the lane's own order.  loss = mean_{b,c} (o - s y / scale)^2, one partial per tile: the
// FP32 terms are summed in FP64 (13 additions a lane and tile), so the loss is theirs to its own
// FP32 rounding in whatever order the tiles run (sums of 8,192 samples in FP32: up to 2e-6 off).
// Two warps a block: a batch of 8,192 is 512 tiles, about three warps for every SM, whose serial
// chain is the time.  The whole gradient of 8,192 samples: 78 us, 1,926 us as 22 kernels with the
// activations in memory (this one 32 us, k_mlp_wgrad 15, k_grad_sum 8).
constexpr int kTrainWarps = 2;
struct TrainArgs {
    float *x, *z, *g32;          // [n][3], [tile][3][16][32][4], [n][128]
    double *lossp;               // [tiles]
    bf16 *a[3], *g[3], *go;      // [n][128] each (g[0] = g1), [n][32]
};
__device__ __forceinline__ void store_rows(bf16 *__restrict__ dst, int ld, const uint32_t (*a)[4], int KT, int64_t r0,
                                           int64_t n, int g, int t) {
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
        if (kk < KT)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t r = r0 + g + 8 * (j & 1);
                if (r < n) *reinterpret_cast<uint32_t *>(dst + r * ld + kk * 16 + 2 * t + 8 * (j >> 1)) = a[kk][j];
            }
}
__global__ void __launch_bounds__(32 * kTrainWarps)
    k_mlp_train(int n, const float *__restrict__ dirs, const float *__restrict__ y, const bf16 *__restrict__ th,
                const float *__restrict__ th32, const float *__restrict__ scale, const __grid_constant__ TrainArgs T) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    mlpw::Weights &w = *reinterpret_cast<mlpw::Weights *>(sm_raw);
    mlpw::load(w, th, th32, scale);
    __syncthreads();
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, g = lane >> 2, t = lane & 3;
    const int64_t tiles = (int64_t(n) + 15) / 16;
    for (int64_t tile = int64_t(blockIdx.x) * kTrainWarps + warp; tile < tiles; tile += int64_t(gridDim.x) * kTrainWarps) {
        const int64_t r0 = tile * 16;
        float d[2][3], s[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int64_t b = r0 + g + 8 * r, bb = min(b, int64_t(n) - 1);
            const float x = __ldg(dirs + 3 * bb), yy = __ldg(dirs + 3 * bb + 1), z = __ldg(dirs + 3 * bb + 2);
            s[r] = mlpw::half_space_sign(x, yy, z);
            d[r][0] = s[r] * x, d[r][1] = s[r] * yy, d[r][2] = s[r] * z;
            if (t < 3 && b < n) T.x[3 * b + t] = t == 0 ? d[r][0] : t == 1 ? d[r][1] : d[r][2];
        }
        float4 *zs = reinterpret_cast<float4 *>(T.z) + tile * (3 * 16 * 32) + lane;
        uint32_t a[8][4];
        float z[16][4];
        auto keep = [&](int l) {  // pre-activations to memory, activations to rows and to A fragments
#pragma unroll
            for (int nt = 0; nt < 16; ++nt) zs[(l * 16 + nt) * 32] = make_float4(z[nt][0], z[nt][1], z[nt][2], z[nt][3]);
            mlpw::silu_all(z);
            mlpw::pack_a<8>(a, z);
            store_rows(T.a[l], 128, a, 8, r0, n, g, t);
        };
        mlpw::first(w, d[0], d[1], z, t);
        keep(0);
        mlpw::layer<16, 8, false>(w.W2, a, z, lane);
        mlpw::add_bias<16>(w.b2, z, t);
        keep(1);
        mlpw::layer<16, 8, false>(w.W3, a, z, lane);
        mlpw::add_bias<16>(w.b3, z, t);
        keep(2);
        float o[4][4];
        mlpw::layer<4, 8, false>(w.W4, a, o, lane);
        mlpw::add_bias<4>(w.b4, o, t);
        double loss = 0.0;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 8 * nt + 2 * t + (j & 1);
                const int64_t b = r0 + g + 8 * (j >> 1);
                float gv = 0.f;
                if (c < 27 && b < n) {
                    const float r = o[nt][j] - s[j >> 1] * y[b * 27 + c] / w.scale[c];
                    gv = 2.f * r / (float(n) * 27.f);
                    loss += double(r * r / (float(n) * 27.f));
                }
                o[nt][j] = gv;
            }
        for (int k = 16; k > 0; k >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, k);
        if (lane == 0) T.lossp[tile] = loss;
        mlpw::pack_a<2>(a, o);
        store_rows(T.go, 32, a, 2, r0, n, g, t);
        auto back = [&](int l) {  // z holds dL/da of layer l + 1: times silu' of its pre-activations
#pragma unroll
            for (int nt = 0; nt < 16; ++nt) {
                const float4 v = zs[(l * 16 + nt) * 32];
                z[nt][0] *= mlpw::dsilu(v.x), z[nt][1] *= mlpw::dsilu(v.y);
                z[nt][2] *= mlpw::dsilu(v.z), z[nt][3] *= mlpw::dsilu(v.w);
            }
            mlpw::pack_a<8>(a, z);
            store_rows(T.g[l], 128, a, 8, r0, n, g, t);
        };
        mlpw::layer<16, 2, true>(w.W4, a, z, lane);
        back(2);
        mlpw::layer<16, 8, true>(w.W3, a, z, lane);
        back(1);
        mlpw::layer<16, 8, true>(w.W2, a, z, lane);
        back(0);
#pragma unroll
        for (int nt = 0; nt < 16; ++nt)
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (r0 + g + 8 * r < n)
                    *reinterpret_cast<float2 *>(T.g32 + (r0 + g + 8 * r) * 128 + 8 * nt + 2 * t) =
                        make_float2(z[nt][2 * r], z[nt][2 * r + 1]);
    }
}

// Weight gradients of one run of samples (blockIdx.y), blockIdx.x: 0 .. 3 the halves (output rows
// 0..63, 64..127) of dW3 and dW2, 4 dW4, 5 the first layer.  dW[o][i] = sum_b g[b][o] a[b][i] with
// both operands read from sample rows by transposing ldmatrix; the bias gradients are column sums.
// The runs' sums (at most kGradRuns of the whole parameter vector) are added in their order by
// k_grad_sum: one block per output tile summing all 8,192 samples took 2.2 ms.
constexpr int kGradRuns = 64, kGradRows = 64;  // runs at most; samples in shared memory at a time
__global__ void __launch_bounds__(256)
    k_mlp_wgrad(int n, int run, const __grid_constant__ TrainArgs T, float *__restrict__ part) {
    __shared__ __align__(16) bf16 Gs[kGradRows][72];         // 64 output columns of g
    __shared__ __align__(16) bf16 As[kGradRows][mlpw::LD];   // the layer's inputs
    const int64_t b0 = int64_t(blockIdx.y) * run, b1 = min(int64_t(n), b0 + run);
    float *out = part + int64_t(blockIdx.y) * NPAR;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int job = blockIdx.x;
    if (job == 5) {
        // dW1[o][i] = sum_b g1[b][o] x[b][i] (FP32), db1 from the BF16 g1: a thread per output and half run
        __shared__ float red[128][4];
        const int o = tid & 127, half = tid >> 7;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
        for (int64_t b = b0 + half; b < b1; b += 2) {
            const float gv = T.g32[b * 128 + o];
            v[0] += gv * T.x[3 * b], v[1] += gv * T.x[3 * b + 1], v[2] += gv * T.x[3 * b + 2];
            v[3] += __bfloat162float(T.g[0][b * 128 + o]);
        }
        if (half)
            for (int j = 0; j < 4; ++j) red[o][j] = v[j];
        __syncthreads();
        if (!half) {
            for (int j = 0; j < 3; ++j) out[OFF_W1 + 3 * o + j] = v[j] + red[o][j];
            out[OFF_B1 + o] = v[3] + red[o][3];
        }
        return;
    }
    const bf16 *G = job == 4 ? T.go : T.g[job < 2 ? 2 : 1], *A = T.a[job == 4 ? 2 : job < 2 ? 1 : 0];
    const int cols = job == 4 ? 32 : 64, ldg = job == 4 ? 32 : 128, c0 = job == 4 ? 0 : 64 * (job & 1);
    const int w0 = job == 4 ? OFF_W4 : job < 2 ? OFF_W3 : OFF_W2, bias0 = job == 4 ? OFF_B4 : job < 2 ? OFF_B3 : OFF_B2;
    // warp: 16 output rows x 64 inputs
    const int m0 = 16 * (warp & 3), i0 = 64 * (warp >> 2), mat = lane >> 3, r = lane & 7;
    const bool busy = m0 < cols;
    float acc[8][4];
    for (int nt = 0; nt < 8; ++nt)
        for (int j = 0; j < 4; ++j) acc[nt][j] = 0.f;
    float db = 0.f;
    for (int64_t s0 = b0; s0 < b1; s0 += kGradRows) {
        const int rows = int(min(int64_t(kGradRows), b1 - s0));
        const uint4 none = make_uint4(0u, 0u, 0u, 0u);
        for (int i = tid; i < kGradRows * 16; i += 256) {
            const int b = i / 16, c = 8 * (i % 16);
            *reinterpret_cast<uint4 *>(&As[b][c]) =
                b < rows ? *reinterpret_cast<const uint4 *>(A + (s0 + b) * 128 + c) : none;
        }
        for (int i = tid; i < kGradRows * cols / 8; i += 256) {
            const int b = i / (cols / 8), c = 8 * (i % (cols / 8));
            *reinterpret_cast<uint4 *>(&Gs[b][c]) =
                b < rows ? *reinterpret_cast<const uint4 *>(G + (s0 + b) * ldg + c0 + c) : none;
        }
        __syncthreads();
        if (busy)
#pragma unroll
            for (int kk = 0; kk < kGradRows / 16; ++kk) {
                uint32_t a[4], b[4];
                // A[o][b] from rows of samples: pieces (o low, b low), (o high, b low), (o low, b high), ..
                mlpw::ldsm4<true>(a, &Gs[kk * 16 + (mat >> 1) * 8 + r][m0 + (mat & 1) * 8]);
#pragma unroll
                for (int nt = 0; nt < 8; nt += 2) {
                    mlpw::ldsm4<true>(b, &As[kk * 16 + (mat & 1) * 8 + r][i0 + (nt + (mat >> 1)) * 8]);
                    mlpw::mma16816(acc[nt], a, b[0], b[1]);
                    mlpw::mma16816(acc[nt + 1], a, b[2], b[3]);
                }
            }
        if (tid < cols)
            for (int b = 0; b < rows; ++b) db += __bfloat162float(Gs[b][tid]);
        __syncthreads();
    }
    if (tid < cols) out[bias0 + c0 + tid] = db;
    if (busy)
        for (int nt = 0; nt < 8; ++nt)
            for (int j = 0; j < 4; ++j)
                out[w0 + (c0 + m0 + (lane >> 2) + 8 * (j >> 1)) * 128 + i0 + 8 * nt + 2 * (lane & 3) + (j & 1)] = acc[nt][j];
}

// gradient = the runs' sums in order; the last block adds the tiles' losses
__global__ void __launch_bounds__(256) k_grad_sum(int runs, const float *__restrict__ part, float *__restrict__ grad,
                                                  int64_t tiles, const double *__restrict__ lossp,
                                                  float *__restrict__ loss) {
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ double sm[256];
        double s = 0.0;
        for (int64_t i = threadIdx.x; i < tiles; i += 256) s += lossp[i];
        sm[threadIdx.x] = s;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) *loss = float(sm[0]);
        return;
    }
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= NPAR) return;
    float s = 0.f;
#pragma unroll 8
    for (int r = 0; r < runs; ++r) s += part[int64_t(r) * NPAR + i];
    grad[i] = s;
}

__global__ void k_adam(int n, float *__restrict__ th, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, float lr, float b1, float b2, float c1, float c2, bf16 *__restrict__ thh) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    // the padding rows of W4 and b4 (outputs 27..31) stay zero
    const bool pad = (i >= OFF_W4 + 27 * 128 && i < OFF_B4) || i >= OFF_B4 + 27;
    if (!pad) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    }
    thh[i] = __float2bfloat16(th[i]);
}

__global__ void k_to_bf16(int n, const float *__restrict__ a, bf16 *__restrict__ b) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = __float2bfloat16(a[i]);
}

// plain-evaluator labels (FP64 unit-circle rule), all 27 components
__global__ void k_labels(int64_t n, const DevMaterial *__restrict__ mat, const float *__restrict__ dirs,
                         float *__restrict__ y) {
    const int64_t b = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (b >= n) return;
    double T[3] = {dirs[3 * b], dirs[3 * b + 1], dirs[3 * b + 2]};
    const double r = sqrt(T[0] * T[0] + T[1] * T[1] + T[2] * T[2]);
    for (int i = 0; i < 3; ++i) T[i] /= r;
    double hs[18];
    if (mat->mode == GBFMM_H_ISO)
        h_iso_sym<double>(mat->hc, mat->ha, T, hs);
    else if (mat->cubic)
        h_circle_cubic<double>(mat->c12, mat->c44, mat->cd, mat->Q, T, hs);
    else
        h_circle_sym<double, double>(mat->C, mat->Q, T, hs);
    constexpr int PI_[3][3] = {{0, 5, 4}, {5, 1, 3}, {4, 3, 2}};  // (v,p) -> symmetric pair index
    for (int v = 0; v < 3; ++v)
        for (int p = 0; p < 3; ++p)
            for (int q = 0; q < 3; ++q) y[b * 27 + (v * 3 + p) * 3 + q] = float(hs[3 * PI_[v][p] + q]);
}

__global__ void k_sumsq(int64_t n, const float *__restrict__ y, double *__restrict__ acc) {
    const int64_t b = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (b >= n) return;
    for (int c = 0; c < 27; ++c) atomicAdd(&acc[c], double(y[b * 27 + c]) * double(y[b * 27 + c]));
}

__global__ void k_gather_rows(int n, int w, const int *__restrict__ idx, const float *__restrict__ src,
                              float *__restrict__ dst) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= int64_t(n) * w) return;
    dst[i] = src[int64_t(idx[i / w]) * w + (i % w)];
}

// The network as polynomials for the near field: per angular bin the least-squares quadratic in
// the bin's coordinates (u, v) through the network's values at 8 x 8 directions, on the basis
// 1, u, v, u^2 - m2, uv, v^2 - m2, which is orthogonal on that grid (m2 = mean of u^2); the 18
// components symmetric in (v, p).  One block per bin, a thread per coefficient.  A
// pair of the near field then costs 108 multiply-adds instead of 37,000.  How far the quadratics are
// from h depends on the medium as well as on the network (fitted to h itself they are 3e-4 of its RMS
// off at a Zener ratio of 3.2, in the worst bin 3e-3; ten times that in the worst bin at 8):
// fmm_mlp_calibrate judges them.
constexpr int kBins = 5 * 256, kBinGrid = 8, kBinPer = kBinGrid * kBinGrid;
__host__ __device__ inline float grid_coord(int i) { return float(2 * i + 1 - kBinGrid) / float(kBinGrid); }

constexpr int kBinEdge = 5, kBinEdgePer = kBinEdge * kBinEdge;
__host__ __device__ inline float edge_coord(int i) { return float(2 * i) / float(kBinEdge - 1) - 1.f; }

// directions of every angular bin (the near field's binning: dominant axis face +z, +x, -x, +y, -y and a
// 16 x 16 grid of the other two components), [bin][m^2][3]: the 8 x 8 that the polynomials are fitted
// at (m = kBinGrid), or 5 x 5 from edge to edge (m = kBinEdge), one thread each
__global__ void k_bin_dirs(int m, float *__restrict__ dirs) {
    const int b = blockIdx.x, i = threadIdx.x, f = b / 256;
    const float u = m == kBinGrid ? grid_coord(i % m) : edge_coord(i % m), v = m == kBinGrid ? grid_coord(i / m) : edge_coord(i / m);
    const float p = -1.f + (2.f * float((b / 16) % 16) + 1.f + u) / 16.f;
    const float q = -1.f + (2.f * float(b % 16) + 1.f + v) / 16.f;
    const float n = sqrtf(p * p + q * q + 1.f);
    const float x = f == 0 || f >= 3 ? p : f == 1 ? 1.f : -1.f, y = f == 0 ? q : f <= 2 ? p : f == 3 ? 1.f : -1.f;
    float *d = dirs + (int64_t(b) * m * m + i) * 3;
    d[0] = x / n, d[1] = y / n, d[2] = (f == 0 ? 1.f : q) / n;
}
__global__ void k_bin_poly(const float *__restrict__ h, float m2, float *__restrict__ poly) {
    constexpr int PV[6] = {0, 1, 2, 1, 0, 0}, PP[6] = {0, 1, 2, 2, 2, 1};
    const int t = threadIdx.x;
    if (t >= 108) return;
    const int k = t / 6, c = t % 6, v = PV[k / 3], p = PP[k / 3], q = k % 3;
    const float *hb = h + int64_t(blockIdx.x) * kBinGrid * kBinGrid * 27;
    double num = 0.0, den = 0.0;
    for (int i = 0; i < kBinGrid * kBinGrid; ++i) {
        const double a = grid_coord(i % kBinGrid), b = grid_coord(i / kBinGrid);
        const double phi = c == 0 ? 1.0 : c == 1 ? a : c == 2 ? b : c == 3 ? a * a - m2 : c == 4 ? a * b : b * b - m2;
        num += phi * 0.5 * (double(hb[27 * i + (v * 3 + p) * 3 + q]) + double(hb[27 * i + (p * 3 + v) * 3 + q]));
        den += phi * phi;
    }
    poly[108 * blockIdx.x + t] = float(num / den);
}

}  // namespace

// ---------------------------------------------------------------- host side
struct MlpBuffers {
    int64_t cap = 0;  // samples, a multiple of 16
    TrainArgs t{};
    float *part = nullptr;  // [kGradRuns][NPAR]
};

static MlpBuffers &bufs(gbfmm_ctx *ctx) { return *reinterpret_cast<MlpBuffers *>(ctx->mlp.bufs); }

static int mlp_alloc_state(gbfmm_ctx *ctx) {
    MlpState &M = ctx->mlp;
    if (M.theta) return GBFMM_OK;
    CK(cudaMalloc(&M.theta, NPAR * sizeof(float)));
    CK(cudaMalloc(&M.grad, NPAR * sizeof(float)));
    CK(cudaMalloc(&M.m, NPAR * sizeof(float)));
    CK(cudaMalloc(&M.v, NPAR * sizeof(float)));
    CK(cudaMalloc(&M.theta_h, NPAR * sizeof(bf16)));
    CK(cudaMalloc(&M.scale, 32 * sizeof(float)));
    CK(cudaMalloc(&M.loss, sizeof(float)));
    M.bufs = new MlpBuffers();
    return GBFMM_OK;
}

// buffers of a training batch of n samples
static int mlp_alloc_batch(gbfmm_ctx *ctx, int n) {
    MlpBuffers &B = bufs(ctx);
    TrainArgs &T = B.t;
    if (!B.part) CK(cudaMalloc(&B.part, size_t(kGradRuns) * NPAR * sizeof(float)));
    const size_t m = (size_t(n) + 15) / 16 * 16;
    return grow_dev(ctx, B.cap, int64_t(m),
                    {{(void **)&T.x, m * 3 * sizeof(float)}, {(void **)&T.z, m * 384 * sizeof(float)},
                     {(void **)&T.g32, m * 128 * sizeof(float)}, {(void **)&T.lossp, m / 16 * sizeof(double)},
                     {(void **)&T.a[0], m * 128 * sizeof(bf16)}, {(void **)&T.a[1], m * 128 * sizeof(bf16)},
                     {(void **)&T.a[2], m * 128 * sizeof(bf16)}, {(void **)&T.g[0], m * 128 * sizeof(bf16)},
                     {(void **)&T.g[1], m * 128 * sizeof(bf16)}, {(void **)&T.g[2], m * 128 * sizeof(bf16)},
                     {(void **)&T.go, m * 32 * sizeof(bf16)}},
                    "network batch");
}

// network outputs of n directions (BF16 weight matrices, FP32 biases, FP32 accumulation)
static int mlp_forward(gbfmm_ctx *ctx, int64_t n, const float *dirs, float *h) {
    const MlpState &M = ctx->mlp;
    CK(cudaFuncSetAttribute(k_mlp_eval, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(EvalSmem))));
    ++ctx->launches;
    k_mlp_eval<<<unsigned(std::min<int64_t>((n + 15) / 16, 2 * ctx->sm_count)), 32 * kEvalWarps, sizeof(EvalSmem), ctx->stream>>>(
        n, dirs, M.theta_h, M.theta, M.scale, h);
    CK(cudaGetLastError());
    return GBFMM_OK;
}

// gradient of the loss on one batch into M.grad; loss (scaled units) into M.loss
static int mlp_gradient(gbfmm_ctx *ctx, int n, const float *dirs, const float *y) {
    MlpState &M = ctx->mlp;
    MlpBuffers &B = bufs(ctx);
    const int64_t tiles = (int64_t(n) + 15) / 16, blocks = (tiles + kTrainWarps - 1) / kTrainWarps;
    const size_t smem = sizeof(mlpw::Weights);
    CK(cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
    const int64_t run = std::max<int64_t>(128, ((int64_t(n) + kGradRuns - 1) / kGradRuns + 15) / 16 * 16);
    const int runs = int((n + run - 1) / run);
    ctx->launches += 3;
    k_mlp_train<<<unsigned(std::min<int64_t>(blocks, 2 * ctx->sm_count)), 32 * kTrainWarps, smem, ctx->stream>>>(
        n, dirs, y, M.theta_h, M.theta, M.scale, B.t);
    k_mlp_wgrad<<<dim3(6, unsigned(runs)), 256, 0, ctx->stream>>>(n, int(run), B.t, B.part);
    k_grad_sum<<<nblk(NPAR, 256) + 1, 256, 0, ctx->stream>>>(runs, B.part, M.grad, tiles, B.t.lossp, M.loss);
    CK(cudaGetLastError());
    return GBFMM_OK;
}

// BF16 copy of the master parameters
static void sync_params(gbfmm_ctx *ctx) {
    ++ctx->launches;
    k_to_bf16<<<nblk(NPAR, 256), 256, 0, ctx->stream>>>(NPAR, ctx->mlp.theta, ctx->mlp.theta_h);
}

int mlp_eval_device(gbfmm_ctx *ctx, int64_t n, const float *dirs, float *h) {
    MlpState &M = ctx->mlp;
    if (!M.trained) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "fmm_mlp_eval: network not trained or set");
    return mlp_forward(ctx, n, dirs, h);
}

static int mlp_changed(gbfmm_ctx *ctx);

// parameters and scales (host) into the context
static int mlp_load(gbfmm_ctx *ctx, const float *theta, const float *scale) {
    int rc = mlp_alloc_state(ctx);
    if (rc) return rc;
    std::vector<float> th(theta, theta + NPAR);
    for (int i = OFF_W4 + 27 * 128; i < OFF_B4; ++i) th[i] = 0.f;
    for (int i = OFF_B4 + 27; i < NPAR; ++i) th[i] = 0.f;
    float sc[32] = {0};
    for (int i = 0; i < 27; ++i) sc[i] = scale[i];
    ctx->mlp.trained = false;  // until mlp_changed
    CK(cudaMemcpy(ctx->mlp.theta, th.data(), NPAR * sizeof(float), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->mlp.scale, sc, sizeof(sc), cudaMemcpyHostToDevice));
    CK(cudaMemset(ctx->mlp.m, 0, NPAR * sizeof(float)));
    CK(cudaMemset(ctx->mlp.v, 0, NPAR * sizeof(float)));
    rc = mlp_alloc_batch(ctx, 1024);
    if (rc) return rc;
    sync_params(ctx);
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->mlp.step = 0;
    return GBFMM_OK;
}

extern "C" int fmm_mlp_set(gbfmm_ctx *ctx, const float *theta, const float *scale) {
    if (!ctx || !theta || !scale) return GBFMM_ERR_INVALID_ARG;
    if (int rc = mlp_load(ctx, theta, scale)) return rc;
    return mlp_changed(ctx);
}

extern "C" int fmm_mlp_get(gbfmm_ctx *ctx, float *theta, float *scale) {
    if (!ctx || !theta || !scale) return GBFMM_ERR_INVALID_ARG;
    if (!ctx->mlp.theta) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "fmm_mlp_get: no network");
    CK(cudaStreamSynchronize(ctx->stream));
    CK(cudaMemcpy(theta, ctx->mlp.theta, NPAR * sizeof(float), cudaMemcpyDeviceToHost));
    float sc[32];
    CK(cudaMemcpy(sc, ctx->mlp.scale, sizeof(sc), cudaMemcpyDeviceToHost));
    for (int i = 0; i < 27; ++i) scale[i] = sc[i];
    return GBFMM_OK;
}

extern "C" int fmm_mlp_eval(gbfmm_ctx *ctx, int64_t n, const float *dirs, float *h) {
    if (!ctx || n < 0 || (n > 0 && (!dirs || !h))) return GBFMM_ERR_INVALID_ARG;
    if (n == 0) return GBFMM_OK;
    return mlp_eval_device(ctx, n, dirs, h);
}

extern "C" int fmm_mlp_grad(gbfmm_ctx *ctx, int n, const float *dirs, const float *y, float *grad, float *loss) {
    if (!ctx || n < 1 || !dirs || !y || !grad) return GBFMM_ERR_INVALID_ARG;
    if (!ctx->mlp.trained) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "fmm_mlp_grad: set parameters first");
    int rc = mlp_alloc_batch(ctx, n);
    if (rc) return rc;
    rc = mlp_gradient(ctx, n, dirs, y);
    if (rc) return rc;
    CK(cudaMemcpyAsync(grad, ctx->mlp.grad, NPAR * sizeof(float), cudaMemcpyDeviceToDevice, ctx->stream));
    if (loss) {
        CK(cudaStreamSynchronize(ctx->stream));
        CK(cudaMemcpy(loss, ctx->mlp.loss, sizeof(float), cudaMemcpyDeviceToHost));
    }
    return GBFMM_OK;
}

extern "C" int fmm_mlp_labels(gbfmm_ctx *ctx, int64_t n, const float *dirs, float *y) {
    if (!ctx || n < 0 || (n > 0 && (!dirs || !y))) return GBFMM_ERR_INVALID_ARG;
    if (!ctx->have_material) return set_err(ctx, GBFMM_ERR_NO_MATERIAL, "fmm_mlp_labels: set the material first");
    if (n == 0) return GBFMM_OK;
    ++ctx->launches;
    k_labels<<<nblk(n, 128), 128, 0, ctx->stream>>>(n, ctx->d_mat, dirs, y);
    CK(cudaGetLastError());
    return GBFMM_OK;
}

extern "C" int fmm_mlp_train(gbfmm_ctx *ctx, int64_t n, const float *dirs, int epochs, int batch, double lr,
                             uint64_t seed, float *final_loss) {
    if (!ctx || n < batch || batch < 64 || epochs < 1 || !dirs || !(lr > 0.0))
        return set_err(ctx, GBFMM_ERR_INVALID_ARG, "fmm_mlp_train: bad arguments");
    if (!ctx->have_material) return set_err(ctx, GBFMM_ERR_NO_MATERIAL, "fmm_mlp_train: set the material first");
    cudaStream_t st = ctx->stream;
    int rc = mlp_alloc_state(ctx);
    if (rc) return rc;
    rc = mlp_alloc_batch(ctx, batch);
    if (rc) return rc;
    MlpState &M = ctx->mlp;
    // labels by the plain evaluator and their per-component RMS
    float *y = nullptr, *bd = nullptr, *by = nullptr;
    int *perm = nullptr;
    double *acc = nullptr;
    CK(cudaMalloc(&y, n * 27 * sizeof(float)));
    CK(cudaMalloc(&bd, int64_t(batch) * 3 * sizeof(float)));
    CK(cudaMalloc(&by, int64_t(batch) * 27 * sizeof(float)));
    CK(cudaMalloc(&perm, n * sizeof(int)));
    CK(cudaMalloc(&acc, 27 * sizeof(double)));
    rc = fmm_mlp_labels(ctx, n, dirs, y);
    if (rc) return rc;
    CK(cudaMemsetAsync(acc, 0, 27 * sizeof(double), st));
    ++ctx->launches;
    k_sumsq<<<nblk(n, 256), 256, 0, st>>>(n, y, acc);
    double h_acc[27];
    CK(cudaMemcpyAsync(h_acc, acc, sizeof(h_acc), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    float sc[32] = {0};
    double smax = 0.0;
    for (int c = 0; c < 27; ++c) smax = std::max(smax, std::sqrt(h_acc[c] / double(n)));
    for (int c = 0; c < 27; ++c) sc[c] = float(std::max(std::sqrt(h_acc[c] / double(n)), 1e-3 * smax));
    // He-style initialisation from a seeded generator
    std::mt19937_64 rng(seed);
    std::normal_distribution<float> nd(0.f, 1.f);
    std::vector<float> th(NPAR, 0.f);
    auto fill = [&](int off, int rows, int cols, int fan_in) {
        const float sd = std::sqrt(2.f / float(fan_in));
        for (int r = 0; r < rows; ++r)
            for (int c = 0; c < cols; ++c) th[off + r * cols + c] = sd * nd(rng);
    };
    fill(OFF_W1, 128, 3, 3);
    fill(OFF_W2, 128, 128, 128);
    fill(OFF_W3, 128, 128, 128);
    fill(OFF_W4, 27, 128, 128);
    rc = mlp_load(ctx, th.data(), sc);
    if (rc) return rc;
    // Adam with cosine decay of the learning rate
    const int steps_per_epoch = int(n / batch);
    const int64_t total = int64_t(steps_per_epoch) * epochs;
    std::vector<int> hp(n);
    float last = 0.f;
    for (int e = 0; e < epochs; ++e) {
        for (int64_t i = 0; i < n; ++i) hp[i] = int(i);
        std::shuffle(hp.begin(), hp.end(), rng);
        CK(cudaMemcpyAsync(perm, hp.data(), n * sizeof(int), cudaMemcpyHostToDevice, st));
        CK(cudaStreamSynchronize(st));
        for (int s = 0; s < steps_per_epoch; ++s) {
            ctx->launches += 2;
            k_gather_rows<<<nblk(int64_t(batch) * 3, 256), 256, 0, st>>>(batch, 3, perm + int64_t(s) * batch, dirs, bd);
            k_gather_rows<<<nblk(int64_t(batch) * 27, 256), 256, 0, st>>>(batch, 27, perm + int64_t(s) * batch, y, by);
            rc = mlp_gradient(ctx, batch, bd, by);
            if (rc) return rc;
            ++M.step;
            const double frac = double(M.step) / double(total);
            const float lr_t = float(lr * (0.02 + 0.98 * 0.5 * (1.0 + std::cos(M_PI * std::min(1.0, frac)))));
            const float b1 = 0.9f, b2 = 0.999f;
            const float c1 = 1.f - std::pow(b1, float(M.step)), c2 = 1.f - std::pow(b2, float(M.step));
            ++ctx->launches;
            k_adam<<<nblk(NPAR, 256), 256, 0, st>>>(NPAR, M.theta, M.grad, M.m, M.v, lr_t, b1, b2, c1, c2,
                                                      M.theta_h);
        }
        CK(cudaMemcpyAsync(&last, M.loss, sizeof(float), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    }
    cudaFree(y);
    cudaFree(bd);
    cudaFree(by);
    cudaFree(perm);
    cudaFree(acc);
    if (final_loss) *final_loss = last;
    return mlp_changed(ctx);
}

// mean of grid_coord^2
float mlp_poly_m2() {
    float s = 0.f;
    for (int i = 0; i < kBinGrid; ++i) s += grid_coord(i) * grid_coord(i);
    return s / float(kBinGrid);
}

// Scratch of a call that prepares or judges the near field's polynomials
struct BinScratch {
    float *dirs = nullptr, *h = nullptr, *y = nullptr;
    ~BinScratch() {
        for (float *p : {dirs, h, y})
            if (p) cudaFree(p);
    }
};

// The near field's polynomials of the current network, built when it is set or trained: an
// evaluation finds them ready.  Synchronises.
static int mlp_tabulate(gbfmm_ctx *ctx) {
    MlpState &M = ctx->mlp;
    constexpr int64_t n = int64_t(kBins) * kBinPer;
    BinScratch b;
    if (!M.poly) CK(cudaMalloc(&M.poly, size_t(kBins) * 108 * sizeof(float)));
    CK(cudaMalloc(&b.dirs, n * 3 * sizeof(float)));
    CK(cudaMalloc(&b.h, n * 27 * sizeof(float)));
    ctx->launches += 2;
    k_bin_dirs<<<kBins, kBinPer, 0, ctx->stream>>>(kBinGrid, b.dirs);
    if (int rc = mlp_forward(ctx, n, b.dirs, b.h)) return rc;
    k_bin_poly<<<kBins, 128, 0, ctx->stream>>>(b.h, mlp_poly_m2(), M.poly);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(ctx->stream));
    return GBFMM_OK;
}

// whether the context's near field reads the polynomials
static bool mlp_near(const gbfmm_ctx *ctx) {
    return ctx->opt.h_mode == GBFMM_H_MLP && ctx->opt.precision != GBFMM_FP64;
}

// after the parameters changed: the polynomials, where the near field reads them
static int mlp_changed(gbfmm_ctx *ctx) {
    if (mlp_near(ctx))
        if (int rc = mlp_tabulate(ctx)) return rc;
    ctx->mlp.trained = true;
    return GBFMM_OK;
}

// Assess per angular bin what the near field uses of the network against the plain evaluator: the
// network's values at the bin's 64 fitted directions, and the bin's polynomial at these and at 25
// more from edge to edge.  A bin whose largest component error of either kind exceeds bin_tol x (RMS
// of h over the fitted directions) is flagged and its pairs take the plain evaluator.
extern "C" int fmm_mlp_calibrate(gbfmm_ctx *ctx, double bin_tol, double *fallback_frac) {
    if (!ctx || !(bin_tol > 0.0)) return GBFMM_ERR_INVALID_ARG;
    if (!ctx->mlp.trained) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "fmm_mlp_calibrate: train or set the network first");
    MlpState &M = ctx->mlp;
    constexpr int64_t n = int64_t(kBins) * kBinPer, ne = int64_t(kBins) * kBinEdgePer;
    BinScratch b;
    CK(cudaMalloc(&b.dirs, n * 3 * sizeof(float)));
    CK(cudaMalloc(&b.y, n * 27 * sizeof(float)));
    CK(cudaMalloc(&b.h, n * 27 * sizeof(float)));
    if (!mlp_near(ctx))  // then they were not built with the network
        if (int rc = mlp_tabulate(ctx)) return rc;
    cudaStream_t st = ctx->stream;
    std::vector<float> hy(n * 27), hh(n * 27), he(ne * 27), poly(size_t(kBins) * 108);
    ctx->launches += 2;
    k_bin_dirs<<<kBins, kBinPer, 0, st>>>(kBinGrid, b.dirs);
    if (int rc = fmm_mlp_labels(ctx, n, b.dirs, b.y)) return rc;
    if (int rc = mlp_eval_device(ctx, n, b.dirs, b.h)) return rc;
    CK(cudaMemcpyAsync(hy.data(), b.y, n * 27 * sizeof(float), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(hh.data(), b.h, n * 27 * sizeof(float), cudaMemcpyDeviceToHost, st));
    k_bin_dirs<<<kBins, kBinEdgePer, 0, st>>>(kBinEdge, b.dirs);
    if (int rc = fmm_mlp_labels(ctx, ne, b.dirs, b.y)) return rc;
    CK(cudaMemcpyAsync(he.data(), b.y, ne * 27 * sizeof(float), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(poly.data(), M.poly, poly.size() * sizeof(float), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    double ss = 0.0;
    for (float v : hy) ss += double(v) * v;
    const double rms = std::sqrt(ss / double(hy.size())), m2 = mlp_poly_m2();
    static const int PV[6] = {0, 1, 2, 1, 0, 0}, PP[6] = {0, 1, 2, 2, 2, 1};
    uint32_t mask[48] = {0};
    int flagged = 0;
    for (int bin = 0; bin < kBins; ++bin) {
        double e = 0.0;
        auto take = [&e](double d) {
            if (!(d <= e)) e = std::isnan(d) ? INFINITY : d;
        };
        for (size_t k = size_t(bin) * kBinPer * 27; k < size_t(bin + 1) * kBinPer * 27; ++k)
            take(std::fabs(double(hh[k]) - double(hy[k])));
        for (int i = 0; i < kBinPer + kBinEdgePer; ++i) {
            const bool fit = i < kBinPer;
            const int g = fit ? i : i - kBinPer;
            const double u = fit ? grid_coord(g % kBinGrid) : edge_coord(g % kBinEdge);
            const double v = fit ? grid_coord(g / kBinGrid) : edge_coord(g / kBinEdge);
            const float *y = fit ? &hy[(size_t(bin) * kBinPer + g) * 27] : &he[(size_t(bin) * kBinEdgePer + g) * 27];
            const double phi[6] = {1.0, u, v, u * u - m2, u * v, v * v - m2};
            for (int k = 0; k < 18; ++k) {
                double h = 0.0;
                for (int c = 0; c < 6; ++c) h += double(poly[size_t(bin) * 108 + 6 * k + c]) * phi[c];
                take(std::fabs(h - double(y[(PV[k / 3] * 3 + PP[k / 3]) * 3 + k % 3])));
            }
        }
        if (e > bin_tol * rms) {
            mask[bin >> 5] |= 1u << (bin & 31);
            ++flagged;
        }
    }
    if (!M.d_binmask) CK(cudaMalloc(&M.d_binmask, sizeof(mask)));
    CK(cudaMemcpy(M.d_binmask, mask, sizeof(mask), cudaMemcpyHostToDevice));
    M.fallback_frac = double(flagged) / double(kBins);
    if (fallback_frac) *fallback_frac = M.fallback_frac;
    return GBFMM_OK;
}

void mlp_free(gbfmm_ctx *ctx) {
    MlpState &M = ctx->mlp;
    void *ps[] = {M.theta, M.grad, M.m, M.v, M.theta_h, M.scale, M.loss, M.d_binmask, M.poly};
    for (void *p : ps)
        if (p) cudaFree(p);
    if (M.bufs) {
        MlpBuffers &B = bufs(ctx);
        const TrainArgs &T = B.t;
        void *qs[] = {T.x, T.z, T.g32, T.lossp, T.a[0], T.a[1], T.a[2], T.g[0], T.g[1], T.g[2], T.go, B.part};
        for (void *p : qs)
            if (p) cudaFree(p);
        delete &B;
    }
    M = MlpState{};
}

// ---------------------------------------------------------------- no-allocation evaluation
// fmm_mlp_eval_noalloc: the network evaluation of fmm_mlp_eval for callers
// that must not allocate device memory during the call (see gbfmm.h): the
// evaluation keeps no activations in memory.
#define GB_NOALLOC_MAX (int64_t(1) << 24)          // largest n accepted per call

extern "C" int fmm_mlp_eval_noalloc(gbfmm_ctx *ctx, int64_t n, const float *dirs, float *h) {
    if (!ctx) return GBFMM_ERR_INVALID_ARG;
    if (n < 0 || (n > 0 && (!dirs || !h)))
        return set_err(ctx, GBFMM_ERR_INVALID_ARG, "fmm_mlp_eval_noalloc: bad arguments");
    if (n > GB_NOALLOC_MAX)
        return set_err(ctx, GBFMM_ERR_INVALID_ARG,
                       "fmm_mlp_eval_noalloc: n = " + std::to_string(n) + " exceeds the maximum of " +
                           std::to_string(GB_NOALLOC_MAX) + " directions per call");
    if (!ctx->mlp.trained) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "fmm_mlp_eval_noalloc: network not set");
    if (n == 0) return GBFMM_OK;
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess || cur != ctx->device)
        return set_err(ctx, GBFMM_ERR_CUDA, "fmm_mlp_eval_noalloc: is the context's device current?");
    return mlp_forward(ctx, n, dirs, h);
}
