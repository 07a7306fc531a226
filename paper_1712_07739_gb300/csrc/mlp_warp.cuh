// Warp-level layers of the angular network.
//
// Sixteen directions form the rows of one m16n8k16 tile; the layers run as warp MMAs (BF16 in,
// FP32 accumulate) with the weights in shared memory and the activations in registers: the FP32
// accumulator fragment of one layer, passed through SiLU and packed to BF16 pairs, is exactly the
// A fragment of the next layer for the same lane (row g = lane / 4 and g + 8, columns
// 8 nt + 2 t, + 1 with t = lane % 4).  B fragments come by ldmatrix, four 8 x 8 pieces (two
// column tiles) an instruction, transposed for the products with the weights' transpose; rows of
// 136 elements keep them free of bank conflicts.  Layout of the parameter vector: W1 [128x3], b1,
// W2 [128x128], b2, W3, b3, W4 [32x128] (rows 27..31 zero), b4 [32].
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace mlpw {

constexpr int OFF_W1 = 0, OFF_B1 = 384, OFF_W2 = 512, OFF_B2 = 16896, OFF_W3 = 17024, OFF_B3 = 33408,
              OFF_W4 = 33536, OFF_B4 = 37632, NPAR = 37664;
constexpr int LD = 136;  // padded row (bf16) of the weight matrices

struct Weights {
    __nv_bfloat16 W2[128 * LD];
    __nv_bfloat16 W3[128 * LD];
    __nv_bfloat16 W4[32 * LD];
    float4 W1[128];  // row and bias
    float b2[128], b3[128], b4[32], scale[32];
};

// cooperative copy of the parameters into shared memory (whole block); the parameter vector's
// matrices start on 16-byte boundaries
__device__ inline void load(Weights &w, const __nv_bfloat16 *__restrict__ th, const float *__restrict__ th32,
                            const float *__restrict__ scale) {
    for (int i = threadIdx.x; i < 128 * 16; i += blockDim.x) {
        const int r = i / 16, c = 8 * (i % 16);
        *reinterpret_cast<uint4 *>(&w.W2[r * LD + c]) = *reinterpret_cast<const uint4 *>(th + OFF_W2 + 8 * i);
        *reinterpret_cast<uint4 *>(&w.W3[r * LD + c]) = *reinterpret_cast<const uint4 *>(th + OFF_W3 + 8 * i);
        if (i < 32 * 16)
            *reinterpret_cast<uint4 *>(&w.W4[r * LD + c]) = *reinterpret_cast<const uint4 *>(th + OFF_W4 + 8 * i);
    }
    for (int i = threadIdx.x; i < 128; i += blockDim.x) {
        w.W1[i] = make_float4(__bfloat162float(th[OFF_W1 + 3 * i]), __bfloat162float(th[OFF_W1 + 3 * i + 1]),
                              __bfloat162float(th[OFF_W1 + 3 * i + 2]), th32[OFF_B1 + i]);
        w.b2[i] = th32[OFF_B2 + i];
        w.b3[i] = th32[OFF_B3 + i];
    }
    for (int i = threadIdx.x; i < 32; i += blockDim.x) {
        w.b4[i] = th32[OFF_B4 + i];
        w.scale[i] = scale[i];
    }
}

// SiLU through the hardware tanh: sigmoid(z) = (1 + tanh(z/2)) / 2, silu = z sigmoid(z),
// silu' = s (1 + z (1 - s))
__device__ __forceinline__ float tanh_hw(float x) {
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float silu(float z) { return 0.5f * z * (1.f + tanh_hw(0.5f * z)); }
__device__ __forceinline__ float dsilu(float z) {
    const float s = 0.5f * (1.f + tanh_hw(0.5f * z));
    return s * (1.f + z * (1.f - s));
}

// sign of the half-space fold (h is odd)
__device__ __forceinline__ float half_space_sign(float x, float y, float z) {
    return (z > 0.f || (z == 0.f && (y > 0.f || (y == 0.f && x >= 0.f)))) ? 1.f : -1.f;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <bool T>
__device__ __forceinline__ void ldsm4(uint32_t r[4], const __nv_bfloat16 *p) {
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    if (T)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// acc[nt] = a (KT steps of 16) times the transpose of W (rows = outputs), or W itself (TR: rows =
// inputs), NT column tiles of 8; sums in ascending k from zero
template <int NT, int KT, bool TR>
__device__ __forceinline__ void layer(const __nv_bfloat16 *__restrict__ W, const uint32_t (*a)[4], float (*acc)[4],
                                      int lane) {
    const int mat = lane >> 3, r = lane & 7;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[nt][j] = 0.f;
#pragma unroll
    for (int kk = 0; kk < KT; ++kk)
#pragma unroll
        for (int nt = 0; nt < NT; nt += 2) {
            uint32_t b[4];
            // pieces in order: (nt, k low half), (nt, k high half), (nt + 1, low), (nt + 1, high)
            ldsm4<TR>(b, TR ? W + (kk * 16 + (mat & 1) * 8 + r) * LD + (nt + (mat >> 1)) * 8
                            : W + ((nt + (mat >> 1)) * 8 + r) * LD + kk * 16 + (mat & 1) * 8);
            mma16816(acc[nt], a[kk], b[0], b[1]);
            mma16816(acc[nt + 1], a[kk], b[2], b[3]);
        }
}

// accumulator fragments -> A fragments of the next product
template <int KT>
__device__ __forceinline__ void pack_a(uint32_t (*a)[4], const float (*v)[4]) {
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) {
        a[kk][0] = pack2(v[2 * kk][0], v[2 * kk][1]);
        a[kk][1] = pack2(v[2 * kk][2], v[2 * kk][3]);
        a[kk][2] = pack2(v[2 * kk + 1][0], v[2 * kk + 1][1]);
        a[kk][3] = pack2(v[2 * kk + 1][2], v[2 * kk + 1][3]);
    }
}

// pre-activations of the first layer (3 inputs) for the folded directions dlo (row g), dhi (row g + 8)
__device__ __forceinline__ void first(const Weights &w, const float dlo[3], const float dhi[3], float (*z)[4], int t) {
#pragma unroll
    for (int nt = 0; nt < 16; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float4 v = w.W1[8 * nt + 2 * t + e];
            z[nt][e] = v.x * dlo[0] + v.y * dlo[1] + v.z * dlo[2] + v.w;
            z[nt][2 + e] = v.x * dhi[0] + v.y * dhi[1] + v.z * dhi[2] + v.w;
        }
}

template <int NT>
__device__ __forceinline__ void add_bias(const float *__restrict__ b, float (*z)[4], int t) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const float2 v = *reinterpret_cast<const float2 *>(b + 8 * nt + 2 * t);
        z[nt][0] += v.x;
        z[nt][1] += v.y;
        z[nt][2] += v.x;
        z[nt][3] += v.y;
    }
}

__device__ __forceinline__ void silu_all(float (*z)[4]) {
#pragma unroll
    for (int nt = 0; nt < 16; ++nt)
#pragma unroll
        for (int j = 0; j < 4; ++j) z[nt][j] = silu(z[nt][j]);
}

}  // namespace mlpw
