// M2L on the tcgen05 tensor cores: offset-grouped dense GEMMs (Sec. 4.1,
// Eq. "m2l"; the M2L stage of Algorithm 2) with FP32 accumulation in TMEM.
//
// Formulation.  At level l the cells form a 2^l grid.  Split it into the 8
// parity classes c = (x & 1, y & 1, z & 1); each class is an m^3 sub-grid,
// m = 2^(l-1).  For a target cell B = 2P + c and an offset o in its
// interaction list, the source A = B - o lies in class c' = (c - o) mod 2 at
// sub-grid position P + s, s = floor((c - o) / 2) in [-1, 1]^3.  The 189
// offsets of class c are therefore, each, a constant shift between two
// sub-grids.
//
// Tiles.  The cells of a (level, class) that hold targets are listed in
// Morton order of their sub-grid position; 128 consecutive ones form a tile,
// and a CTA takes TPC = 3 consecutive tiles and one group of nsub operator
// rows.  The M2L of a tile is
//     S[cell, n] = (2^l / H)^2  sum_o  sum_k  W_c'[cell + s_o, k] T_o[n, k]
// with k = (node m, component wr) and n = (node l, stress component ab):
// per tile one GEMM of M = 128 cells, N = nsub and K = (active offsets) x
// 9 p^3, accumulated in tensor memory (TPC accumulators of nsub columns).
// Each pipeline stage holds the three tiles' multipole rows (gathered by
// cp.async, one row per thread and tile, into the swizzled layout the MMA
// reads; sources outside the sub-grid or without segments read as zeros)
// and one block of operator rows (TMA) that all three tiles use: a stage
// moves 66 KB for 7.1 MFLOP, mostly rows of the level's multipole table,
// which stay in L2 far better than the 1.6 GB of operators.  Offsets whose
// sources are all empty are skipped.
//
// Precision: BF16 operands (hi); for the offsets nearest to the target
// (max |o_i| = 2, the largest far-field terms) the residuals W_lo = W - hi(W)
// and T_lo = T - hi(T) add two more passes, hi*hi + lo*hi + hi*lo.  Other
// modes: TF32 operands; FP16 operands with a power-of-two scale per level for
// W and one for the operators (FP16 carries 3 more mantissa bits than BF16).
//
// Few cells.  Levels 2 .. 4 hold 8 classes of at most 8, 64 and 512 cells, so their tiles above are
// mostly padding and every CTA streams its operator rows of 189 offsets for a handful of cells
// (6,011 segments, p = 6: 23 GB of operators for 68 GFLOP of products, 8.7 of 9.5 ms).  k_m2l_few
// takes the cells of these levels together, 384 to a CTA whatever their level and class, all 316
// offsets, and spreads the offsets over CTAs (sections of the offset list) so that one set of
// cells occupies the GPU; each operator byte is then read once per set.  The sections' sums go to
// scratch and are added in their order (k_few_sum).
//
// Warp roles (320 threads): warp 0 loads the operator rows by TMA, warp 1
// owns TMEM and issues the MMAs, warps 2-9 gather the multipole rows (the
// copies count in the stage's barrier as they arrive) and then read the accumulator out (warp w reads TMEM
// lanes 32 (w % 4) .. 32 (w % 4) + 31, every second 16 columns).  The
// bookkeeping of single threads bounds a stage: with the ring's position by
// division and descriptors formed for every MMA the tensor pipe was 44 % busy
// (levels 2-4 of 50,000 segments, p = 5, free targets, 2.8 ms) whatever the
// gathering did; counted rings and descriptors a constant apart make it 56 %
// (1.7 ms).  Gathering by TMA (tile::gather4) instead is slower (6,011
// segments, p = 6, whole pass 1.92 ms against 1.43).  Every mbarrier wait is
// bounded; on time-out a device status word gets
// GBFMM_ERR_TIMEOUT and the block winds down, freeing its tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "internal.cuh"
#include "m2l_tc.cuh"

namespace {

// geometry of the offsets, the same for every context of the process (which of them has a residual
// operator is the context's: M2LParams::lo)
struct OffsetEntry {
    short top;        // operator index 0..315
    signed char cls;  // source parity class
    signed char sx, sy, sz;
};

__constant__ OffsetEntry c_offs[8][189];

struct M2LParams {
    const uint8_t *Whi, *Wlo;         // packed W (hi, residual)
    int wrow[GB_TC_MAXLEV];           // first row of a level
    int row_bytes;                    // K_pad x element size
    CUtensorMap tmT;                  // T hi: (Kp, Np, 316)
    CUtensorMap tmTlo;                // T residual: (Kp, Np, n_lo)
    int kb;         // K blocks of 64
    int kb_res;     // K blocks the residual passes cover (the leading ones)
    int nsub;       // N per MMA (multiple of 16, <= 256)
    int ncta;       // operator rows per CTA (= nsub)
    int nvalid;     // 6 p^3
    int tmem_cols;  // power of two >= ncta
    int split;      // residual passes on the near offsets, at the levels whose bit is set in split_levels
    int split_levels;
    int drop_first; // failure-detection test: arm the first stage but issue no load into it
    int kstep;      // operand elements per 128-byte row: 64 (bf16, fp16) or 32 (tf32)
    uint32_t idesc; // tcgen05 instruction descriptor
    const unsigned *wmax;  // FP16 mode: per-level max |W| bits (the W scale), else null
    float inv_op_scale;    // FP16 mode: 1 / operator scale, else 1
    int nblk;              // operators as A: 128-row blocks of operator rows (a CTA takes two)
    int o_lo, o_hi;        // this launch takes the entries o_lo .. o_hi - 1 of each class's offset list
    int accumulate;        // 0: the epilogue writes the local values, 1: it adds to them
    short lo[316];         // residual operator of an offset, -1 without
};

// FP16 mode: power of two that brings a level's largest |W| into [2^12, 2^13)
// (FP16 is normal from 2^-14 to 65504, so 26 binades below the largest value
// keep full relative precision); 1 for a level without values
__device__ __forceinline__ float wscale_of(unsigned bits) {
    const float mx = __uint_as_float(bits);
    if (!(mx > 0.f)) return 1.f;
    int e;
    frexpf(mx, &e);  // mx = f 2^e, f in [0.5, 1)
    return ldexpf(1.f, 13 - e);
}

// Two forms of the tile GEMM (gbfmm_options.m2l_kernel):
//  cells as A (SWAP = false): three tiles of 128 target cells per CTA are the M = 128
//    operands of three MMAs that share one block of nsub operator rows (B, N = nsub);
//  operators as A (SWAP = true): two 128-row blocks of operator rows are the M = 128
//    operands (TMA) of two MMAs that share the CTA's two tiles of target cells as one
//    N = 256 operand, so a gathered row feeds 256 instead of nsub output columns and a
//    stage gathers 32 instead of 48 KB for about the same tensor work.
constexpr int kTcThreads = 320;  // warps: operators, MMA, eight for the multipole rows and the epilogue
constexpr int kTileA = 128 * 128;  // one tile's multipole rows per stage: 16 KB
template <bool SWAP> constexpr int tpc_of() { return SWAP ? 2 : 3; }  // tiles of 128 cells per CTA

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait: gives up after ~10 s of device time (a healthy wait lasts microseconds)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int *status) {
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (globaltimer() - t0 > 10000000000ull) {
            atomicExch(status, GBFMM_ERR_TIMEOUT);
            return false;
        }
    }
}

// 16-byte global -> shared copy; src_bytes = 0 writes zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
// this thread's copies so far count once in the barrier when they have arrived
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *tm, int c0, int c1, int c2,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// UMMA shared-memory descriptor, K-major, 128-byte swizzle: start address,
// leading offset 16 B (unused inside one swizzle atom), stride offset 1024 B
// between 8-row groups, descriptor version 1, layout SWIZZLE_128B (2).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= uint64_t((addr >> 4) & 0x3FFF);
    d |= uint64_t(1) << 16;
    d |= uint64_t(1024 >> 4) << 32;
    d |= uint64_t(1) << 46;
    d |= uint64_t(2) << 61;
    return d;
}

// instruction descriptor: D f32 (bits 4-5 = 1), A and B format (bits 7-9,
// 10-12: 1 = bf16 for kind::f16, 2 = tf32 for kind::tf32), both K-major,
// N >> 3 at bits 17-22, M >> 4 at bits 24-28
inline uint32_t idesc_of(int M, int N, bool tf32, bool fp16) {
    // operand formats: kind::tf32 -> 2 (TF32); kind::f16 -> 0 (F16) or 1 (BF16); D in F32
    const uint32_t f = tf32 ? 2u : (fp16 ? 0u : 1u);
    return (1u << 4) | (f << 7) | (f << 10) | (uint32_t(N >> 3) << 17) | (uint32_t(M >> 4) << 24);
}

template <bool TF32>
__device__ __forceinline__ void mma_issue(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if (TF32)
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                tmem_d),
            "l"(a), "l"(b), "r"(idesc), "r"(acc));
    else
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                tmem_d),
            "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Target lists.  Every cell of levels 2 .. L-1 has one slot: level l starts
// at cell_base(l) - cell_base(2), then class c (m^3 slots each), then the
// Morton code of the cell's sub-grid position.  The cells holding targets are
// listed in slot order; 128 consecutive ones of a (level, class) make a tile.
__host__ __device__ inline int64_t slot_base(int l) { return cell_base_d(l) - cell_base_d(2); }

__device__ __forceinline__ uint32_t morton_part(uint32_t v) {  // 10 bits -> every third bit
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}
__device__ __forceinline__ uint32_t morton_compact(uint32_t v) {
    v &= 0x09249249u;
    v = (v | (v >> 2)) & 0x030c30c3u;
    v = (v | (v >> 4)) & 0x0300f00fu;
    v = (v | (v >> 8)) & 0x030000ffu;
    v = (v | (v >> 16)) & 0x3ffu;
    return v;
}

// Segments: one per (level, class), index (l - 2) * 8 + c.  seg[s] = {first
// list entry, cells, first tile}; seg[n_seg].z = total tiles.
constexpr int kMaxSeg = 8 * GB_TC_MAXLEV;

// number of K-block iterations of one work item (same count on every warp);
// split: the residual passes apply at this level
__device__ __forceinline__ int passes_of(const M2LParams &P, int o, int split) { return (split && P.lo[o] >= 0) ? 3 : 1; }

// the stage a role works on and its phase: counted, not divided (a division by the run-time number
// of stages costs more than the rest of a stage's bookkeeping)
struct Ring {
    int s = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next(int stages) {
        if (++s == stages) s = 0, ph ^= 1u;
    }
};

// one stage's MMAs with the cells as A: the tiles in tm, four K steps each; begun: tiles whose
// accumulator holds a sum.  Descriptors of a stage differ in the address field only.
template <bool TF32, int TPC>
__device__ __forceinline__ void mma_tiles(uint32_t tmem, int nsub, uint32_t rows, uint32_t ops, uint32_t idesc, uint32_t tm,
                                          uint32_t begun) {
    const uint64_t ad = sw128_desc(rows), bd = sw128_desc(ops);
#pragma unroll
    for (int t = 0; t < TPC; ++t)
        if ((tm >> t) & 1u)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                mma_issue<TF32>(tmem + t * nsub, ad + uint32_t(t * (kTileA >> 4) + 2 * kk), bd + uint32_t(2 * kk), idesc,
                                kk > 0 ? 1u : (begun >> t) & 1u);
}

// which of a CTA's tiles take part in an offset: those with a source (operators as A: all of them,
// the tiles are one operand)
template <bool SWAP, int TPC, int W>
__device__ __forceinline__ uint32_t tiles_at(const uint32_t (&act)[TPC][W], int o) {
    uint32_t m = 0u;
#pragma unroll
    for (int t = 0; t < TPC; ++t) m |= ((act[t][o / 32] >> (o % 32)) & 1u) << t;
    return SWAP ? (1u << TPC) - 1u : m;
}

// A warp's share of a stage's multipole rows: rows 16 g .. 16 g + 15 of every tile, as copies of 8
// lanes per 128-byte row piece (lane l moves piece l % 8 of rows 4 i + l / 8).  take_rows spreads the
// table rows that the lanes found (lane l: for row l % 16 of tile l / 16, then of tile 2; -1 without) to the copying lanes: addresses and sizes (0 writes zeros).
template <int TPC>
__device__ __forceinline__ void take_rows(const int own[2], int lane, const uint8_t *table, int row_bytes,
                                          const uint8_t *(&src)[TPC][4], uint32_t (&size)[TPC][4]) {
#pragma unroll
    for (int t = 0; t < TPC; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int v = __shfl_sync(0xffffffffu, own[t / 2], 16 * (t & 1) + 4 * i + (lane >> 3));
            src[t][i] = table + 16 * (lane & 7) + int64_t(max(v, 0)) * row_bytes;
            size[t][i] = v < 0 ? 0u : 16u;
        }
}
// one stage's copies of the tiles in tm; dst: this lane's place in the stage's first tile for even and
// odd i (16-byte piece c of row r lies at (c ^ (r & 7)) * 16)
template <int TPC>
__device__ __forceinline__ void copy_rows(uint32_t tm, const uint32_t dst[2], int64_t at, const uint8_t *const (&src)[TPC][4],
                                          const uint32_t (&size)[TPC][4]) {
#pragma unroll
    for (int t = 0; t < TPC; ++t)
        if ((tm >> t) & 1u)
#pragma unroll
            for (int i = 0; i < 4; ++i) cp_async16(dst[i & 1] + t * kTileA + i * 512, src[t][i] + at, size[t][i]);
}

template <bool TF32, bool SWAP>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_m2l_tc(const __grid_constant__ M2LParams P, const int4 *__restrict__ seg, int n_seg,
             const int *__restrict__ list, const int *__restrict__ occ, const int *__restrict__ tocc,
             const TreeBox *__restrict__ box, float *__restrict__ S, double *__restrict__ S64,
             int *__restrict__ status, int stages, int groups) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr int TPC = tpc_of<SWAP>();
    constexpr int kStageA = TPC * kTileA;  // the tiles' gathered multipole rows
    // operator rows per stage: nsub rows (cells as A) or two 128-row blocks (operators as A)
    const int stageB = SWAP ? 2 * kTileA : P.ncta * 128;
    const int stage_bytes = kStageA + stageB;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + stages * stage_bytes);
    // bars[0..stages): full, [stages..2 stages): empty, [2 stages]: accumulator ready
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * stages + 1);

    __shared__ int s_level, s_cls, s_rows, s_nrow, s_stop;  // s_rows, s_nrow: first list entry, cells of the CTA
    __shared__ short s_tgt[TPC][128][3];  // sub-grid positions of the tiles' target cells
    __shared__ uint32_t s_active[6];      // offsets with at least one occupied source cell
    __shared__ uint32_t s_tact[TPC][6];   // the same, of one tile
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int tile = blockIdx.x / groups, group = blockIdx.x % groups;
    if (threadIdx.x == 0) {
        s_level = -1;
        s_stop = *reinterpret_cast<volatile int *>(status) != 0;
        if (tile < seg[n_seg].z)
            for (int si = 0; si < n_seg; ++si) {
                const int4 sg = seg[si];
                const int nt = ((sg.y + 127) / 128 + TPC - 1) / TPC;
                if (tile >= sg.z && tile < sg.z + nt) {
                    s_level = si / 8 + 2;
                    s_cls = si % 8;
                    s_rows = sg.x + 128 * TPC * (tile - sg.z);  // first list entry of the CTA's tiles
                    s_nrow = min(128 * TPC, sg.y - 128 * TPC * (tile - sg.z));
                    break;
                }
            }
    }
    if (threadIdx.x < 6) {
        s_active[threadIdx.x] = 0u;
        for (int t = 0; t < TPC; ++t) s_tact[t][threadIdx.x] = 0u;
    }
    __syncthreads();
    if (s_level < 0 || s_stop) return;  // surplus block, or an earlier block timed out
    const int level = s_level, cls = s_cls, nrow = s_nrow;
    const int split = P.split && ((P.split_levels >> level) & 1);
    const int mbc = SWAP ? min(2, P.nblk - 2 * group) : 1;  // operator blocks of this CTA (operators as A)
    const int m = 1 << (level - 1), n = 1 << level;
    const int64_t cbase = cell_base_d(level);
    for (int r = threadIdx.x; r < 128 * TPC; r += blockDim.x) {
        int sx = -1024, sy = -1024, sz = -1024;  // rows past the CTA's cells: far outside the sub-grid
        if (r < nrow) {
            const uint32_t code = uint32_t(list[s_rows + r]);
            sx = int(morton_compact(code)), sy = int(morton_compact(code >> 1)), sz = int(morton_compact(code >> 2));
        }
        s_tgt[r / 128][r % 128][0] = short(sx), s_tgt[r / 128][r % 128][1] = short(sy);
        s_tgt[r / 128][r % 128][2] = short(sz);
    }
    __syncthreads();

    // active offsets: lane r of warp w checks rows 4r .. 4r + 3 of every tile
    for (int oi = P.o_lo + warp; oi < P.o_hi; oi += kTcThreads / 32) {
        const OffsetEntry e = c_offs[cls][oi];
        const int ccx = e.cls & 1, ccy = (e.cls >> 1) & 1, ccz = e.cls >> 2;
        for (int t = 0; t < TPC; ++t) {
            bool hit = false;
            for (int q = 0; q < 4; ++q) {
                const int row = 4 * lane + q;
                const int px = s_tgt[t][row][0] + e.sx, py = s_tgt[t][row][1] + e.sy, pz = s_tgt[t][row][2] + e.sz;
                if (px >= 0 && py >= 0 && pz >= 0 && px < m && py < m && pz < m) {
                    const int64_t g = cbase + (int64_t(2 * pz + ccz) * n + (2 * py + ccy)) * n + (2 * px + ccx);
                    hit |= occ[g] > 0;
                }
            }
            if (__any_sync(0xffffffffu, hit) && lane == 0) {
                atomicOr(&s_active[oi / 32], 1u << (oi % 32));
                atomicOr(&s_tact[t][oi / 32], 1u << (oi % 32));
            }
        }
    }

    if (threadIdx.x == 0) {
        // full: the operator-load thread (expect_tx) + 256 gathering threads; empty: the MMA commit
        for (int s = 0; s < stages; ++s) mbar_init(smem_u32(&bars[s]), 257);
        for (int s = stages; s < 2 * stages + 1; ++s) mbar_init(smem_u32(&bars[s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(P.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[stages]), accb = smem_u32(&bars[2 * stages]);
    const uint32_t smem0 = smem_u32(smem);

    if (warp == 0 && lane == 0) {
        // ---------------- operator rows (B) by TMA
        Ring rg;
        bool ok = true, drop = P.drop_first != 0;
        for (int oi = P.o_lo; oi < P.o_hi && ok; ++oi) {
            if (!((s_active[oi / 32] >> (oi % 32)) & 1u)) continue;
            const OffsetEntry e = c_offs[cls][oi];
            const int np = passes_of(P, e.top, split);
            for (int pass = 0; pass < np && ok; ++pass) {
                const CUtensorMap *tb = (pass == 2) ? &P.tmTlo : &P.tmT;
                const int tidx = (pass == 2) ? P.lo[e.top] : e.top;
                for (int kb = 0; kb < (pass == 0 ? P.kb : P.kb_res); ++kb, rg.next(stages)) {
                    const int s = rg.s;
                    if (!mbar_wait(empty0 + 8 * s, rg.ph ^ 1, status)) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = full0 + 8 * s;
                    mbar_expect_tx(fb, uint32_t(SWAP ? mbc * kTileA : stageB));
                    if (drop) {  // the MMA warp's wait on this stage runs out
                        drop = false;
                        continue;
                    }
                    if (SWAP)
                        for (int mb = 0; mb < mbc; ++mb)
                            tma_load_3d(smem0 + s * stage_bytes + kStageA + mb * kTileA, tb, kb * P.kstep,
                                        group * 256 + mb * 128, tidx, fb);
                    else
                        tma_load_3d(smem0 + s * stage_bytes + kStageA, tb, kb * P.kstep, group * P.ncta, tidx, fb);
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer
        const uint32_t idesc = P.idesc;
        Ring rg;
        uint32_t begun = 0u;  // tiles whose accumulator holds a sum
        bool ok = true;
        for (int oi = P.o_lo; oi < P.o_hi && ok; ++oi) {
            if (!((s_active[oi / 32] >> (oi % 32)) & 1u)) continue;
            const uint32_t tm = tiles_at<SWAP>(s_tact, oi);
            const OffsetEntry e = c_offs[cls][oi];
            const int np = passes_of(P, e.top, split);
            for (int pass = 0; pass < np && ok; ++pass) {
                for (int kb = 0; kb < (pass == 0 ? P.kb : P.kb_res); ++kb, rg.next(stages)) {
                    const int s = rg.s;
                    if (!mbar_wait(full0 + 8 * s, rg.ph, status)) {
                        ok = false;
                        break;
                    }
                    // the gathered rows were written through the generic proxy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t a = smem0 + s * stage_bytes;
                    if (SWAP) {
                        // the two tiles' 256 rows (contiguous, 1024 B per 8 rows) are the N operand
                        const uint64_t bd = sw128_desc(a);
                        for (int mb = 0; mb < mbc; ++mb) {
                            const uint64_t ad = sw128_desc(a + kStageA + mb * kTileA);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                mma_issue<TF32>(tmem + mb * 256, ad + uint32_t(2 * kk), bd + uint32_t(2 * kk), idesc,
                                                (begun || kk > 0) ? 1u : 0u);
                        }
                    } else {
                        mma_tiles<TF32, TPC>(tmem, P.nsub, a, a + kStageA, idesc, tm, begun);
                    }
                    begun |= tm;
                    mma_commit(empty0 + 8 * s);
                }
            }
        }
        // fires when every MMA issued above has completed (no MMA, no wait: see the epilogue)
        if (s_active[0] | s_active[1] | s_active[2] | s_active[3] | s_active[4] | s_active[5]) mma_commit(accb);
    } else if (warp >= 2) {
        const int wrow0 = 16 * (warp - 2);  // this warp's first row of every tile
        const uint32_t place[2] = {uint32_t((wrow0 + (lane >> 3)) * 128 + (((lane & 7) ^ (lane >> 3)) << 4)),
                                   uint32_t((wrow0 + (lane >> 3)) * 128 + (((lane & 7) ^ (4 + (lane >> 3))) << 4))};
        {
            // ---------------- multipole rows (A): gathered by cp.async into the 128-byte
            // swizzled K-major layout; sources outside the sub-grid, or empty, read as zeros.  Each
            // warp finds the sources of its 16 rows of every tile once per offset.  A stage's copies
            // count in its barrier when they arrive, so no thread waits for them and every stage
            // stays in flight; the MMA thread orders them before the tensor core's reads.
            Ring rg;
            bool ok = true;
            for (int oi = P.o_lo; oi < P.o_hi && ok; ++oi) {
                if (!((s_active[oi / 32] >> (oi % 32)) & 1u)) continue;
                const uint32_t tm = tiles_at<SWAP>(s_tact, oi);
                const OffsetEntry e = c_offs[cls][oi];
                int own[2] = {-1, -1};
#pragma unroll
                for (int k = 0; k < (TPC + 1) / 2; ++k) {
                    const int t = 2 * k + lane / 16, r = wrow0 + lane % 16;
                    if (t >= TPC) continue;
                    const int px = s_tgt[t][r][0] + e.sx, py = s_tgt[t][r][1] + e.sy, pz = s_tgt[t][r][2] + e.sz;
                    if (px >= 0 && py >= 0 && pz >= 0 && px < m && py < m && pz < m) {
                        const int ccx = e.cls & 1, ccy = (e.cls >> 1) & 1, ccz = e.cls >> 2;
                        if (occ[cbase + (int64_t(2 * pz + ccz) * n + (2 * py + ccy)) * n + (2 * px + ccx)] > 0)
                            own[k] = P.wrow[level] + ((e.cls * m + pz) * m + py) * m + px;
                    }
                }
                __syncwarp();
                const int np = passes_of(P, e.top, split);
                for (int pass = 0; pass < np && ok; ++pass) {
                    const uint8_t *src[TPC][4];
                    uint32_t size[TPC][4];
                    take_rows<TPC>(own, lane, pass == 1 ? P.Wlo : P.Whi, P.row_bytes, src, size);
                    for (int kb = 0; kb < (pass == 0 ? P.kb : P.kb_res); ++kb, rg.next(stages)) {
                        const int s = rg.s;
                        if (!mbar_wait(empty0 + 8 * s, rg.ph ^ 1, status)) {
                            ok = false;
                            break;
                        }
                        const uint32_t dst[2] = {smem0 + s * stage_bytes + place[0], smem0 + s * stage_bytes + place[1]};
                        copy_rows<TPC>(tm, dst, int64_t(kb) * 128, src, size);
                        cp_async_arrive(full0 + 8 * s);
                    }
                    ok = __all_sync(0xffffffffu, ok);
                }
            }
            cp_async_wait_all();
        }
        __syncwarp();
        // ---------------- epilogue: TMEM -> scaled FP32 local values of the tile's target cells
        bool any_src = false;
        for (int i = 0; i < 6; ++i) any_src |= s_active[i] != 0u;
        const bool ok = any_src ? mbar_wait(accb, 0, status) : true;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int half = (warp - 2) / 4;  // two warps share a quadrant's rows: every second 16 columns
        const int q = warp % 4;
        const int trow = q * 32 + lane;  // TMEM lane = tile row
        float sc = float(double(n) / box->H) * float(double(n) / box->H);
        if (P.wmax) sc *= P.inv_op_scale / wscale_of(P.wmax[level]);
        const int cx = cls & 1, cy = (cls >> 1) & 1, cz = cls >> 2;
        if (SWAP) {
            // TMEM lane = operator row (of block mb), column = target cell (tile col / 128)
            for (int mb = 0; mb < mbc; ++mb) {
                const int nr = group * 256 + mb * 128 + trow;  // this thread's operator row
                const bool rv = nr < P.nvalid;
                for (int c0 = 16 * half; c0 < 256; c0 += 32) {
                    float v[16];
                    if (ok && any_src) tmem_ld16(tmem + (uint32_t(q * 32) << 16) + uint32_t(mb * 256 + c0), v);
                    for (int i = 0; i < 16; ++i) {
                        const int cell = c0 + i, t = cell >> 7, r = cell & 127;
                        if (!ok || !rv || cell >= nrow) continue;
                        const int64_t g = cbase +
                                          (int64_t(2 * s_tgt[t][r][2] + cz) * n + (2 * s_tgt[t][r][1] + cy)) * n +
                                          (2 * s_tgt[t][r][0] + cx);
                        const int64_t e = g * int64_t(P.nvalid) + nr;
                        if (!any_src) {
                            if (!P.accumulate) {
                                if (S64) S64[e] = 0.0;
                                else S[e] = 0.f;
                            }
                        } else if (P.accumulate) {
                            if (S64) S64[e] += double(v[i]) * double(sc);
                            else S[e] += v[i] * sc;
                        } else {
                            if (S64) S64[e] = double(v[i]) * double(sc);
                            else S[e] = v[i] * sc;
                        }
                    }
                }
            }
        }
        for (int t = 0; t < (SWAP ? 0 : TPC); ++t) {
            const bool valid = ok && t * 128 + trow < nrow;
            int64_t g = 0;
            if (valid)
                g = cbase + (int64_t(2 * s_tgt[t][trow][2] + cz) * n + (2 * s_tgt[t][trow][1] + cy)) * n +
                    (2 * s_tgt[t][trow][0] + cx);
            float *dst = S + g * int64_t(P.nvalid);
            double *dst64 = S64 ? S64 + g * int64_t(P.nvalid) : nullptr;  // FP64 local values, when kept
            bool any_t = false;
            for (int i = 0; i < 6; ++i) any_t |= s_tact[t][i] != 0u;
            if (ok && !any_t) {
                // no occupied source among this launch's offsets: zero local values (or nothing to add)
                if (valid && !P.accumulate)
                    for (int col = group * P.ncta + half; col < min(P.nvalid, (group + 1) * P.ncta); col += 2) {
                        if (dst64) dst64[col] = 0.0;
                        else dst[col] = 0.f;
                    }
            } else if (ok) {
                for (int c0 = 16 * half; c0 < P.nsub; c0 += 32) {
                    float v[16];
                    tmem_ld16(tmem + (uint32_t(q * 32) << 16) + uint32_t(t * P.nsub + c0), v);
                    const int col = group * P.ncta + c0;
                    if (valid)
                        for (int i = 0; i < 16; ++i)
                            if (col + i < P.nvalid) {
                                if (P.accumulate) {
                                    if (dst64) dst64[col + i] += double(v[i]) * double(sc);
                                    else dst[col + i] += v[i] * sc;
                                } else {
                                    if (dst64) dst64[col + i] = double(v[i]) * double(sc);
                                    else dst[col + i] = v[i] * sc;
                                }
                            }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(P.tmem_cols));
    }
}

// ---------------------------------------------------------------- few cells
constexpr int kFewTop = 4;     // deepest level taken together: 64 + 512 + 4,096 cells at most
constexpr int kFewRows = 384;  // cells per CTA (three tiles of 128)
constexpr int kFewSections = 64;
constexpr int kFewSetsMax = (64 + 512 + 4096 + kFewRows - 1) / kFewRows;
struct FewCount {
    int cells, sets, sections;
};
struct FewParams {
    M2LParams P;
    int groups;
    const uint32_t *masks;  // [tile][10]: offsets with a source, by k_few_mask
};
__constant__ signed char c_o316[316][3];

// sections of the offset list for a number of cell sets: about four CTAs per SM, no fewer than
// m2l_chunks (each section is one accumulation in tensor memory).  M2L stage with two / three / four /
// six per SM: 6,011 segments 0.95 / 0.93 / 0.96 / 0.99 ms, 50,000 segments 1.44 / 1.37 / 1.33 / 1.33
__host__ __device__ inline int few_sections(int sets, int groups, int chunks, int sms) {
    const int want = (4 * sms + sets * groups - 1) / (sets * groups);
    const int top = chunks > kFewSections ? chunks : kFewSections;
    return want < chunks ? chunks : (want > top ? top : want);
}

// cells of levels 2 .. top that hold targets, in slot order (level, class, Morton code), so that the
// 128 cells of a tile mostly share a class, whose list has 189 of the 316 offsets:
// x | y << 5 | z << 10 | level << 15
__global__ void __launch_bounds__(1024) k_few_list(int top, int groups, int chunks, int sms, const int *__restrict__ tocc,
                                                   int *__restrict__ list, FewCount *__restrict__ cnt) {
    __shared__ int s_warp[32], s_base;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    const int n_all = int(slot_base(top + 1));
    for (int i0 = 0; i0 < n_all; i0 += 1024) {
        const int i = i0 + threadIdx.x;
        int code = 0;
        bool on = false;
        if (i < n_all) {
            int l = 2;
            while (l < top && i >= int(slot_base(l + 1))) ++l;
            const int m3 = 1 << (3 * (l - 1)), k = i - int(slot_base(l)), cls = k / m3, n = 1 << l;
            const uint32_t mc = uint32_t(k % m3);
            const int x = 2 * int(morton_compact(mc)) + (cls & 1), y = 2 * int(morton_compact(mc >> 1)) + ((cls >> 1) & 1),
                      z = 2 * int(morton_compact(mc >> 2)) + (cls >> 2);
            on = tocc[cell_base_d(l) + (int64_t(z) * n + y) * n + x] > 0;
            code = x | (y << 5) | (z << 10) | (l << 15);
        }
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (lane == 0) s_warp[w] = __popc(m);
        __syncthreads();
        int before = s_base;
        for (int k = 0; k < w; ++k) before += s_warp[k];
        if (on) list[before + __popc(m & ((1u << lane) - 1u))] = code;
        __syncthreads();
        if (threadIdx.x == 1023) s_base = before + s_warp[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const int n = s_base, sets = (n + kFewRows - 1) / kFewRows;
        *cnt = FewCount{n, sets, sets ? few_sections(sets, groups, chunks, sms) : 0};
    }
}

// table row of cell (x, y, z) of a level
__device__ __forceinline__ int packed_row(const M2LParams &P, int level, int x, int y, int z) {
    const int m = 1 << (level - 1), cls = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
    return P.wrow[level] + ((cls * m + z / 2) * m + y / 2) * m + x / 2;
}

// the source at cell - o when it lies in the cell's interaction list and holds segments
__device__ __forceinline__ bool few_source(int code, int ox, int oy, int oz, const int *__restrict__ occ, int &level,
                                           int &x, int &y, int &z) {
    const int tx = code & 31, ty = (code >> 5) & 31, tz = (code >> 10) & 31;
    level = code >> 15;
    const int n = 1 << level;
    x = tx - ox, y = ty - oy, z = tz - oz;
    if (x < 0 || y < 0 || z < 0 || x >= n || y >= n || z >= n) return false;
    if (abs((tx >> 1) - (x >> 1)) > 1 || abs((ty >> 1) - (y >> 1)) > 1 || abs((tz >> 1) - (z >> 1)) > 1) return false;
    return occ[cell_base_d(level) + (int64_t(z) * n + y) * n + x] > 0;
}

// offsets at which a tile of 128 listed cells has a source; one block per tile and 32 offsets
__global__ void __launch_bounds__(512) k_few_mask(const FewCount *__restrict__ cnt, const int *__restrict__ list,
                                                  const int *__restrict__ occ, uint32_t *__restrict__ masks) {
    const int cells = cnt->cells, r0 = blockIdx.x * 128, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (r0 >= cells) return;
    __shared__ uint32_t s_m;
    if (threadIdx.x == 0) s_m = 0u;
    __syncthreads();
    for (int b = w; b < 32; b += 16) {
        const int o = 32 * blockIdx.y + b;
        bool hit = false;
        for (int q = 0; q < 4; ++q) {
            const int r = r0 + 32 * q + lane;
            int l, x, y, z;
            if (o < 316 && r < cells) hit |= few_source(list[r], c_o316[o][0], c_o316[o][1], c_o316[o][2], occ, l, x, y, z);
        }
        if (__any_sync(0xffffffffu, hit) && lane == 0) atomicOr(&s_m, 1u << b);
    }
    __syncthreads();
    if (threadIdx.x == 0) masks[10 * blockIdx.x + blockIdx.y] = s_m;
}

// Item (section, operator group, cell set), the sets fastest: CTAs that run together read the same
// operator rows.  Levels up to 4 go here whatever their cells: with few of them the operators' bytes
// bound the time (6,011 segments, p = 6: 8.6 ms per class, 0.8 here; 157 segments, p = 4: 390 and 16
// us; 50,000 segments, L = 5, p = 5, free targets: 6.2 and 1.7 ms), and a level 4 full of cells is 13
// sets, better spread than 16 tiles (a million segments: whole pass 166.1 and 163.6 ms).  Level 5
// would be 86 sets against 96 tiles that already fill the GPU.  Tiles of one class skip the offsets
// of the others' lists (27 % of the gathered rows had a source without that).
template <bool TF32>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_m2l_few(const __grid_constant__ FewParams F, const FewCount *__restrict__ cnt, const int *__restrict__ list,
              const int *__restrict__ occ, float *__restrict__ part, int Np, int *__restrict__ status, int stages) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const M2LParams &P = F.P;
    constexpr int TPC = 3, kStageA = TPC * kTileA;
    const int stageB = P.ncta * 128, stage_bytes = kStageA + stageB;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + stages * stage_bytes);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * stages + 1);
    __shared__ int s_code[kFewRows];
    __shared__ short s_off[316];  // the section's offsets in order, with the tiles that have a source: o | tiles << 9
    __shared__ int s_noff;
    __shared__ int s_stop;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int sets = cnt->sets, sections = cnt->sections, cells = cnt->cells;
    if (threadIdx.x == 0) s_stop = *reinterpret_cast<volatile int *>(status) != 0;
    __syncthreads();
    if (int(blockIdx.x) >= sets * F.groups * sections || s_stop) return;  // surplus block, or an earlier time-out
    const int set = blockIdx.x % sets, group = (blockIdx.x / sets) % F.groups, sec = blockIdx.x / (sets * F.groups);
    const int nrow = min(kFewRows, cells - set * kFewRows), tiles = (nrow + 127) / 128;
    for (int r = threadIdx.x; r < kFewRows; r += kTcThreads) s_code[r] = r < nrow ? list[set * kFewRows + r] : -1;
    __syncthreads();
    if (warp == 0) {
        // the set's offsets (any tile's) are cut into sections of equal length; word w of lane w
        uint32_t own[TPC] = {0u, 0u, 0u}, u = 0u;
        if (lane < 10)
            for (int t = 0; t < TPC; ++t) {
                if (t < tiles) own[t] = F.masks[10 * (TPC * set + t) + lane];
                u |= own[t];
            }
        int rank = __popc(u);
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, rank, d);
            if (lane >= d) rank += v;
        }
        const int total = __shfl_sync(0xffffffffu, rank, 31), lo = total * sec / sections,
                  hi = total * (sec + 1) / sections;
        rank -= __popc(u) + lo;
        for (uint32_t b = u; b; b &= b - 1, ++rank)
            if (rank >= 0 && rank < hi - lo) {
                const int k = __ffs(b) - 1;
                s_off[rank] = short((32 * lane + k) | (((own[0] >> k) & 1u) << 9) | (((own[1] >> k) & 1u) << 10) |
                                    (((own[2] >> k) & 1u) << 11));
            }
        if (lane == 0) s_noff = hi - lo;
    }
    if (threadIdx.x == 0) {
        // full: the operator-load thread (expect_tx) + 256 gathering threads; empty: the MMA commit
        for (int s = 0; s < stages; ++s) mbar_init(smem_u32(&bars[s]), 257);
        for (int s = stages; s < 2 * stages + 1; ++s) mbar_init(smem_u32(&bars[s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(P.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[stages]), accb = smem_u32(&bars[2 * stages]);
    const uint32_t smem0 = smem_u32(smem);
    const int noff = s_noff;

    if (warp == 0 && lane == 0) {
        // ---------------- operator rows (B) by TMA
        Ring rg;
        bool ok = true, drop = P.drop_first != 0;
        for (int oi = 0; oi < noff && ok; ++oi) {
            const int o = s_off[oi] & 511;
            const int np = passes_of(P, o, P.split);
            for (int pass = 0; pass < np && ok; ++pass) {
                const CUtensorMap *tb = pass == 2 ? &P.tmTlo : &P.tmT;
                const int tidx = pass == 2 ? P.lo[o] : o;
                for (int kb = 0; kb < (pass == 0 ? P.kb : P.kb_res); ++kb, rg.next(stages)) {
                    const int s = rg.s;
                    if (!mbar_wait(empty0 + 8 * s, rg.ph ^ 1, status)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(full0 + 8 * s, uint32_t(stageB));
                    if (drop) {  // the MMA warp's wait on this stage runs out
                        drop = false;
                        continue;
                    }
                    tma_load_3d(smem0 + s * stage_bytes + kStageA, tb, kb * P.kstep, group * P.ncta, tidx, full0 + 8 * s);
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer
        Ring rg;
        uint32_t begun = 0u;
        bool ok = true;
        for (int oi = 0; oi < noff && ok; ++oi) {
            const int o = s_off[oi] & 511;
            const uint32_t tm = uint32_t(s_off[oi]) >> 9;
            const int np = passes_of(P, o, P.split);
            for (int pass = 0; pass < np && ok; ++pass)
                for (int kb = 0; kb < (pass == 0 ? P.kb : P.kb_res); ++kb, rg.next(stages)) {
                    const int s = rg.s;
                    if (!mbar_wait(full0 + 8 * s, rg.ph, status)) {
                        ok = false;
                        break;
                    }
                    // the gathered rows were written through the generic proxy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t a = smem0 + s * stage_bytes;
                    mma_tiles<TF32, TPC>(tmem, P.nsub, a, a + kStageA, P.idesc, tm, begun);
                    begun |= tm;
                    mma_commit(empty0 + 8 * s);
                }
        }
        // fires when every MMA issued above has completed
        if (noff > 0) mma_commit(accb);
    } else if (warp >= 2) {
        const bool any = noff > 0;
        const int wrow0 = 16 * (warp - 2);
        const uint32_t place[2] = {uint32_t((wrow0 + (lane >> 3)) * 128 + (((lane & 7) ^ (lane >> 3)) << 4)),
                                   uint32_t((wrow0 + (lane >> 3)) * 128 + (((lane & 7) ^ (4 + (lane >> 3))) << 4))};
        {
            // ---------------- multipole rows (A), as in k_m2l_tc
            Ring rg;
            bool ok = true;
            for (int oi = 0; oi < noff && ok; ++oi) {
                const int o = s_off[oi] & 511;
                const uint32_t tm = uint32_t(s_off[oi]) >> 9;
                const int ox = c_o316[o][0], oy = c_o316[o][1], oz = c_o316[o][2];
                int own[2] = {-1, -1}, res[2] = {-1, -1};  // res: in levels with residual passes
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int t = 2 * k + lane / 16;
                    const int code = t < TPC ? s_code[t * 128 + wrow0 + lane % 16] : -1;
                    int l, x, y, z;
                    if (code >= 0 && few_source(code, ox, oy, oz, occ, l, x, y, z)) {
                        own[k] = packed_row(P, l, x, y, z);
                        if ((P.split_levels >> l) & 1) res[k] = own[k];
                    }
                }
                __syncwarp();
                const int np = passes_of(P, o, P.split);
                for (int pass = 0; pass < np && ok; ++pass) {
                    const uint8_t *src[TPC][4];
                    uint32_t size[TPC][4];
                    take_rows<TPC>(pass == 0 ? own : res, lane, pass == 1 ? P.Wlo : P.Whi, P.row_bytes, src, size);
                    for (int kb = 0; kb < (pass == 0 ? P.kb : P.kb_res); ++kb, rg.next(stages)) {
                        const int s = rg.s;
                        if (!mbar_wait(empty0 + 8 * s, rg.ph ^ 1, status)) {
                            ok = false;
                            break;
                        }
                        const uint32_t dst[2] = {smem0 + s * stage_bytes + place[0], smem0 + s * stage_bytes + place[1]};
                        copy_rows<TPC>(tm, dst, int64_t(kb) * 128, src, size);
                        cp_async_arrive(full0 + 8 * s);
                    }
                    ok = __all_sync(0xffffffffu, ok);
                }
            }
            cp_async_wait_all();
        }
        __syncwarp();
        // ---------------- epilogue: TMEM -> this section's sums
        uint32_t t_act = 0u;  // tiles with a source in this section
        for (int oi = 0; oi < noff; ++oi) t_act |= uint32_t(s_off[oi]) >> 9;
        const bool ok = any ? mbar_wait(accb, 0, status) : true;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int half = (warp - 2) / 4;  // two warps share a quadrant's rows: every second 16 columns
        const int q = warp % 4, trow = q * 32 + lane;
        for (int t = 0; t < tiles; ++t) {
            const int r = t * 128 + trow;
            float *dst = part + (int64_t(sec) * cells + set * kFewRows + r) * Np + group * P.ncta;
            for (int c0 = 16 * half; c0 < P.nsub; c0 += 32) {
                float v[16];
                for (int i = 0; i < 16; ++i) v[i] = 0.f;
                if (ok && ((t_act >> t) & 1u)) tmem_ld16(tmem + (uint32_t(q * 32) << 16) + uint32_t(t * P.nsub + c0), v);
                if (ok && r < nrow)
                    for (int i = 0; i < 4; ++i)
                        reinterpret_cast<float4 *>(dst + c0)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2],
                                                                              v[4 * i + 3]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(P.tmem_cols));
    }
}

// local values of the listed cells: the sections' sums in their order (two-float), scaled
__global__ void k_few_sum(const FewCount *__restrict__ cnt, const int *__restrict__ list, const float *__restrict__ part,
                          int Np, int nvalid, const unsigned *__restrict__ wmax, float inv_op_scale,
                          const TreeBox *__restrict__ box, float *__restrict__ S, double *__restrict__ S64) {
    const int cell = blockIdx.x;
    if (cell >= cnt->cells) return;
    const int code = list[cell], level = code >> 15, n = 1 << level;
    const int64_t g = cell_base_d(level) + (int64_t((code >> 10) & 31) * n + ((code >> 5) & 31)) * n + (code & 31);
    float sc = float(double(n) / box->H) * float(double(n) / box->H);
    if (wmax) sc *= inv_op_scale / wscale_of(wmax[level]);
    const int64_t step = int64_t(cnt->cells) * Np;
    for (int k = threadIdx.x; k < nvalid; k += blockDim.x) {
        const float *p = part + int64_t(cell) * Np + k;
        float hi = 0.f, lo = 0.f;
        for (int s = 0; s < cnt->sections; ++s) {
            const float b = __ldg(p + s * step), t = hi + b, bb = t - hi;
            lo += (hi - (t - bb)) + (b - bb);
            hi = t;
        }
        if (S64) S64[g * nvalid + k] = (double(hi) + double(lo)) * double(sc);
        else S[g * nvalid + k] = (hi + lo) * sc;
    }
}

// ---------------------------------------------------------------- operators
// T_o[n = l*6 + ab][k = m*9 + wr] = Klat[o (p-1) + l - m][ab][wr] (unit cell);
// hi = bf16(T), lo = bf16(T - hi) (residual table only for split offsets).
template <typename E>
__device__ __forceinline__ E to_elem(double v);
template <>
__device__ __forceinline__ __nv_bfloat16 to_elem<__nv_bfloat16>(double v) {
    return __double2bfloat16(v);
}
template <>
__device__ __forceinline__ float to_elem<float>(double v) {
    return float(v);
}
template <>
__device__ __forceinline__ __half to_elem<__half>(double v) {
    return __double2half(v);
}
__device__ __forceinline__ double elem_value(__half x) { return double(__half2float(x)); }
__device__ __forceinline__ double elem_value(__nv_bfloat16 x) { return double(__bfloat162float(x)); }
__device__ __forceinline__ double elem_value(float x) { return double(x); }

template <typename E>
__global__ void k_build_ops(int p, int lat_n, int Np, int Kp, int Kp_lo, const double *__restrict__ Klat,
                            const int *__restrict__ off_xyz, const int *__restrict__ lo_of, int n_off,
                            double scale, E *__restrict__ Thi, E *__restrict__ Tlo) {
    const int64_t total = int64_t(n_off) * Np * Kp;
    const int P3 = p * p * p;
    const int R0 = (lat_n - 1) / 2;
    for (int64_t idx = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; idx < total;
         idx += int64_t(gridDim.x) * blockDim.x) {
        const int k = int(idx % Kp);
        const int nn = int((idx / Kp) % Np);
        const int o = int(idx / (int64_t(Kp) * Np));
        double v = 0.0;
        if (nn < 6 * P3 && k < 9 * P3) {
            const int l = nn / 6, ab = nn % 6, mm = k / 9, wr = k % 9;
            const int ox = off_xyz[3 * o], oy = off_xyz[3 * o + 1], oz = off_xyz[3 * o + 2];
            const int Dx = ox * (p - 1) + (l % p) - (mm % p) + R0;
            const int Dy = oy * (p - 1) + ((l / p) % p) - ((mm / p) % p) + R0;
            const int Dz = oz * (p - 1) + (l / (p * p)) - (mm / (p * p)) + R0;
            v = scale * Klat[((int64_t(Dz) * lat_n + Dy) * lat_n + Dx) * 54 + ab * 9 + wr];
        }
        const E hi = to_elem<E>(v);
        Thi[idx] = hi;
        const int li = lo_of[o];
        if (li >= 0 && Tlo && k < Kp_lo) Tlo[(int64_t(li) * Np + nn) * Kp_lo + k] = to_elem<E>(v - elem_value(hi));
    }
}

// ---------------------------------------------------------------- Legendre-moment operands
// With gbfmm_options.m2l_basis = 1 the GEMM runs on the Legendre moments of
// each source cell instead of its node values: W'_k = sum_m P_k(ybar_m) W_m
// with P_k(t) = P_k1(2 t_1 - 1) P_k2(2 t_2 - 1) P_k3(2 t_3 - 1) (degrees
// k_i < p), which, since the node values come from Lagrange interpolation
// of degree p - 1, equals sum_j P_k(y_j) q_j over the cell's sources, and
// the operators become T' = T V^-1 (V = V1 x V1 x V1, V1[n][a] = P_n(2 t_a - 1)),
// so T' W' = T W exactly.  The moments are bounded by sum |q| and the rows of
// T' decay with the degree (Legendre coefficients of a smooth kernel), so the
// products summed in one GEMM do not cancel the way the oscillating node
// values of equispaced interpolation do, and 16-bit operands and FP32
// accumulation lose far less.  Every transform is separable: three passes
// of a p x p matrix along the node axes.
// Basis matrices, passed by value (they depend on p, which differs between contexts)
struct BasisMats {
    double V[GB_MAXP * GB_MAXP];   // V1[n][a]
    double Ct[GB_MAXP * GB_MAXP];  // (V1^-1)^T[n][a]
    float Vf[GB_MAXP * GB_MAXP];   // V1 in FP32 (moments of the FP32 pass)
    short pos[GB_MAXP * GB_MAXP * GB_MAXP];  // K position of moment (kz p + ky) p + kx: by total degree
};

// out[.., n, ..] = sum_a M[n][a] in[.., a, ..] along one node axis of a [p^3][9] block,
// summed in the precision R of the values
template <typename R, typename MT>
__device__ __forceinline__ void axis_pass(int p, int axis, const MT *M, const R *__restrict__ in, R *__restrict__ out) {
    const int P3 = p * p * p, stride = axis == 0 ? 1 : (axis == 1 ? p : p * p);
    for (int e = threadIdx.x; e < 9 * P3; e += blockDim.x) {
        const int m = e / 9, wr = e - 9 * m;
        const int n = (m / stride) % p, base = m - n * stride;
        R acc = R(0);
        for (int a = 0; a < p; ++a) acc += R(M[n * p + a]) * in[(base + a * stride) * 9 + wr];
        out[e] = acc;
    }
}

// Modal operator rows T'[o][n][k'] (FP64 arithmetic).  mode 0: largest |T'| into
// *absmax (the FP16 scale); mode 1: write hi (and lo for split offsets).
template <typename E>
__global__ void k_build_ops_modal(int p, int lat_n, int Np, int Kp, int Kp_lo, const double *__restrict__ Klat,
                                  const int *__restrict__ off_xyz, const int *__restrict__ lo_of, double scale,
                                  const __grid_constant__ BasisMats B, int mode, unsigned long long *__restrict__ absmax,
                                  E *__restrict__ Thi, E *__restrict__ Tlo) {
    extern __shared__ double sm_modal[];
    const int P3 = p * p * p, R0 = (lat_n - 1) / 2;
    const int o = blockIdx.x / Np, nn = blockIdx.x % Np;
    double *a = sm_modal, *b = sm_modal + 9 * P3;
    const int64_t row = (int64_t(o) * Np + nn) * Kp;
    const int li = lo_of[o];
    if (nn >= 6 * P3) {  // padding rows
        if (mode == 1)
            for (int k = threadIdx.x; k < Kp; k += blockDim.x) {
                Thi[row + k] = to_elem<E>(0.0);
                if (li >= 0 && Tlo && k < Kp_lo) Tlo[(int64_t(li) * Np + nn) * Kp_lo + k] = to_elem<E>(0.0);
            }
        return;
    }
    const int l = nn / 6, ab = nn % 6;
    const int ox = off_xyz[3 * o], oy = off_xyz[3 * o + 1], oz = off_xyz[3 * o + 2];
    for (int e = threadIdx.x; e < 9 * P3; e += blockDim.x) {
        const int mm = e / 9, wr = e % 9;
        const int Dx = ox * (p - 1) + (l % p) - (mm % p) + R0;
        const int Dy = oy * (p - 1) + ((l / p) % p) - ((mm / p) % p) + R0;
        const int Dz = oz * (p - 1) + (l / (p * p)) - (mm / (p * p)) + R0;
        a[e] = Klat[((int64_t(Dz) * lat_n + Dy) * lat_n + Dx) * 54 + ab * 9 + wr];
    }
    __syncthreads();
    axis_pass<double, double>(p, 0, B.Ct, a, b);
    __syncthreads();
    axis_pass<double, double>(p, 1, B.Ct, b, a);
    __syncthreads();
    axis_pass<double, double>(p, 2, B.Ct, a, b);
    __syncthreads();
    if (mode == 0) {
        double mx = 0.0;
        for (int e = threadIdx.x; e < 9 * P3; e += blockDim.x) mx = fmax(mx, fabs(b[e]));
        for (int s = 16; s > 0; s >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, s));
        if ((threadIdx.x & 31) == 0 && mx > 0.0) atomicMax(absmax, (unsigned long long)__double_as_longlong(mx));
        return;
    }
    // column of moment kk, component wr: 9 pos[kk] + wr (moments ordered by total degree)
    for (int k = threadIdx.x; k < Kp; k += blockDim.x) {
        const int e = k < 9 * P3 ? 9 * B.pos[k / 9] + k % 9 : k;
        const double v = k < 9 * P3 ? scale * b[k] : 0.0;
        const E hi = to_elem<E>(v);
        Thi[row + e] = hi;
        if (li >= 0 && Tlo && e < Kp_lo) Tlo[(int64_t(li) * Np + nn) * Kp_lo + e] = to_elem<E>(v - elem_value(hi));
    }
}

// Node values -> Legendre moments, in place, for the occupied cells of levels 2 + blockIdx.y
template <typename TW>
__global__ void k_w_modal(int p, const __grid_constant__ BasisMats B, TW *__restrict__ W, const int *__restrict__ occ) {
    extern __shared__ __align__(16) unsigned char sm_wm[];
    const int P3 = p * p * p, level = 2 + blockIdx.y;
    TW *a = reinterpret_cast<TW *>(sm_wm), *b = a + 9 * P3;
    const int64_t cells = int64_t(1) << (3 * level), base = cell_base_d(level);
    for (int64_t lin = blockIdx.x; lin < cells; lin += gridDim.x) {
        if (occ[base + lin] <= 0) continue;
        TW *w = W + (base + lin) * int64_t(9 * P3);
        __syncthreads();
        for (int e = threadIdx.x; e < 9 * P3; e += blockDim.x) a[e] = w[e];
        __syncthreads();
        if constexpr (sizeof(TW) == 8) {
            axis_pass<TW, double>(p, 0, B.V, a, b);
            __syncthreads();
            axis_pass<TW, double>(p, 1, B.V, b, a);
            __syncthreads();
            axis_pass<TW, double>(p, 2, B.V, a, b);
        } else {
            axis_pass<TW, float>(p, 0, B.Vf, a, b);
            __syncthreads();
            axis_pass<TW, float>(p, 1, B.Vf, b, a);
            __syncthreads();
            axis_pass<TW, float>(p, 2, B.Vf, a, b);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < 9 * P3; e += blockDim.x) w[9 * B.pos[e / 9] + e % 9] = b[e];
    }
}

// W (FP32, [cell][kv]: kv = 9 p^3 node values or moments, or r2 compressed values) ->
// parity-split hi / lo, [class][mz][my][mx][Kp] per level, one block per cell at a time, levels
// 2 + blockIdx.y.  Rows of cells without segments are not written: the gather never reads them
// (their copies are zero fills).
struct PackArgs {
    int64_t ofs[GB_TC_MAXLEV];  // elements
    int split_levels;           // levels with residuals
};
template <typename E, typename TW>
__global__ void k_pack_w(const __grid_constant__ PackArgs A, int kv, int Kp, const TW *__restrict__ W,
                         const int *__restrict__ occ, const unsigned *__restrict__ wmax, E *__restrict__ Whi,
                         E *__restrict__ Wlo) {
    const int level = 2 + blockIdx.y, n = 1 << level, m = n / 2;
    const double s = wmax ? double(wscale_of(wmax[level])) : 1.0;
    E *hi = Whi + A.ofs[level], *lo = (A.split_levels >> level) & 1 ? Wlo + A.ofs[level] : nullptr;
    const int64_t cells = int64_t(n) * n * n;
    for (int64_t lin = blockIdx.x; lin < cells; lin += gridDim.x) {
        const int64_t g = cell_base_d(level) + lin;
        if (occ[g] <= 0) continue;
        const int x = int(lin % n), y = int((lin / n) % n), z = int(lin / (int64_t(n) * n));
        const int cls = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
        const int64_t row = (((int64_t(cls) * m + z / 2) * m + y / 2) * m + x / 2) * Kp;
        for (int k = threadIdx.x; k < Kp; k += blockDim.x) {
            const double v = k < kv ? double(W[g * kv + k]) : 0.0;
            const double vs = s * v;
            const E h = to_elem<E>(vs);
            hi[row + k] = h;
            if (lo) lo[row + k] = to_elem<E>(vs - elem_value(h));
        }
    }
}

// largest |W| over the occupied cells of every level (non-negative floats order like their bit
// patterns), one block per cell at a time, levels 2 + blockIdx.y
template <typename TW>
__global__ void k_wmax(int kv, const TW *__restrict__ W, const int *__restrict__ occ, unsigned *__restrict__ wmax) {
    const int level = 2 + blockIdx.y;
    const int64_t cells = int64_t(1) << (3 * level), base = cell_base_d(level);
    float mx = 0.f;
    for (int64_t lin = blockIdx.x; lin < cells; lin += gridDim.x) {
        if (occ[base + lin] <= 0) continue;
        const TW *w = W + (base + lin) * int64_t(kv);
        for (int k = threadIdx.x; k < kv; k += blockDim.x) mx = fmaxf(mx, fabsf(float(w[k])));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx > 0.f) atomicMax(wmax + level, __float_as_uint(mx));
}

// largest |K| over the kernel lattice, skipping the singular origin
__global__ void k_lattice_absmax(int64_t n_pts, int64_t origin, const double *__restrict__ Klat,
                                 unsigned long long *__restrict__ out) {
    double mx = 0.0;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n_pts * 54;
         i += int64_t(gridDim.x) * blockDim.x)
        if (i / 54 != origin && isfinite(Klat[i])) mx = fmax(mx, fabs(Klat[i]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx > 0.0) atomicMax(out, (unsigned long long)__double_as_longlong(mx));
}

// Target flags of one level: the slot of every cell that holds targets
__global__ void k_mb_flags(int level, const int *__restrict__ tocc, int *__restrict__ flags) {
    const int n = 1 << level, m = n / 2;
    const int64_t cells = int64_t(n) * n * n, m3 = int64_t(m) * m * m;
    for (int64_t lin = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; lin < cells;
         lin += int64_t(gridDim.x) * blockDim.x) {
        const int x = int(lin % n), y = int((lin / n) % n), z = int(lin / (int64_t(n) * n));
        const int cls = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
        const uint32_t code = morton_part(uint32_t(x >> 1)) | (morton_part(uint32_t(y >> 1)) << 1) |
                              (morton_part(uint32_t(z >> 1)) << 2);
        flags[slot_base(level) + cls * m3 + code] = tocc[cell_base_d(level) + lin] > 0 ? 1 : 0;
    }
}

// compact list of the flagged slots (Morton code of the cell within its class)
__global__ void k_mb_list(int n, int L, const int *__restrict__ flags, const int *__restrict__ pos,
                          int *__restrict__ list) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        if (!flags[k]) continue;
        int l = 2;
        while (l + 1 < L && k >= slot_base(l + 1)) ++l;
        const int64_t m3 = int64_t(1) << (3 * (l - 1));
        list[pos[k]] = int((k - slot_base(l)) % m3);
    }
}

// segment table: {first list entry, cells, first CTA}; seg[n_seg].z = CTAs (per operator group)
__global__ void k_seg_table(int L, int tpc, const int *__restrict__ pos, int4 *__restrict__ seg) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int tiles = 0, si = 0;
    for (int l = 2; l < L; ++l) {
        const int64_t m3 = int64_t(1) << (3 * (l - 1));
        for (int c = 0; c < 8; ++c, ++si) {
            const int64_t s0 = slot_base(l) + c * m3;
            const int first = pos[s0], cnt = pos[s0 + m3] - first;
            seg[si] = make_int4(first, cnt, tiles, 0);
            tiles += ((cnt + 127) / 128 + tpc - 1) / tpc;  // CTAs: tpc tiles each
        }
    }
    seg[si] = make_int4(0, 0, tiles, 0);
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled get_encoder() {
    static EncodeTiled fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    }
    return fn;
}

inline unsigned nblk(int64_t n, int b) { return unsigned(std::min<int64_t>((n + b - 1) / b, 1 << 20)); }

}  // namespace

// V1[n][a] = P_n(2 t_a - 1) on the p equispaced nodes t_a = a / (p - 1), and the
// transpose of its inverse (Gauss-Jordan with partial pivoting, FP64)
static bool basis_matrices(int p, double *V, double *Ct) {
    for (int a = 0; a < p; ++a) {
        const double x = 2.0 * a / (p - 1) - 1.0;
        double pm = 1.0, pc = x;
        for (int n = 0; n < p; ++n) {
            const double v = n == 0 ? 1.0 : (n == 1 ? x : 0.0);
            if (n <= 1) {
                V[n * p + a] = v;
                continue;
            }
            const double nx = ((2.0 * n - 1.0) * x * pc - (n - 1.0) * pm) / n;
            pm = pc;
            pc = nx;
            V[n * p + a] = nx;
        }
    }
    double A[GB_MAXP][2 * GB_MAXP];
    for (int i = 0; i < p; ++i)
        for (int j = 0; j < 2 * p; ++j) A[i][j] = j < p ? V[i * p + j] : (j - p == i ? 1.0 : 0.0);
    for (int c = 0; c < p; ++c) {
        int piv = c;
        for (int r = c + 1; r < p; ++r)
            if (std::fabs(A[r][c]) > std::fabs(A[piv][c])) piv = r;
        if (std::fabs(A[piv][c]) < 1e-300) return false;
        for (int j = 0; j < 2 * p; ++j) std::swap(A[c][j], A[piv][j]);
        const double d = A[c][c];
        for (int j = 0; j < 2 * p; ++j) A[c][j] /= d;
        for (int r = 0; r < p; ++r)
            if (r != c) {
                const double f = A[r][c];
                for (int j = 0; j < 2 * p; ++j) A[r][j] -= f * A[c][j];
            }
    }
    for (int n = 0; n < p; ++n)
        for (int a = 0; a < p; ++a) Ct[n * p + a] = A[a][p + n];  // (V1^-1)[a][n]
    return true;
}

static BasisMats basis_of(const TcPlan &T, int p) {
    BasisMats B;
    std::memset(&B, 0, sizeof(B));
    for (int i = 0; i < p * p; ++i) {
        B.V[i] = T.basisV[i];
        B.Ct[i] = T.basisCt[i];
        B.Vf[i] = float(T.basisV[i]);
    }
    // moments ordered by total degree kx + ky + kz (then by index): the leading K
    // blocks hold the low-order moments, which carry most of each product
    int next = 0;
    for (int deg = 0; deg <= 3 * (p - 1); ++deg)
        for (int kk = 0; kk < p * p * p; ++kk)
            if (kk % p + (kk / p) % p + kk / (p * p) == deg) B.pos[kk] = short(next++);
    return B;
}

// Offsets, their parity-class lists and the operator tables.
int m2l_tc_setup(gbfmm_ctx *ctx) {
    const int p = ctx->opt.p, P3 = p * p * p;
    TcPlan &T = ctx->tc;
    T.tf32 = ctx->opt.m2l_split == 3 ? 1 : 0;
    T.fp16 = (ctx->opt.m2l_split >= 4) ? 1 : 0;
    T.esz = T.tf32 ? 4 : 2;
    // compressed M2L: the GEMM's K and N are the kept source and target ranks
    T.svd = ctx->opt.m2l_svd_tol > 0.0 ? 1 : 0;
    if (T.svd)
        if (int rc = svd_bases(ctx)) return rc;
    T.Kp = ((((T.svd ? T.r2 : 9 * P3)) + 63) / 64) * 64;
    const int nv = T.svd ? T.r1 : 6 * P3;
    T.swap = ctx->opt.m2l_kernel == 1 ? 1 : 0;
    T.tpc = T.swap ? 2 : 3;
    if (T.swap) {
        // operators as A: blocks of 128 operator rows, two per CTA; N = 256 cells per MMA;
        // two accumulators of 256 columns
        T.nblk = (nv + 127) / 128;
        T.Np = T.nblk * 128;
        T.groups = (T.nblk + 1) / 2;
        T.nsub = 256;
        T.ncta = 256;
        T.tmem_cols = 512;
    } else {
        // N per MMA (= operator rows per CTA): multiple of 16, one accumulator per
        // tile, 3 x nsub <= 512 TMEM columns
        int best = 0, best_waste = 1 << 30;
        for (int ns = 16; ns * 3 <= 512 && ns <= 256; ns += 16) {
            const int g = (nv + ns - 1) / ns;
            const int waste = g * ns - nv + g * 32;  // padding plus a per-group cost (the tiles' rows are re-read)
            if (waste < best_waste) {
                best_waste = waste;
                best = ns;
            }
        }
        T.nsub = best;
        T.ncta = best;
        T.groups = (nv + T.ncta - 1) / T.ncta;
        T.Np = T.groups * T.ncta;
        T.nblk = 0;
        T.tmem_cols = 32;
        while (T.tmem_cols < 3 * T.nsub) T.tmem_cols *= 2;
    }
    // the 316 offsets, and which of them get the residual passes
    std::vector<int> off;
    std::vector<int> lo_of;
    int n_lo = 0;
    for (int oz = -3; oz <= 3; ++oz)
        for (int oy = -3; oy <= 3; ++oy)
            for (int ox = -3; ox <= 3; ++ox) {
                const int mx = std::max(std::abs(ox), std::max(std::abs(oy), std::abs(oz)));
                if (mx < 2) continue;
                off.push_back(ox);
                off.push_back(oy);
                off.push_back(oz);
                const int sm = ctx->opt.m2l_split;
                const bool split = !T.tf32 && (sm == 2 || sm == 6 || ((sm == 0 || sm == 5) && mx == 2));
                lo_of.push_back(split ? n_lo++ : -1);
            }
    T.n_off = int(off.size() / 3);
    T.n_lo = n_lo;
    for (int i = 0; i < T.n_off && i < 320; ++i) T.lo_host[i] = short(lo_of[i]);
    OffsetEntry ent[8][189];
    for (int c = 0; c < 8; ++c) {
        const int cc[3] = {c & 1, (c >> 1) & 1, c >> 2};
        int cnt = 0;
        for (int i = 0; i < T.n_off; ++i) {
            const int o[3] = {off[3 * i], off[3 * i + 1], off[3 * i + 2]};
            bool in = true;
            for (int d = 0; d < 3; ++d)
                if (o[d] < -3 + cc[d] || o[d] > 2 + cc[d]) in = false;
            if (!in) continue;
            OffsetEntry &e = ent[c][cnt++];
            e.top = short(i);
            int sc = 0;
            signed char sh[3];
            for (int d = 0; d < 3; ++d) {
                const int t = cc[d] - o[d];  // in [-2, 3]
                const int fl = (t >= 0) ? t / 2 : -((-t + 1) / 2);
                sh[d] = (signed char)fl;
                sc |= (t - 2 * fl) << d;
            }
            e.cls = (signed char)sc;
            e.sx = sh[0];
            e.sy = sh[1];
            e.sz = sh[2];
        }
        if (cnt != 189) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "m2l setup: class offset count != 189");
    }
    CK(cudaMemcpyToSymbol(c_offs, ent, sizeof(ent)));
    signed char o316[316][3];
    for (int i = 0; i < 316; ++i)
        for (int d = 0; d < 3; ++d) o316[i][d] = (signed char)off[3 * i + d];
    CK(cudaMemcpyToSymbol(c_o316, o316, sizeof(o316)));
    int *d_off = nullptr, *d_lo = nullptr;
    CK(cudaMalloc(&d_off, off.size() * sizeof(int)));
    CK(cudaMalloc(&d_lo, lo_of.size() * sizeof(int)));
    CK(cudaMemcpy(d_off, off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(d_lo, lo_of.data(), lo_of.size() * sizeof(int), cudaMemcpyHostToDevice));
    // the residual passes read the leading m2l_split_kblocks blocks of K only
    const int kstep = 128 / T.esz;
    T.Kp_lo = ctx->opt.m2l_split_kblocks > 0 ? std::min(T.Kp, ctx->opt.m2l_split_kblocks * kstep) : T.Kp;
    const size_t hi_elems = size_t(T.n_off) * T.Np * T.Kp, lo_elems = size_t(T.n_lo) * T.Np * T.Kp_lo;
    if (T.Thi) cudaFree(T.Thi);
    if (T.Tlo) cudaFree(T.Tlo);
    T.Thi = T.Tlo = nullptr;
    CK(cudaMalloc(&T.Thi, hi_elems * T.esz));
    CK(cudaMalloc(&T.Tlo, std::max<size_t>(lo_elems, 1) * T.esz));
    T.split = n_lo > 0 ? 1 : 0;
    T.op_scale = 1.0;
    T.modal = (ctx->opt.m2l_basis == 1 && !T.svd) ? 1 : 0;
    if (T.modal && !basis_matrices(p, T.basisV, T.basisCt))
        return set_err(ctx, GBFMM_ERR_INVALID_ARG, "m2l setup: singular Legendre basis matrix");
    const size_t sm_modal = size_t(2) * 9 * P3 * sizeof(double);
    if (T.modal) {
        CK(cudaFuncSetAttribute(k_build_ops_modal<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm_modal)));
        CK(cudaFuncSetAttribute(k_build_ops_modal<__half>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm_modal)));
        CK(cudaFuncSetAttribute(k_build_ops_modal<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(sm_modal)));
        CK(cudaFuncSetAttribute(k_w_modal<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm_modal)));
        CK(cudaFuncSetAttribute(k_w_modal<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm_modal / 2)));
    }
    const BasisMats B = basis_of(T, p);
    if (T.svd) {
        // U^T T_o R for every offset (FP64), with the FP16 scale from their largest entry
        if (int rc = svd_operators(ctx, d_off, d_lo, T.n_off)) {
            cudaFree(d_off);
            cudaFree(d_lo);
            return rc;
        }
        if (T.fp16 && !T.d_wmax) CK(cudaMalloc(&T.d_wmax, GB_TC_MAXLEV * sizeof(unsigned)));
    } else if (T.fp16 && T.modal) {
        // one power of two for all operators from the largest modal entry
        unsigned long long *d_mx = nullptr, mx_bits = 0;
        CK(cudaMalloc(&d_mx, sizeof(unsigned long long)));
        CK(cudaMemsetAsync(d_mx, 0, sizeof(unsigned long long), ctx->stream));
        ++ctx->launches;
        k_build_ops_modal<__half><<<unsigned(T.n_off * T.Np), 256, sm_modal, ctx->stream>>>(
            p, ctx->lat_n, T.Np, T.Kp, T.Kp_lo, ctx->d_Klat, d_off, d_lo, 1.0, B, 0, d_mx, (__half *)nullptr, (__half *)nullptr);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(&mx_bits, d_mx, sizeof(mx_bits), cudaMemcpyDeviceToHost, ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
        cudaFree(d_mx);
        double mx = 0.0;
        std::memcpy(&mx, &mx_bits, sizeof(mx));
        if (mx > 0.0) {
            int e = 0;
            std::frexp(mx, &e);
            T.op_scale = std::ldexp(1.0, 14 - e);
        }
        if (!T.d_wmax) CK(cudaMalloc(&T.d_wmax, GB_TC_MAXLEV * sizeof(unsigned)));
    } else if (T.fp16) {
        // one power of two for all operators: the largest lattice value maps below 2^14
        unsigned long long *d_mx = nullptr, mx_bits = 0;
        CK(cudaMalloc(&d_mx, sizeof(unsigned long long)));
        CK(cudaMemsetAsync(d_mx, 0, sizeof(unsigned long long), ctx->stream));
        const int64_t n_pts = int64_t(ctx->lat_n) * ctx->lat_n * ctx->lat_n;
        const int64_t origin = n_pts / 2;  // lattice centre, D = 0
        ++ctx->launches;
        k_lattice_absmax<<<1024, 256, 0, ctx->stream>>>(n_pts, origin, ctx->d_Klat, d_mx);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(&mx_bits, d_mx, sizeof(mx_bits), cudaMemcpyDeviceToHost, ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
        cudaFree(d_mx);
        double mx = 0.0;
        std::memcpy(&mx, &mx_bits, sizeof(mx));
        if (mx > 0.0) {
            int e = 0;
            std::frexp(mx, &e);
            T.op_scale = std::ldexp(1.0, 14 - e);
        }
        if (!T.d_wmax) CK(cudaMalloc(&T.d_wmax, GB_TC_MAXLEV * sizeof(unsigned)));
    }
    if (!T.svd) ++ctx->launches;
    if (T.svd) {
        // written by svd_operators
    } else if (T.modal) {
        const unsigned g = unsigned(T.n_off * T.Np);
        if (T.tf32)
            k_build_ops_modal<float><<<g, 256, sm_modal, ctx->stream>>>(p, ctx->lat_n, T.Np, T.Kp, T.Kp_lo, ctx->d_Klat, d_off,
                                                                        d_lo, 1.0, B, 1, nullptr, (float *)T.Thi,
                                                                        (float *)nullptr);
        else if (T.fp16)
            k_build_ops_modal<__half><<<g, 256, sm_modal, ctx->stream>>>(p, ctx->lat_n, T.Np, T.Kp, T.Kp_lo, ctx->d_Klat, d_off,
                                                                         d_lo, T.op_scale, B, 1, nullptr,
                                                                         (__half *)T.Thi, (__half *)T.Tlo);
        else
            k_build_ops_modal<__nv_bfloat16><<<g, 256, sm_modal, ctx->stream>>>(
                p, ctx->lat_n, T.Np, T.Kp, T.Kp_lo, ctx->d_Klat, d_off, d_lo, 1.0, B, 1, nullptr, (__nv_bfloat16 *)T.Thi,
                (__nv_bfloat16 *)T.Tlo);
    } else if (T.tf32)
        k_build_ops<float><<<nblk(int64_t(hi_elems), 256), 256, 0, ctx->stream>>>(
            p, ctx->lat_n, T.Np, T.Kp, T.Kp_lo, ctx->d_Klat, d_off, d_lo, T.n_off, 1.0, (float *)T.Thi, (float *)nullptr);
    else if (T.fp16)
        k_build_ops<__half><<<nblk(int64_t(hi_elems), 256), 256, 0, ctx->stream>>>(
            p, ctx->lat_n, T.Np, T.Kp, T.Kp_lo, ctx->d_Klat, d_off, d_lo, T.n_off, T.op_scale, (__half *)T.Thi,
            (__half *)T.Tlo);
    else
        k_build_ops<__nv_bfloat16><<<nblk(int64_t(hi_elems), 256), 256, 0, ctx->stream>>>(
            p, ctx->lat_n, T.Np, T.Kp, T.Kp_lo, ctx->d_Klat, d_off, d_lo, T.n_off, 1.0, (__nv_bfloat16 *)T.Thi,
            (__nv_bfloat16 *)T.Tlo);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(ctx->stream));
    cudaFree(d_off);
    cudaFree(d_lo);
    if (!T.d_status) CK(cudaMalloc(&T.d_status, sizeof(int)));
    CK(cudaMemset(T.d_status, 0, sizeof(int)));
    T.ready_ops = true;
    return GBFMM_OK;
}

static int encode(gbfmm_ctx *ctx, CUtensorMap *tm, void *base, int rank, const cuuint64_t *dims,
                  const cuuint64_t *strides, const cuuint32_t *boxd, const TcPlan &T) {
    EncodeTiled enc = get_encoder();
    if (!enc) return set_err(ctx, GBFMM_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    const CUtensorMapDataType dt = T.tf32   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : T.fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                            : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    CUresult r = enc(tm, dt, cuuint32_t(rank),
                     base, dims, strides, boxd, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_err(ctx, GBFMM_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string(r));
    return GBFMM_OK;
}

// deepest level whose cells k_m2l_few takes (1: none): with the cells as A, and runs of offsets
// that its scratch is sized for
static int few_top_of(const gbfmm_ctx *ctx) {
    if (ctx->tc.swap || ctx->opt.m2l_chunks > kFewSections) return 1;
    return std::min(ctx->L - 1, kFewTop);
}

// The sections' sums and the launch of k_m2l_few for n target points: every number of cells up to
// what the levels hold and n points can occupy (p = 6, levels to 4: 169 MB; 600 points: 27 MB).
static int few_alloc(gbfmm_ctx *ctx, int64_t n) {
    TcPlan &T = ctx->tc;
    const int chunks = std::max(1, ctx->opt.m2l_chunks);
    int64_t cells = 0, rows = 0;
    for (int l = 2; l <= T.few_top; ++l) cells += std::min(int64_t(1) << (3 * l), n);
    T.few_work = 0;
    for (int64_t k = 1; k <= (cells + kFewRows - 1) / kFewRows; ++k) {
        const int64_t sec = few_sections(int(k), T.groups, chunks, ctx->sm_count);
        rows = std::max(rows, sec * std::min(k * kFewRows, cells));
        T.few_work = std::max<int>(T.few_work, int(k * sec * T.groups));
    }
    PassScratch &ws = ctx->ws();
    return grow_dev(ctx, ws.few_cap, rows * T.Np, {{(void **)&ws.few_part, size_t(rows) * T.Np * sizeof(float)}},
                    "M2L sections");
}

// Per-tree buffers: packed W (hi / lo), tensor maps, work list.
int m2l_tc_prepare(gbfmm_ctx *ctx) {
    TcPlan &T = ctx->tc;
    const int L = ctx->L;
    if (L - 1 >= GB_TC_MAXLEV) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "tensor-core M2L: too many levels");
    int64_t tot = 0;
    for (int l = 2; l < L; ++l) {
        T.wofs[l] = tot;
        tot += (int64_t(1) << (3 * l)) * T.Kp;
    }
    if (int rc = grow_dev(ctx, T.w_cap, tot, {{&T.Whi, size_t(tot) * T.esz}, {&T.Wlo, size_t(tot) * T.esz}},
                          "packed multipole values"))
        return rc;
    // levels 2 .. few_top go through k_m2l_few: its cell list, counts and the sections' sums
    T.few_top = few_top_of(ctx);
    if (T.few_top >= 2) {
        if (int rc = few_alloc(ctx, ctx->N)) return rc;
        if (!T.few_list)
            CK(cudaMalloc(&T.few_list, 16 + (cell_base(kFewTop + 1) - cell_base(2)) * sizeof(int) +
                                           (kFewSetsMax * 3 * 10) * sizeof(uint32_t)));
    }
    // cell slots, target list and segment table (filled on the device per pass)
    const int64_t slots = slot_base(L);
    int64_t tiles = 0;  // CTAs per operator group, upper bound: every cell holds targets
    for (int l = std::max(2, T.few_top + 1); l < L; ++l) tiles += 8 * ((((int64_t(1) << (3 * (l - 1))) + 127) / 128 + T.tpc - 1) / T.tpc);
    if (int rc = grow_dev(ctx, T.slot_cap, slots,
                          {{(void **)&T.d_flags, slots * sizeof(int)}, {(void **)&T.d_pos, (slots + 1) * sizeof(int)},
                           {(void **)&T.d_list, slots * sizeof(int)}},
                          "M2L target lists"))
        return rc;
    if (!T.d_seg) CK(cudaMalloc(&T.d_seg, (kMaxSeg + 1) * sizeof(int4)));
    T.n_slots = slots;
    T.n_seg = 8 * (L - 2);
    T.n_work = int(tiles * T.groups);
    if (T.svd) return svd_prepare(ctx);
    return GBFMM_OK;
}

int m2l_tc_run(gbfmm_ctx *ctx, const float *Wf, const double *W64, const int *occ, const int *tocc, float *Sf,
               double *S64, bool fine, int64_t n_targets) {
    TcPlan &T = ctx->tc;
    // fine: the adaptive tree's children (level ctx->L) take part through fine_m2l, after the
    // tensor-core M2L of levels 2 .. L-1
    const int L = ctx->L, p = ctx->opt.p, P3 = p * p * p;
    M2LParams prm;  // copied by value into the launch (kernel parameter space)
    std::memset(&prm, 0, sizeof(prm));
    if (T.fp16) CK(cudaMemsetAsync(T.d_wmax, 0, GB_TC_MAXLEV * sizeof(unsigned), ctx->stream));
    const BasisMats B = basis_of(T, p);
    const int split_levels = ctx->opt.m2l_split_levels ? ctx->opt.m2l_split_levels : ~0;
    // compressed M2L: every cell's multipole values -> r2 coefficients R^T W first
    if (T.svd)
        if (int rc = svd_transform_w(ctx, Wf, fine)) return rc;
    const float *Wsrc = T.svd ? T.Wc : Wf;
    const int kv = T.svd ? T.r2 : 9 * P3;  // valid values per cell row
    PackArgs pk{};
    pk.split_levels = T.split ? split_levels : 0;
    for (int l = 2; l < L; ++l) {
        pk.ofs[l] = T.wofs[l];
        prm.wrow[l] = int(T.wofs[l] / T.Kp);
    }
    // blocks stride over the cells of a level, one row of blocks per level
    const dim3 gw(unsigned(std::min<int64_t>(int64_t(1) << (3 * (L - 1)), 8 * ctx->sm_count)), unsigned(L - 2));
    cudaStream_t st = ctx->stream;
    if (T.modal && !T.svd) {
        // node values -> Legendre moments (in place: nothing reads these W after the M2L)
        ++ctx->launches;
        if (W64)
            k_w_modal<double><<<gw, 256, size_t(2) * 9 * P3 * sizeof(double), st>>>(p, B, const_cast<double *>(W64), occ);
        else
            k_w_modal<float><<<gw, 256, size_t(2) * 9 * P3 * sizeof(float), st>>>(p, B, const_cast<float *>(Wf), occ);
    }
    if (T.tf32) {
        ++ctx->launches;
        if (W64)
            k_pack_w<float><<<gw, 256, 0, st>>>(pk, kv, T.Kp, W64, occ, nullptr, (float *)T.Whi, (float *)nullptr);
        else
            k_pack_w<float><<<gw, 256, 0, st>>>(pk, kv, T.Kp, Wsrc, occ, nullptr, (float *)T.Whi, (float *)nullptr);
    } else if (T.fp16) {
        ctx->launches += 2;
        if (W64) {
            k_wmax<<<gw, 256, 0, st>>>(kv, W64, occ, T.d_wmax);
            k_pack_w<__half><<<gw, 256, 0, st>>>(pk, kv, T.Kp, W64, occ, T.d_wmax, (__half *)T.Whi, (__half *)T.Wlo);
        } else {
            k_wmax<<<gw, 256, 0, st>>>(kv, Wsrc, occ, T.d_wmax);
            k_pack_w<__half><<<gw, 256, 0, st>>>(pk, kv, T.Kp, Wsrc, occ, T.d_wmax, (__half *)T.Whi, (__half *)T.Wlo);
        }
    } else {
        ++ctx->launches;
        if (W64)
            k_pack_w<__nv_bfloat16><<<gw, 256, 0, st>>>(pk, kv, T.Kp, W64, occ, nullptr, (__nv_bfloat16 *)T.Whi,
                                                        (__nv_bfloat16 *)T.Wlo);
        else
            k_pack_w<__nv_bfloat16><<<gw, 256, 0, st>>>(pk, kv, T.Kp, Wsrc, occ, nullptr, (__nv_bfloat16 *)T.Whi,
                                                        (__nv_bfloat16 *)T.Wlo);
    }
    CK(cudaGetLastError());
    prm.Whi = static_cast<const uint8_t *>(T.Whi);
    prm.Wlo = static_cast<const uint8_t *>(T.Wlo);
    prm.row_bytes = T.Kp * T.esz;
    {
        const cuuint64_t dims[3] = {cuuint64_t(T.Kp), cuuint64_t(T.Np), cuuint64_t(T.n_off)};
        const cuuint64_t strides[2] = {cuuint64_t(T.Kp) * T.esz, cuuint64_t(T.Kp) * T.esz * T.Np};
        // box: one K block of operator rows: nsub rows (cells as A) or a 128-row block (operators as A)
        const cuuint32_t boxd[3] = {cuuint32_t(128 / T.esz), cuuint32_t(T.swap ? 128 : T.nsub), 1};
        int rc = encode(ctx, &prm.tmT, T.Thi, 3, dims, strides, boxd, T);
        if (rc) return rc;
        const cuuint64_t dl[3] = {cuuint64_t(T.Kp_lo), cuuint64_t(T.Np), cuuint64_t(std::max(T.n_lo, 1))};
        const cuuint64_t sl[2] = {cuuint64_t(T.Kp_lo) * T.esz, cuuint64_t(T.Kp_lo) * T.esz * T.Np};
        rc = encode(ctx, &prm.tmTlo, T.Tlo, 3, dl, sl, boxd, T);
        if (rc) return rc;
    }
    prm.kstep = 128 / T.esz;
    prm.kb = T.Kp / prm.kstep;
    prm.kb_res = ctx->opt.m2l_split_kblocks > 0 ? std::min(prm.kb, ctx->opt.m2l_split_kblocks) : prm.kb;
    prm.idesc = idesc_of(128, T.nsub, T.tf32, T.fp16);  // M = 128; N = nsub, or 256 cells (operators as A)
    prm.nblk = T.nblk;
    prm.wmax = T.fp16 ? T.d_wmax : nullptr;
    prm.inv_op_scale = float(1.0 / T.op_scale);
    prm.nsub = T.nsub;
    prm.ncta = T.ncta;
    prm.nvalid = T.svd ? T.r1 : 6 * P3;
    prm.tmem_cols = T.tmem_cols;
    prm.split = T.split;
    prm.split_levels = split_levels;
    for (int i = 0; i < 316; ++i) prm.lo[i] = T.lo_host[i];
    prm.drop_first = T.inject_drop;
    T.inject_drop = 0;
    const int stage_bytes = T.tpc * kTileA + (T.swap ? 2 * kTileA : T.ncta * 128);
    // as many stages as fit in the shared memory a block may opt into, next to the
    // kernel's static arrays, the 1 KB alignment pad and the barriers
    int dev = 0, optin = 0, stages = 0;
    size_t smem = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    auto fit = [&](const void *kern) -> int {
        cudaFuncAttributes fa;
        CK(cudaFuncGetAttributes(&fa, kern));
        const int64_t room = int64_t(optin) - int64_t(fa.sharedSizeBytes) - 1024 - (2 * 6 + 2) * 8 - 64;
        stages = int(std::min<int64_t>(6, room / stage_bytes));
        if (stages < 2) return set_err(ctx, GBFMM_ERR_INVALID_ARG, "tensor-core M2L: operator block too large");
        smem = size_t(stages) * stage_bytes + 1024 + (2 * stages + 2) * 8 + 64;
        CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
        return GBFMM_OK;
    };
    float *Sout = T.svd ? T.Sc : Sf;  // compressed: the r1 coefficients of every target cell
    if (T.svd) CK(cudaMemsetAsync(T.Sc, 0, size_t(ctx->n_cells) * T.r1 * sizeof(float), st));
    const int few = T.few_top;
    if (few >= 2) {
        if (int rc = few_alloc(ctx, n_targets)) return rc;  // (free targets may occupy more cells than the sources)
        float *part = ctx->ws().few_part;
        FewParams fp;
        fp.P = prm;
        fp.P.split = T.split && (split_levels & ((2 << few) - 4));
        fp.groups = T.groups;
        auto kern = T.tf32 ? k_m2l_few<true> : k_m2l_few<false>;
        if (int rc = fit((const void *)kern)) return rc;
        FewCount *cnt = reinterpret_cast<FewCount *>(T.few_list);
        int *list = reinterpret_cast<int *>(T.few_list) + 4;
        fp.masks = reinterpret_cast<const uint32_t *>(list + (cell_base(kFewTop + 1) - cell_base(2)));
        ctx->launches += 4;
        k_few_list<<<1, 1024, 0, st>>>(few, T.groups, std::max(1, ctx->opt.m2l_chunks), ctx->sm_count, tocc, list, cnt);
        k_few_mask<<<dim3(unsigned((cell_base(few + 1) - cell_base(2) + 127) / 128), 10), 512, 0, st>>>(
            cnt, list, occ, const_cast<uint32_t *>(fp.masks));
        kern<<<T.few_work, kTcThreads, smem, st>>>(fp, cnt, list, occ, part, T.Np, T.d_status, stages);
        k_few_sum<<<unsigned(cell_base(few + 1) - cell_base(2)), 256, 0, st>>>(
            cnt, list, part, T.Np, prm.nvalid, prm.wmax, prm.inv_op_scale, ctx->d_box, Sout, S64);
        CK(cudaGetLastError());
        prm.drop_first = 0;
    }
    if (L - 1 > few) {
        // target cells of the deeper levels: flags by slot, their scan, the list and the segments
        if (few >= 2) CK(cudaMemsetAsync(T.d_flags, 0, slot_base(few + 1) * sizeof(int), st));
        for (int l = std::max(2, few + 1); l < L; ++l) {
            ++ctx->launches;
            k_mb_flags<<<nblk(int64_t(1) << (3 * l), 256), 256, 0, st>>>(l, tocc, T.d_flags);
        }
        scan_counts(ctx, T.n_slots, T.d_flags, T.d_pos);
        ctx->launches += 2;
        k_mb_list<<<nblk(T.n_slots, 256), 256, 0, st>>>(int(T.n_slots), L, T.d_flags, T.d_pos, T.d_list);
        k_seg_table<<<1, 32, 0, st>>>(L, T.tpc, T.d_pos, T.d_seg);
        auto kern = T.tf32 ? (T.swap ? k_m2l_tc<true, true> : k_m2l_tc<true, false>)
                           : (T.swap ? k_m2l_tc<false, true> : k_m2l_tc<false, false>);
        if (int rc = fit((const void *)kern)) return rc;
        // offset chunks: each launch accumulates a run of consecutive offsets of every class's list
        // in tensor memory; the chunks' sums are added outside the tensor cores, in the local values
        const int chunks = std::max(1, std::min(189, ctx->opt.m2l_chunks));
        for (int c = 0; c < chunks; ++c) {
            prm.o_lo = (189 * c) / chunks;
            prm.o_hi = (189 * (c + 1)) / chunks;
            prm.accumulate = c > 0 ? 1 : 0;
            if (c > 0) prm.drop_first = 0;
            ++ctx->launches;
            kern<<<T.n_work, kTcThreads, smem, st>>>(prm, T.d_seg, 8 * (L - 2), T.d_list, occ, tocc, ctx->d_box, Sout, S64,
                                              T.d_status, stages, T.groups);
            CK(cudaGetLastError());
        }
    }
    if (T.svd) {
        if (fine)
            if (int rc = fine_m2l(ctx)) return rc;
        return svd_expand_s(ctx, Sf, fine);  // S = U S'
    }
    return GBFMM_OK;
}

// read and clear the device status word of the tensor-core M2L
int m2l_tc_status(gbfmm_ctx *ctx, int *out) {
    *out = 0;
    if (!ctx->tc.d_status) return GBFMM_OK;
    CK(cudaStreamSynchronize(ctx->stream));
    CK(cudaMemcpy(out, ctx->tc.d_status, sizeof(int), cudaMemcpyDeviceToHost));
    CK(cudaMemset(ctx->tc.d_status, 0, sizeof(int)));
    return GBFMM_OK;
}

void m2l_tc_free(gbfmm_ctx *ctx) {
    TcPlan &T = ctx->tc;
    svd_free(ctx, ctx->borrowed_material);
    void *ps[] = {T.Thi, T.Tlo, T.Whi, T.Wlo, T.d_status, T.d_flags, T.d_pos, T.d_list, T.d_seg, T.d_wmax,
                  T.few_list};
    for (void *q : ps)
        if (q) cudaFree(q);
    T = TcPlan{};
}
