// Near field of Algorithm 2 (the direct sum over neighbouring leaves) and L2P.
//
// Nodal forces (targets = sources): h is odd, so one h serves both directions of a point
// pair.  The sources of a leaf A are the points of the 14 leaves A + o, o in the upper half
// of the 3 x 3 x 3 neighbourhood (A itself first), as one list; a pair (target i of A, list
// entry j) with j > i adds to the strain at i and, with the sign reversed, to the one at j.
// Free targets meet the list of all 27 leaves in one direction.
//
// Work items are (leaf, target tile, list section).  A warp takes one item at a time: 32
// list entries are staged in shared memory, the item's targets go in chunks of tg lanes (a
// power of two), and lane (ti, tj) meets the tg entries of group tj one after the other in an
// order rotated by ti, so the 32 lanes of a step hold 32 different entries and add the
// reverse sums to shared memory without exchanging anything.  A list of all 14 leaves keeps
// the steps full where single leaf pairs would not (a leaf of the 1,000,000-segment walls
// holds 34 points on average); the tiles are cut so that no warp gets more than a bounded
// number of pairs, since clustered networks put a thousand points in one leaf (with one warp
// per leaf pair a 3,001-segment network took 560 ms in FP64 for 4 ms of arithmetic).
//
// The learned h (GBFMM_H_MLP) runs in the same kernel: pairs whose direction lies in an angular
// bin the calibration accepted, and farther apart than mlp_min_dist segment lengths, take the
// network in its tabulated form, the others the plain rule.  Pairs are queued by kind and
// worked off 32 at a time, since lanes of mixed kinds would pay for both.
//
// Sums: an item writes one row of six doubles (strain) for every target and, in the
// symmetric form, for every list entry of its section; k_near_combine adds a point's rows in
// a fixed order, applies the stiffness and adds the far field (L2P).  Nothing depends on which
// warp takes which item or on where the rows lie, so results repeat exactly.
//
// Bound: instruction issue and the FMA pipe (250,000-segment walls, cubic, Q = 16: issue slots 75 %
// and FMA pipe 59 % busy, ~1,280 warp instructions per 32 pairs for both directions, DRAM 28
// GB/s).  Near field with L2P: those walls 33.9 ms, 50,003 segments of loops (Q = 32) 8.8, 6,101 in a
// turned crystal 3.0, 3,001 in FP64 12.1, 2,000 isotropic in FP64 2.7.  Whole calls, with one h by
// the pointwise rule, 108-entry source tensors and one warp per leaf pair before: 83 -> 45 ms, 36 ->
// 10.2, 80 to 90 -> 3.2, 490 to 580 -> 15.8, 66 to 146 -> 3.8 (uneven leaves made these vary).
//
// Precision of the FP32 form: positions are FP32 pairs (value + remainder) relative to the
// leaf centre, so every separation is correct to its own rounding, also of close pairs; h and
// the contraction run in FP32; every sum over pairs is a two-float sum (~48 bits).
#include <algorithm>
#include <cmath>

#include "internal.cuh"
#include "kernel_math.cuh"
#include "unit_circle.cuh"

namespace {

inline unsigned nblk(int64_t n, int b) { return unsigned((n + b - 1) / b); }

__device__ __forceinline__ void cell_xyz3(int64_t lin, int n, int &x, int &y, int &z) {
    x = int(lin % n);
    y = int((lin / n) % n);
    z = int(lin / (int64_t(n) * n));
}

// h models of the near kernels: closed form; moment form of a cubic medium; any medium, point by
// point (FP32) or in moment form (FP64, and FP32 beside the learned h)
constexpr int HM_ISO = 0, HM_CUBIC = 1, HM_POINTS = 2, HM_GENERAL = 3;

// ---------------------------------------------------------------- point records
// FP32: four float4 per point, (y hi, |S|^2) (y lo, segment) (b', 0) (S, 0), y relative to the
// leaf centre; FP64: five double2, (y0, y1) (y2, segment) (b0', b1') (b2', S0) (S1, S2), y
// absolute.  b' = omega / 2 times the Burgers vector times the factor of h.  Structure of arrays
// (row r of point i at r n + i), so a staging warp reads whole lines: 64 (80) bytes a point
// where a 6 x 18 tensor takes 432 (864).
struct GaussWeights {
    double w[GB_MAXG];
    int n;
};

__device__ __forceinline__ void leaf_centre(const TreeBox *box, int nl, int64_t leaf, double c[3]) {
    int cx, cy, cz;
    cell_xyz3(leaf, nl, cx, cy, cz);
    const double h = box->H / nl;
    c[0] = box->origin[0] + (cx + 0.5) * h;
    c[1] = box->origin[1] + (cy + 0.5) * h;
    c[2] = box->origin[2] + (cz + 0.5) * h;
}

__device__ __forceinline__ void split_position(const double *y, const double c[3], float hi[3], float lo[3]) {
    for (int d = 0; d < 3; ++d) {
        const double v = y[d] - c[d];
        hi[d] = float(v);
        lo[d] = float(v - double(hi[d]));
    }
}

template <typename R>
__global__ void k_near_records(int64_t N, int L, const TreeBox *__restrict__ box, const double *__restrict__ y,
                               const int *__restrict__ perm, const int *__restrict__ pleaf,
                               const double *__restrict__ segv, GaussWeights gw, double fac, void *__restrict__ rec) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= N) return;
    const int k = perm[i];
    const int64_t s = k / gw.n;
    const double f = 0.5 * gw.w[k - int(s) * gw.n] * fac;
    double S[3], b[3];
    for (int d = 0; d < 3; ++d) {
        S[d] = segv[6 * s + d];
        b[d] = f * segv[6 * s + 3 + d];
    }
    if constexpr (sizeof(R) == 4) {
        float4 *r = static_cast<float4 *>(rec);
        double c[3];
        leaf_centre(box, 1 << (L - 1), pleaf[i], c);
        float hi[3], lo[3];
        split_position(y + 3 * i, c, hi, lo);
        r[i] = make_float4(hi[0], hi[1], hi[2], float(S[0] * S[0] + S[1] * S[1] + S[2] * S[2]));
        r[N + i] = make_float4(lo[0], lo[1], lo[2], __int_as_float(int(s)));
        r[2 * N + i] = make_float4(float(b[0]), float(b[1]), float(b[2]), 0.f);
        r[3 * N + i] = make_float4(float(S[0]), float(S[1]), float(S[2]), 0.f);
    } else {
        double2 *r = static_cast<double2 *>(rec);
        r[i] = make_double2(y[3 * i], y[3 * i + 1]);
        r[N + i] = make_double2(y[3 * i + 2], __longlong_as_double(s));
        r[2 * N + i] = make_double2(b[0], b[1]);
        r[3 * N + i] = make_double2(b[2], S[0]);
        r[4 * N + i] = make_double2(S[1], S[2]);
    }
}

// free targets, sorted by leaf: the position rows alone, segment -1
template <typename R>
__global__ void k_near_targets(int64_t n, int L, const TreeBox *__restrict__ box, const double *__restrict__ x,
                               const int *__restrict__ leaf_of, void *__restrict__ rec) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= n) return;
    if constexpr (sizeof(R) == 4) {
        float4 *r = static_cast<float4 *>(rec);
        double c[3];
        leaf_centre(box, 1 << (L - 1), leaf_of[i], c);
        float hi[3], lo[3];
        split_position(x + 3 * i, c, hi, lo);
        r[i] = make_float4(hi[0], hi[1], hi[2], 0.f);
        r[n + i] = make_float4(lo[0], lo[1], lo[2], __int_as_float(-1));
    } else {
        double2 *r = static_cast<double2 *>(rec);
        r[i] = make_double2(x[3 * i], x[3 * i + 1]);
        r[n + i] = make_double2(x[3 * i + 2], __longlong_as_double(-1));
    }
}

// ---------------------------------------------------------------- work plan
// Per leaf with targets: where its rows start, the length of its source list, and its tiles:
// ca target tiles of ta targets (a split leaf of the adaptive tree: ca groups of children), cb
// list sections of sb entries.  Rows: [cb][targets] forward, then [ca][list] reverse.
struct NearPlan {
    long long base;
    int ns, ta, ca, sb, cb, pad;
};
struct NearItem {
    int leaf, a, b, pad;
};

constexpr int kPlanSizes = 8;  // candidates of pairs per item: 512 4^k, the last without bound
// counters: [0] pairs, [1 + k] rows, [1 + kPlanSizes + k] items of candidate k, then the
// allocation cursors of rows and items and the items taken
constexpr int kCntRows = 1 + 2 * kPlanSizes, kCntItems = kCntRows + 1, kCntNext = kCntItems + 1, kCnt = kCntNext + 1;

__device__ __forceinline__ int64_t plan_size(int k) {
    return k == kPlanSizes - 1 ? (int64_t(1) << 62) : int64_t(512) << (2 * k);
}

// tiles of a leaf with nt targets and ns list entries at w pairs per item.  List sections first
// (a section costs nt rows, a target tile ns, and ns is about 14 nt), at least 32 entries long;
// then target tiles of a multiple of 8.  A split leaf's tiles are groups of children.
__device__ __forceinline__ void plan_tiles(int nt, int ns, bool split, int64_t w, int &ta, int &ca, int &sb, int &cb) {
    const int64_t pairs = int64_t(nt) * ns;
    ta = nt, ca = 1, sb = ns, cb = 1;
    if (ns == 0) return;
    if (split) {
        while (ca < 8 && pairs / ca > w) ca *= 2;
        ta = 8 / ca;
        const int64_t c = min((pairs / ca + w - 1) / w, int64_t((ns + 31) / 32));
        if (c > 1) {
            sb = int(((ns + c - 1) / c + 31) / 32 * 32);
            cb = (ns + sb - 1) / sb;
        }
        return;
    }
    if (pairs <= w) return;
    const int64_t c = min((pairs + w - 1) / w, int64_t((ns + 31) / 32));
    sb = int(((ns + c - 1) / c + 31) / 32 * 32);
    cb = (ns + sb - 1) / sb;
    const int64_t each = int64_t(nt) * min(sb, ns);
    if (each > w) {
        const int64_t t = min((each + w - 1) / w, int64_t((nt + 7) / 8));
        ta = int(((nt + t - 1) / t + 7) / 8 * 8);
        ca = (nt + ta - 1) / ta;
    }
}

// leaf A + o of direction nb (0..26), -1 outside the grid
__device__ __forceinline__ int64_t neighbour(int x, int y, int z, int nb, int nl) {
    const int bx = x + nb % 3 - 1, by = y + (nb / 3) % 3 - 1, bz = z + nb / 9 - 1;
    if (bx < 0 || by < 0 || bz < 0 || bx >= nl || by >= nl || bz >= nl) return -1;
    return (int64_t(bz) * nl + by) * nl + bx;
}

// pairs of the pass and, for every candidate size, its rows and items (exact integer sums)
template <bool SYM>
__global__ void __launch_bounds__(256) k_near_totals(int64_t nl, int L, const int *__restrict__ tstart,
                                                     const int *__restrict__ sstart, const int *__restrict__ ref_start,
                                                     unsigned long long *__restrict__ cnt) {
    constexpr int D0 = SYM ? 13 : 0;
    const int64_t l = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    long long v[1 + 2 * kPlanSizes];
    for (int i = 0; i < 1 + 2 * kPlanSizes; ++i) v[i] = 0;
    if (l < nl) {
        const int nt = tstart[l + 1] - tstart[l];
        if (nt > 0) {
            const int nlv = 1 << (L - 1);
            int x, y, z, ns = 0;
            cell_xyz3(l, nlv, x, y, z);
            for (int nb = D0; nb < 27; ++nb) {
                const int64_t B = neighbour(x, y, z, nb, nlv);
                if (B >= 0) ns += sstart[B + 1] - sstart[B];
            }
            const bool split = ref_start && ref_start[l + 1] > ref_start[l];
            v[0] = (long long)nt * ns;
            for (int k = 0; k < kPlanSizes; ++k) {
                int ta, ca, sb, cb;
                plan_tiles(nt, ns, split, plan_size(k), ta, ca, sb, cb);
                v[1 + k] = (long long)cb * nt + (SYM ? (long long)ca * ns : 0);
                v[1 + kPlanSizes + k] = (long long)ca * cb;
            }
        }
    }
    __shared__ long long sm[8];
    for (int i = 0; i < 1 + 2 * kPlanSizes; ++i) {
        long long s = v[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) sm[threadIdx.x / 32] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long t = 0;
            for (int w = 0; w < int(blockDim.x) / 32; ++w) t += sm[w];
            if (t) atomicAdd(&cnt[i], (unsigned long long)t);
        }
    }
}

// The size is the smallest candidate whose rows and items fit the buffers and that leaves a
// resident warp at most sixteen items (four at least: a warp's last item is then a small part of its
// time; 50,000 segments, near field: 9.3 ms with eight to two items, 8.5 with these, 8.6 with twice
// as many), but not above 32,768 pairs where the buffers allow (about 1 ms of a warp): every
// quantity depends on the network and the options alone, so results do not depend on a buffer's
// history.
template <bool SYM>
__global__ void __launch_bounds__(256) k_near_plan(int64_t nl, int L, int warps, long long cap_rows, long long cap_items,
                                                   const int *__restrict__ tstart, const int *__restrict__ sstart,
                                                   const int *__restrict__ ref_start,
                                                   unsigned long long *__restrict__ cnt, NearPlan *__restrict__ plan,
                                                   int *__restrict__ lp, NearItem *__restrict__ items) {
    constexpr int D0 = SYM ? 13 : 0, ND = 27 - D0;
    const int64_t l = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    const int lane = threadIdx.x % 32;
    int nt = 0, ns = 0, ta = 1, ca = 0, sb = 1, cb = 0;
    if (l < nl) nt = tstart[l + 1] - tstart[l];
    if (nt > 0) {
        const int nlv = 1 << (L - 1);
        int x, y, z;
        cell_xyz3(l, nlv, x, y, z);
        for (int d = 0; d < ND; ++d) {
            const int64_t B = neighbour(x, y, z, D0 + d, nlv);
            lp[ND * l + d] = ns;
            if (B >= 0) ns += sstart[B + 1] - sstart[B];
        }
        int64_t want = int64_t(cnt[0] / (16ull * (unsigned long long)warps));
        want = min(want, int64_t(32768));
        int k = 0;
        while (k < kPlanSizes - 1 && (plan_size(k) < want || (long long)cnt[1 + k] > cap_rows ||
                                      (long long)cnt[1 + kPlanSizes + k] > cap_items))
            ++k;
        plan_tiles(nt, ns, ref_start && ref_start[l + 1] > ref_start[l], plan_size(k), ta, ca, sb, cb);
    }
    // one allocation per warp
    long long rows = (long long)cb * nt + (SYM ? (long long)ca * ns : 0), n_it = (long long)ca * cb;
    long long r0 = rows, i0 = n_it;
    for (int o = 1; o < 32; o <<= 1) {
        const long long a = __shfl_up_sync(0xffffffffu, r0, o), b = __shfl_up_sync(0xffffffffu, i0, o);
        if (lane >= o) r0 += a, i0 += b;
    }
    long long rb = 0, ib = 0;
    if (lane == 31) {
        if (r0) rb = (long long)atomicAdd(&cnt[kCntRows], (unsigned long long)r0);
        if (i0) ib = (long long)atomicAdd(&cnt[kCntItems], (unsigned long long)i0);
    }
    rb = __shfl_sync(0xffffffffu, rb, 31) + r0 - rows;
    ib = __shfl_sync(0xffffffffu, ib, 31) + i0 - n_it;
    if (nt > 0) {
        plan[l] = NearPlan{rb, ns, ta, ca, sb, cb, 0};
        for (int a = 0; a < ca; ++a)
            for (int b = 0; b < cb; ++b) items[ib++] = NearItem{int(l), a, b, 0};
    }
}

// ---------------------------------------------------------------- pair kernel
// Two-float sums: the value is hi + lo, and each addition keeps its exact rounding error
// (Knuth's two-sum), so a sum of FP32 terms carries ~48 mantissa bits without FP64 arithmetic
// (FP64 runs at a small fraction of the FP32 rate on this part).
__device__ __forceinline__ void tsum2(float &hi, float &lo, float bhi, float blo) {
    const float s = hi + bhi;
    const float bb = s - hi;
    lo += ((hi - (s - bb)) + (bhi - bb)) + blo;
    hi = s;
}

// a sum in the kernel's precision: two-float or FP64
template <typename R>
struct Acc;
template <>
struct Acc<float> {
    float hi, lo;
    __device__ __forceinline__ void zero() { hi = lo = 0.f; }
    // a pair's value, of any size beside the sum: the ordered form (four operations for six) loses up to
    // an ulp of a term larger than the sum, so a close pair would cost the others' digits (250,000
    // segments, whole pass: 43.5 ms with the ordered form, 44.3 with this one)
    __device__ __forceinline__ void add(float v) {
        const float s = hi + v;
        const float bb = s - hi;
        lo += (hi - (s - bb)) + (v - bb);
        hi = s;
    }
    __device__ __forceinline__ void add(const Acc &o) { tsum2(hi, lo, o.hi, o.lo); }
    __device__ __forceinline__ Acc shfl_xor(int o) const {
        return Acc{__shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lo, o)};
    }
    __device__ __forceinline__ double value() const { return double(hi) + double(lo); }
};
template <>
struct Acc<double> {
    double v;
    __device__ __forceinline__ void zero() { v = 0.0; }
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add(const Acc &o) { v += o.v; }
    __device__ __forceinline__ Acc shfl_xor(int o) const { return Acc{__shfl_xor_sync(0xffffffffu, v, o)}; }
    __device__ __forceinline__ double value() const { return v; }
};

// a point in registers
template <typename R>
struct Pt;
template <>
struct Pt<float> {
    float hi[3], lo[3], b[3], S[3], len2;
    int seg;
};
template <>
struct Pt<double> {
    double hi[3], b[3], S[3], len2;
    long long seg;
};

// rows of staged points in shared memory
template <typename R, int N>
struct Stage;
template <int N>
struct Stage<float, N> {
    float4 r[4][N];
    __device__ __forceinline__ void load_target(const void *rec, int64_t n, int64_t i, int k, bool full) {
        const float4 *g = static_cast<const float4 *>(rec);
        r[0][k] = __ldg(g + i);
        r[1][k] = __ldg(g + n + i);
        if (full) {
            r[2][k] = __ldg(g + 2 * n + i);
            r[3][k] = __ldg(g + 3 * n + i);
        }
    }
    // position moved by o leaf edges (eh + el, two floats) to the target leaf's centre
    __device__ __forceinline__ void load_source(const void *rec, int64_t n, int64_t i, int k, int ox, int oy, int oz,
                                                float eh, float el) {
        const float4 *g = static_cast<const float4 *>(rec);
        float4 a = __ldg(g + i), c = __ldg(g + n + i);
        tsum2(a.x, c.x, float(ox) * eh, float(ox) * el);
        tsum2(a.y, c.y, float(oy) * eh, float(oy) * el);
        tsum2(a.z, c.z, float(oz) * eh, float(oz) * el);
        r[0][k] = a;
        r[1][k] = c;
        r[2][k] = __ldg(g + 2 * n + i);
        r[3][k] = __ldg(g + 3 * n + i);
    }
    __device__ __forceinline__ Pt<float> get(int k, bool full) const {
        Pt<float> p;
        const float4 a = r[0][k], c = r[1][k];
        p.hi[0] = a.x, p.hi[1] = a.y, p.hi[2] = a.z, p.len2 = a.w;
        p.lo[0] = c.x, p.lo[1] = c.y, p.lo[2] = c.z, p.seg = __float_as_int(c.w);
        if (full) {
            const float4 b = r[2][k], s = r[3][k];
            p.b[0] = b.x, p.b[1] = b.y, p.b[2] = b.z;
            p.S[0] = s.x, p.S[1] = s.y, p.S[2] = s.z;
        }
        return p;
    }
};
template <int N>
struct Stage<double, N> {
    double2 r[5][N];
    __device__ __forceinline__ void load_target(const void *rec, int64_t n, int64_t i, int k, bool full) {
        const double2 *g = static_cast<const double2 *>(rec);
        for (int q = 0; q < (full ? 5 : 2); ++q) r[q][k] = __ldg(g + q * n + i);
    }
    __device__ __forceinline__ void load_source(const void *rec, int64_t n, int64_t i, int k, int, int, int, float,
                                                float) {
        load_target(rec, n, i, k, true);
    }
    __device__ __forceinline__ Pt<double> get(int k, bool full) const {
        Pt<double> p;
        p.hi[0] = r[0][k].x, p.hi[1] = r[0][k].y, p.hi[2] = r[1][k].x;
        p.seg = __double_as_longlong(r[1][k].y);
        if (full) {
            p.b[0] = r[2][k].x, p.b[1] = r[2][k].y, p.b[2] = r[3][k].x;
            p.S[0] = r[3][k].y, p.S[1] = r[4][k].x, p.S[2] = r[4][k].y;
        }
        return p;
    }
};

// separation x_i - y_j
__device__ __forceinline__ void separation(const Pt<float> &p, const Pt<float> &s, float d[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = (p.hi[k] - s.hi[k]) + (p.lo[k] - s.lo[k]);
}
__device__ __forceinline__ void separation(const Pt<double> &p, const Pt<double> &s, double d[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = p.hi[k] - s.hi[k];
}

constexpr int kTargets = 64;  // targets of an item staged at a time
constexpr int kRanges = 112;  // list ranges of one target leaf: 14 leaves x 8 children

template <typename R, bool SYM, bool LEARN>
struct WarpShared {
    static constexpr int kEntries = LEARN ? 64 : 32;  // list entries staged at a time
    Stage<R, kTargets> tg;
    Stage<R, kEntries> sr;
    Acc<R> fwd[6][kTargets];
    Acc<R> rev[SYM ? 6 : 1][SYM ? kEntries : 1];
    int src[kEntries], pos[kEntries];  // sorted index and list position of the staged entries
    int rstart[kRanges], rpos[kRanges], rpre[kRanges + 1];
    unsigned char rdir[kRanges];
    unsigned short queue[LEARN ? 2 : 1][LEARN ? 64 : 2];  // queued pairs: the plain rule's, the network's
};

// learned h: accepted bins, their polynomials, and the smallest distance squared over |S|^2
struct NearLearned {
    const uint32_t *binmask;  // bit set: the bin takes the plain rule
    const float4 *poly;       // [bin][27]: 18 components x 6 coefficients (mlp.cu)
    float rmin2, m2;
    float fac;                // 4 pi Q times the kernel's unit of the moduli: what the pairs' Burgers vectors leave out
};

struct NearTree {
    int L;
    int64_t N;            // source points
    int64_t n_t;          // target points
    const TreeBox *box;
    const int *tstart, *sstart;
    const int *ref_start, *child_start;  // adaptive tree (else null)
    const void *trec, *srec;
    const NearPlan *plan;
    const int *lp;
    const NearItem *items;
    unsigned long long *cnt;
    double *rows;
};

template <typename R>
constexpr int near_warps() { return sizeof(R) == 4 ? 4 : 2; }
template <typename R>
constexpr int near_blocks() { return sizeof(R) == 4 ? 3 : 4; }

// stress rows of one pair by the plain rule
template <typename R, int HM>
__device__ __forceinline__ void rows_plain(const NearMedium<R> &md, const R *tab, const R T[3], R Y[3][6]) {
    if constexpr (HM == HM_CUBIC) {
        rows_cubic<R>(md, tab, T, Y);
    } else {
        R hs[18];
        if constexpr (HM == HM_POINTS)
            h_general_points(md, tab, T, hs);
        else
            h_general_moments<R>(md, tab, T, hs);
        stress_rows<R, true>(md, hs, Y);
    }
}

// Angular bin of a direction folded into the upper half-space (h is odd): dominant axis face
// (+z, +x, -x, +y, -y) and a 16 x 16 grid of the two other components; (u, v): the place in the
// bin, -1 .. 1; the sign of the fold is returned.  Any length.
__device__ __forceinline__ float dir_bin(const float d[3], int &bin, float &u, float &v) {
    const float sg = (d[2] > 0.f || (d[2] == 0.f && (d[1] > 0.f || (d[1] == 0.f && d[0] >= 0.f)))) ? 1.f : -1.f;
    const float x = sg * d[0], y = sg * d[1], z = sg * d[2];
    const float ax = fabsf(x), ay = fabsf(y), az = fabsf(z);
    int f;
    float p, q, m;
    if (az >= ax && az >= ay) {
        f = 0, p = x, q = y, m = az;
    } else if (ax >= ay) {
        f = x > 0.f ? 1 : 2, p = y, q = z, m = ax;
    } else {
        f = y > 0.f ? 3 : 4, p = x, q = z, m = ay;
    }
    const float im = recip(m), tp = (p * im + 1.f) * 8.f, tq = (q * im + 1.f) * 8.f;
    const int bu = min(15, max(0, int(tp))), bv = min(15, max(0, int(tq)));
    bin = f * 256 + bu * 16 + bv;
    u = 2.f * (tp - float(bu)) - 1.f;
    v = 2.f * (tq - float(bv)) - 1.f;
    return sg;
}

// h of one pair by the network's polynomial in its bin, in the pair kernel's unit
__device__ __forceinline__ void h_learned(const NearLearned &ln, const float d[3], float hs[18]) {
    int bin;
    float u, v;
    const float sg = ln.fac * dir_bin(d, bin, u, v);
    const float b1 = u, b2 = v, b3 = u * u - ln.m2, b4 = u * v, b5 = v * v - ln.m2;
    const float4 *q = ln.poly + 27 * bin;
#pragma unroll
    for (int k = 0; k < 18; k += 2) {
        const float4 a = __ldg(q + 3 * (k / 2)), b = __ldg(q + 3 * (k / 2) + 1), c = __ldg(q + 3 * (k / 2) + 2);
        hs[k] = sg * (a.x + a.y * b1 + a.z * b2 + a.w * b3 + b.x * b4 + b.y * b5);
        hs[k + 1] = sg * (b.z + b.w * b1 + c.x * b2 + c.y * b3 + c.z * b4 + c.w * b5);
    }
}

// A block of nt targets (from point tb) against the ns staged entries with the learned h.  The
// pairs are visited along the diagonals of an M x M square (M = 32, or 64 where either side is
// longer), classified, and queued by kind; 32 queued pairs make a step.  Pairs fewer than M - 1
// places apart on that path share neither target nor entry, so a step whose pairs are adds to
// the sums directly (the plain queue nearly always); otherwise lanes that share one add in the
// order of their numbers.  Sorting costs ~90 instructions a visited pair and saves the ~1,900 of
// the general rule for each learned one (100,000 segments in a turned crystal, Q = 32, a fifth
// of the pairs learned; with the network's layers evaluated per pair, one-sided: 2,236 ms).
template <int HM, bool SYM, typename Shared>
__device__ __forceinline__ void learned_block(Shared &ws, const NearMedium<float> &md, const NearLearned &ln,
                                              const float *tab, const uint32_t *mask, int tb, int nt, int ns, int lane) {
    const int sh = nt > 32 || ns > 32 ? 6 : 5, M = 1 << sh;
    const unsigned below = (1u << lane) - 1u;
    int n0 = 0, n1 = 0;  // queued: plain, learned
    for (int q0 = 0; q0 < M * M; q0 += 32) {
        const int ti = (q0 + lane) & (M - 1), jl = (ti + (q0 >> sh)) & (M - 1);
        if ((q0 & (M - 1)) < nt) {
            bool on = ti < nt && jl < ns, net = false;
            if (SYM) on = on && ws.src[jl] > tb + ti;
            if (on) {
                const Pt<float> pi = ws.tg.get(ti, false), pj = ws.sr.get(jl, false);
                float d[3], u, v;
                separation(pi, pj, d);
                const float r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
                on = pj.seg != pi.seg && r2 > 0.f;
                int bin;
                dir_bin(d, bin, u, v);
                net = r2 >= ln.rmin2 * fmaxf(pi.len2, pj.len2) && !((mask[bin >> 5] >> (bin & 31)) & 1u);
            }
            const unsigned m0 = __ballot_sync(0xffffffffu, on && !net), m1 = __ballot_sync(0xffffffffu, on && net);
            if (on) ws.queue[net][net ? n1 + __popc(m1 & below) : n0 + __popc(m0 & below)] = (unsigned short)(q0 + lane);
            n0 += __popc(m0);
            n1 += __popc(m1);
        }
        const bool last = q0 + 32 >= M * M;
#pragma unroll 1
        for (int w = 0; w < 2; ++w) {
            int n = w ? n1 : n0;
            while (n >= 32 || (last && n > 0)) {
                __syncwarp();
                const int cnt = min(n, 32);
                const bool on = lane < cnt;
                const int place = on ? ws.queue[w][lane] : 0;
                const int span = ws.queue[w][cnt - 1] - ws.queue[w][0];
                const int it = place & (M - 1), je = (it + (place >> sh)) & (M - 1);
                float ef[6], er[6];
                if (on) {
                    const Pt<float> pi = ws.tg.get(it, SYM), pj = ws.sr.get(je, true);
                    float d[3];
                    separation(pi, pj, d);
                    const float r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
                    const float ir = rsqrt_refined(r2), ir2 = ir * ir;
                    float Y[3][6];
                    if (w == 0) {
                        const float T[3] = {d[0] * ir, d[1] * ir, d[2] * ir};
                        rows_plain<float, HM>(md, tab, T, Y);
                    } else {
                        float hs[18];
                        h_learned(ln, d, hs);
                        stress_rows<float, HM >= HM_POINTS>(md, hs, Y);
                    }
                    strain_of<float>(Y, pj.b[0], pj.b[1], pj.b[2], ir2 * pj.S[0], ir2 * pj.S[1], ir2 * pj.S[2], ef);
                    if (SYM)
                        strain_of<float>(Y, pi.b[0], pi.b[1], pi.b[2], -ir2 * pi.S[0], -ir2 * pi.S[1], -ir2 * pi.S[2],
                                         er);
                }
                int ri = on ? 0 : -1, rj = ri, rounds = 0;  // this lane's turn at its target and its entry
                if (span >= M - 1) {
                    ri = __popc(__match_any_sync(0xffffffffu, on ? it : 64 + lane) & below);
                    rj = __popc(__match_any_sync(0xffffffffu, on ? je : 64 + lane) & below);
                    if (!on) ri = rj = -1;
                    rounds = __reduce_max_sync(0xffffffffu, max(ri, rj));
                }
#pragma unroll 1
                for (int r = 0; r <= rounds; ++r) {
                    if (ri == r)
#pragma unroll
                        for (int e = 0; e < 6; ++e) ws.fwd[e][it].add(ef[e]);
                    if (SYM && rj == r)
#pragma unroll
                        for (int e = 0; e < 6; ++e) ws.rev[e][je].add(er[e]);
                    __syncwarp();
                }
                // the rest of the queue moves up
                n -= cnt;
                const unsigned short rest = lane < n ? ws.queue[w][32 + lane] : (unsigned short)0;
                __syncwarp();
                if (lane < n) ws.queue[w][lane] = rest;
            }
            if (w) n1 = n;
            else n0 = n;
        }
    }
    __syncwarp();
}

template <typename R, int HM, bool SYM, bool LEARN>
__global__ void __launch_bounds__(near_warps<R>() * 32, near_blocks<R>())
    k_near_pairs(const __grid_constant__ NearTree tr, const __grid_constant__ NearMedium<R> md,
                 const __grid_constant__ NearLearned ln) {
    constexpr int NW = near_warps<R>(), D0 = SYM ? 13 : 0, ND = 27 - D0;
    extern __shared__ __align__(16) unsigned char sm_near[];
    typedef WarpShared<R, SYM, LEARN> Shared;
    Shared &ws = reinterpret_cast<Shared *>(sm_near)[threadIdx.x / 32];
    R *tab = reinterpret_cast<R *>(sm_near + NW * sizeof(Shared));
    const int lane = threadIdx.x % 32;
    __shared__ uint32_t s_mask[LEARN ? 48 : 1];
    if constexpr (HM == HM_POINTS)
        point_table(md.Q, tab);
    else if (HM != HM_ISO)
        moment_table<R>(md.Q, md.np, tab);
    if (LEARN)
        for (int i = threadIdx.x; i < 40; i += blockDim.x) s_mask[i] = ln.binmask[i];
    __syncthreads();
    const int nlv = 1 << (tr.L - 1);
    const double edge = tr.box->H / nlv;
    const float eh = float(edge), el = float(edge - double(eh));
    const long long n_items = (long long)tr.cnt[kCntItems];
    while (true) {
        long long it = 0;
        if (lane == 0) it = (long long)atomicAdd(&tr.cnt[kCntNext], 1ull);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_items) return;
        const NearItem item = tr.items[it];
        const int64_t A = item.leaf;
        const NearPlan pl = tr.plan[A];
        const int tA0 = tr.tstart[A], tA1 = tr.tstart[A + 1], nt = tA1 - tA0;
        int ax, ay, az;
        cell_xyz3(A, nlv, ax, ay, az);
        const int s0 = item.b * pl.sb, s1 = min(pl.ns, s0 + pl.sb);
        const long long fbase = pl.base + (long long)item.b * nt;
        const long long rbase = pl.base + (long long)pl.cb * nt + (long long)item.a * pl.ns;
        const int rA = SYM && tr.ref_start && tr.ref_start[A + 1] > tr.ref_start[A] ? tr.ref_start[A] : -1;
        bool add = false;  // reverse rows: store, or add to what an earlier target block stored
        if (SYM && rA >= 0) {
            // a split leaf's children meet different parts of the list: the rows start from zero
            for (int k = s0 + lane; k < s1; k += 32)
                for (int e = 0; e < 6; ++e) tr.rows[(rbase + k) * 6 + e] = 0.0;
            add = true;
            __syncwarp();
        }
        const int g0 = rA >= 0 ? item.a * pl.ta : 0, g1 = rA >= 0 ? g0 + pl.ta : 1;  // children of the tile
        for (int ch = g0; ch < g1; ++ch) {
            const int b0 = rA >= 0 ? tr.child_start[9 * rA + ch] : tA0 + item.a * pl.ta;
            const int b1 = rA >= 0 ? tr.child_start[9 * rA + ch + 1] : min(tA1, tA0 + (item.a + 1) * pl.ta);
            for (int tb = b0; tb < b1; tb += kTargets) {
                const int nb_t = min(kTargets, b1 - tb);
                __syncwarp();
                // the block's part of the list: whole leaves, or (two split leaves) the children
                // adjacent to this one; in the own leaf only entries from the block's start on
                int nr = 0, total = 0;
                const int ne = rA >= 0 ? ND * 8 : ND;
                for (int e0 = 0; e0 < ne; e0 += 32) {
                    const int e = e0 + lane;
                    int len = 0, start = 0, lpos = 0, dir = 0;
                    if (e < ne) {
                        dir = rA >= 0 ? e / 8 : e;
                        const int ss = rA >= 0 ? e % 8 : 0, nb = D0 + dir;
                        const int64_t B = neighbour(ax, ay, az, nb, nlv);
                        if (B >= 0) {
                            const int sB0 = tr.sstart[B], sB1 = tr.sstart[B + 1];
                            lpos = tr.lp[ND * A + dir];
                            const int rB = rA >= 0 && dir > 0 && tr.ref_start[B + 1] > tr.ref_start[B] ? tr.ref_start[B] : -1;
                            if (rB >= 0) {
                                const int ox = nb % 3 - 1, oy = (nb / 3) % 3 - 1, oz = nb / 9 - 1;
                                const int dx = 2 * ox + (ss & 1) - (ch & 1),
                                          dy = 2 * oy + ((ss >> 1) & 1) - ((ch >> 1) & 1),
                                          dz = 2 * oz + (ss >> 2) - (ch >> 2);
                                if (abs(dx) <= 1 && abs(dy) <= 1 && abs(dz) <= 1) {
                                    start = tr.child_start[9 * rB + ss];
                                    len = tr.child_start[9 * rB + ss + 1] - start;
                                    lpos += start - sB0;
                                }
                            } else if (ss == 0) {
                                start = sB0, len = sB1 - sB0;
                            }
                            int skip = max(0, s0 - lpos);
                            if (SYM && dir == 0) skip = max(skip, tb - tA0);
                            len = max(0, min(len, s1 - lpos) - skip);
                            start += skip, lpos += skip;
                        }
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, len > 0);
                    int pre = len;
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, pre, o);
                        if (lane >= o) pre += v;
                    }
                    if (len > 0) {
                        const int k = nr + __popc(m & ((1u << lane) - 1u));
                        ws.rstart[k] = start, ws.rpos[k] = lpos, ws.rpre[k] = total + pre - len;
                        ws.rdir[k] = (unsigned char)(D0 + dir);
                    }
                    nr += __popc(m);
                    total += __shfl_sync(0xffffffffu, pre, 31);
                }
                for (int k = lane; k < nb_t; k += 32) {
                    ws.tg.load_target(tr.trec, tr.n_t, tb + k, k, SYM);
                    for (int e = 0; e < 6; ++e) ws.fwd[e][k].zero();
                }
                for (int m0 = 0; m0 < total; m0 += Shared::kEntries) {
                    const int ns = min(Shared::kEntries, total - m0);
                    __syncwarp();
                    for (int k = lane; k < ns; k += 32) {
                        int lo = 0, hi = nr;  // last range that starts at or before this entry
                        while (hi - lo > 1) {
                            const int mid = (lo + hi) >> 1;
                            if (ws.rpre[mid] <= m0 + k) lo = mid;
                            else hi = mid;
                        }
                        const int off = m0 + k - ws.rpre[lo], j = ws.rstart[lo] + off, nb = ws.rdir[lo];
                        ws.src[k] = j;
                        ws.pos[k] = ws.rpos[lo] + off;
                        ws.sr.load_source(tr.srec, tr.N, j, k, nb % 3 - 1, (nb / 3) % 3 - 1, nb / 9 - 1, eh, el);
                    }
                    if (SYM)
                        for (int k = lane; k < Shared::kEntries; k += 32)
                            for (int e = 0; e < 6; ++e) ws.rev[e][k].zero();
                    __syncwarp();
                    if constexpr (LEARN) learned_block<HM, SYM>(ws, md, ln, tab, s_mask, tb, nb_t, ns, lane);
                    for (int c0 = LEARN ? nb_t : 0; c0 < nb_t;) {
                        // tg steps cover tg targets: the next power of two where that wastes at most
                        // two steps, else the largest that fits
                        const int left = nb_t - c0;
                        const int tg = left >= 30 ? 32 : left >= 15 ? 16 : left >= 7 ? 8 : left >= 3 ? 4 : left;
                        const int ti = lane & (tg - 1), tj = lane / tg;
                        const int i = tb + c0 + ti;
                        const bool vi = ti < left;
                        const Pt<R> pi = ws.tg.get(vi ? c0 + ti : 0, SYM);
                        Acc<R> f[6];
#pragma unroll
                        for (int e = 0; e < 6; ++e) f[e].zero();
                        for (int s = 0; s < tg; ++s) {
                            const int jl = tj * tg + ((ti + s) & (tg - 1));
                            bool on = vi && jl < ns;
                            if (SYM) on = on && ws.src[jl] > i;
                            if (on) {
                                const Pt<R> pj = ws.sr.get(jl, true);
                                R d[3];
                                separation(pi, pj, d);
                                const R r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
                                if (pj.seg != pi.seg && r2 > R(0)) {
                                    const R ir = rsqrt_refined(r2), ir2 = ir * ir;
                                    const R T[3] = {d[0] * ir, d[1] * ir, d[2] * ir};
                                    R Y[3][6], e6[6];
                                    if constexpr (HM != HM_ISO) rows_plain<R, HM>(md, tab, T, Y);
                                    auto strain = [&](const Pt<R> &p, R f) {
                                        if constexpr (HM == HM_ISO)
                                            strain_iso<R>(md, T, p.b[0], p.b[1], p.b[2], f * p.S[0], f * p.S[1],
                                                          f * p.S[2], e6);
                                        else
                                            strain_of<R>(Y, p.b[0], p.b[1], p.b[2], f * p.S[0], f * p.S[1], f * p.S[2],
                                                         e6);
                                    };
                                    strain(pj, ir2);
#pragma unroll
                                    for (int e = 0; e < 6; ++e) f[e].add(e6[e]);
                                    if (SYM) {
                                        strain(pi, -ir2);
#pragma unroll
                                        for (int e = 0; e < 6; ++e) {
                                            Acc<R> a = ws.rev[e][jl];
                                            a.add(e6[e]);
                                            ws.rev[e][jl] = a;
                                        }
                                    }
                                }
                            }
                            if (SYM) __syncwarp();
                        }
                        // the lanes that share a target (fixed order), then the block's sums
                        for (int o = tg; o < 32; o <<= 1)
#pragma unroll
                            for (int e = 0; e < 6; ++e) f[e].add(f[e].shfl_xor(o));
                        if (vi && tj == 0)
#pragma unroll
                            for (int e = 0; e < 6; ++e) {
                                Acc<R> a = ws.fwd[e][c0 + ti];
                                a.add(f[e]);
                                ws.fwd[e][c0 + ti] = a;
                            }
                        c0 += tg;
                    }
                    if (SYM) {
                        __syncwarp();
                        for (int k = lane; k < ns; k += 32) {
                            double *row = tr.rows + (rbase + ws.pos[k]) * 6;
                            for (int e = 0; e < 6; ++e) {
                                const double v = ws.rev[e][k].value();
                                row[e] = add ? row[e] + v : v;
                            }
                        }
                    }
                }
                __syncwarp();
                for (int k = lane; k < nb_t; k += 32) {
                    double *row = tr.rows + (fbase + (tb - tA0) + k) * 6;
                    for (int e = 0; e < 6; ++e) row[e] = ws.fwd[e][k].value();
                }
                add = true;
            }
        }
    }
}

// ---------------------------------------------------------------- combine
// Far field (L2P) plus the stress of the summed strain rows, LANES threads per point.  Eight lanes
// share a point's 3 p basis values, take every eighth (y, z) row of the p^3 local values and every
// eighth of its rows, and are added by a fixed tree: in the smallest calls one thread's chain is
// the time.  One thread per point where there are enough points to fill the GPU: the 32 points of a
// warp then mostly read the same local values.  One lane / eight, p = 5, us: 628 points 50 / 24, 8,000
// 214 / 68, 24,000 87 / 81, 48,000 114 / 118, 64,000 98 / 138, 200,000 200 / 409, 4M 2,036 / 6,962; FP64
// 628 points 103 / 34, 24,000 141 / 140, 48,000 234 / 232, 64,000 218 / 295.
constexpr int64_t kCombinePoints = 40000;  // up to this many points: eight lanes

template <int LANES, typename SR>
__device__ __forceinline__ void l2p(int p, const NodeTab<SR> &nt, SR *basis, int g, const double c0[3], double ih,
                                    const double *x, const SR *__restrict__ Sl, double out[6]) {
    for (int i = g; i < 3 * p; i += LANES) {
        const int d = i / p;
        basis[i] = lagrange_at<SR>(nt, p, i - d * p, SR((x[d] - (d == 0 ? c0[0] : d == 1 ? c0[1] : c0[2])) * ih));
    }
    __syncwarp();
    SR acc[6] = {SR(0), SR(0), SR(0), SR(0), SR(0), SR(0)};
    for (int r = g; r < p * p; r += LANES) {
        const SR wyz = basis[p + r % p] * basis[2 * p + r / p];
        SR v[6] = {SR(0), SR(0), SR(0), SR(0), SR(0), SR(0)};
        for (int lx = 0; lx < p; ++lx) {
            const SR w = basis[lx];
            const SR *s6 = Sl + (r * p + lx) * 6;  // 24 or 48 bytes, read in pairs
            if constexpr (sizeof(SR) == 4) {
                const float2 *q = reinterpret_cast<const float2 *>(s6);
                const float2 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2);
                v[0] += w * a.x, v[1] += w * a.y, v[2] += w * b.x, v[3] += w * b.y, v[4] += w * c.x, v[5] += w * c.y;
            } else {
                const double2 *q = reinterpret_cast<const double2 *>(s6);
                const double2 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2);
                v[0] += w * a.x, v[1] += w * a.y, v[2] += w * b.x, v[3] += w * b.y, v[4] += w * c.x, v[5] += w * c.y;
            }
        }
        for (int e = 0; e < 6; ++e) acc[e] += wyz * v[e];
    }
    for (int e = 0; e < 6; ++e) {
        for (int o = LANES / 2; o > 0; o >>= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
        out[e] = double(acc[e]);
    }
}

template <bool SYM, int LANES, typename SR>
__global__ void __launch_bounds__(256) k_near_combine(int p, const __grid_constant__ NodeTab<SR> nt,
                                                      const __grid_constant__ NearTree tr,
                                                      const double *__restrict__ C, const int *__restrict__ tleaf,
                                                      const double *__restrict__ xt, const SR *__restrict__ S,
                                                      double *__restrict__ sig, const int *__restrict__ pfine,
                                                      const SR *__restrict__ S7) {
    __shared__ SR s_basis[256 / LANES][3 * GB_MAXP + 1];  // (+ 1: one thread per point would meet one bank)
    const int64_t t0 = (blockIdx.x * int64_t(256) + threadIdx.x) / LANES;
    const int g = threadIdx.x % LANES;
    const bool valid = t0 < tr.n_t;
    const int64_t t = valid ? t0 : tr.n_t - 1;  // surplus lanes repeat the last point
    const int nlv = 1 << (tr.L - 1);
    const int64_t leaf = tleaf[t];
    int cx, cy, cz;
    cell_xyz3(leaf, nlv, cx, cy, cz);
    double far[6];
    const int f = pfine ? pfine[t] : -1;
    {
        const int P3 = p * p * p;
        double h = tr.box->H / nlv, ih = double(nlv) / tr.box->H;
        double c0[3] = {tr.box->origin[0] + cx * h, tr.box->origin[1] + cy * h, tr.box->origin[2] + cz * h};
        const SR *Sl = S + (cell_base_d(tr.L - 1) + leaf) * int64_t(P3) * 6;
        if (f >= 0) {
            // a point of a split leaf: its child's local values and cell (adaptive tree)
            h *= 0.5;
            ih *= 2.0;
            c0[0] += (f & 1) * h;
            c0[1] += ((f >> 1) & 1) * h;
            c0[2] += ((f >> 2) & 1) * h;
            Sl = S7 + int64_t(f) * P3 * 6;
        }
        l2p<LANES, SR>(p, nt, s_basis[threadIdx.x / LANES], g, c0, ih, xt + 3 * t, Sl, far);
    }
    double e6[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    auto add_row = [&](long long r) {
        const double2 *q = reinterpret_cast<const double2 *>(tr.rows + r * 6);
        const double2 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2);
        e6[0] += a.x, e6[1] += a.y, e6[2] += b.x, e6[3] += b.y, e6[4] += c.x, e6[5] += c.y;
    };
    {
        const NearPlan pl = tr.plan[leaf];
        const int nt_l = tr.tstart[leaf + 1] - tr.tstart[leaf], k = int(t - tr.tstart[leaf]);
        for (int b = g; b < pl.cb; b += LANES) add_row(pl.base + (long long)b * nt_l + k);
    }
    if (SYM) {
        const int rank = int(t - tr.sstart[leaf]);
        for (int d = g; d < 14; d += LANES) {
            // the leaf that holds this one in direction d of its list
            const int64_t A = neighbour(cx, cy, cz, 13 - d, nlv);
            if (A < 0) continue;
            const int nt_a = tr.tstart[A + 1] - tr.tstart[A];
            if (nt_a == 0) continue;
            const NearPlan pl = tr.plan[A];
            const long long r = pl.base + (long long)pl.cb * nt_a + tr.lp[14 * A + d] + rank;
            const bool splitA = tr.ref_start && tr.ref_start[A + 1] > tr.ref_start[A];
            // a plain leaf's tile meets its own leaf from the tile's first target on; a split
            // leaf's rows were zeroed first
            const int ca = splitA || d > 0 ? pl.ca : min(pl.ca, rank / pl.ta + 1);
            const int nb = 13 + d, ox = nb % 3 - 1, oy = (nb / 3) % 3 - 1, oz = nb / 9 - 1;
            const bool skip = splitA && pl.ca == 8 && f >= 0 && d > 0;  // one child per tile: adjacent ones only
            for (int a = 0; a < ca; ++a) {
                if (skip && (abs(2 * ox + (f & 1) - (a & 1)) > 1 || abs(2 * oy + ((f >> 1) & 1) - ((a >> 1) & 1)) > 1 ||
                             abs(2 * oz + ((f >> 2) & 1) - (a >> 2)) > 1))
                    continue;
                add_row(r + (long long)a * pl.ns);
            }
        }
    }
    __syncwarp();
    for (int e = 0; e < 6; ++e)
        for (int o = LANES / 2; o > 0; o >>= 1) e6[e] += __shfl_xor_sync(0xffffffffu, e6[e], o);
    if (!valid) return;
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        if (LANES > 1 && g != m) continue;
        double s = 0.0;
        for (int e = 0; e < 6; ++e) s += C[6 * m + e] * e6[e];
        sig[6 * t + m] = s + far[m];
    }
}

}  // namespace

// ---------------------------------------------------------------- host side
float mlp_poly_m2();  // mlp.cu

static bool near_learned(const gbfmm_ctx *ctx) {
    return ctx->mat.mode == GBFMM_H_MLP && ctx->opt.precision != GBFMM_FP64;
}

// The pair kernel's unit of the moduli: the power of two at their largest entry.  Its rules form
// det(zz)^-2, the sixth power of a modulus, and FP32 holds that for moduli from 4e-7 to 2e6 only
// (with moduli in Pa every term with it vanishes and h is finite and wrong); in this unit the moduli
// are of order one whatever the caller's, and no rounding changes.
static double near_unit(const DevMaterial &m) {
    double v = 0.0;
    for (int i = 0; i < 6; ++i) v = std::max(v, m.V[7 * i]);
    return std::ldexp(1.0, std::ilogb(v));
}

// Burgers vectors carry the factor of h that its sums leave out: 1 / (4 pi Q) of the unit-circle
// rule, the isotropic rule's factor (an inverse modulus, in the kernel's unit)
static double near_factor(const DevMaterial &m) {
    return m.mode == GBFMM_H_ISO ? m.hc * near_unit(m) : 1.0 / (4.0 * M_PI * m.Q);
}

// constants of a medium in the kernel's unit; the strain of a pair has none, so nothing is scaled
// back but the network's h, whose unit is the caller's (NearLearned)
template <typename R>
static NearMedium<R> near_medium(const DevMaterial &m) {
    NearMedium<R> n{};
    n.Q = m.Q;
    n.np = (m.Q - 1) / 2;
    const double iu = 1.0 / near_unit(m), c12 = iu * m.c12, c44 = iu * m.c44, D = iu * m.cd;
    const double cp = c12 + c44, ydiag = D + 2.0 * c44;
    n.k1 = R(iu * (m.V[1] * (1.0 - m.ha) + 2.0 * m.V[21]));
    n.k3 = R(iu * m.V[21] * (1.0 - m.ha));
    n.k6 = R(iu * 6.0 * m.V[21]);
    // adj_ii = al - be z_i^2 + ga z_j^2 z_k^2, adj_ij = mcp z_i z_j (c44 + D z_k^2)
    const double al = c44 * (c44 + D + cp), be = c44 * (D + cp), ga = D * (D + 2.0 * cp), mcp = -cp;
    const double d0 = c44 * c44 * (c44 + D + cp), d1 = c44 * D * (D + 2.0 * cp);
    n.d1 = R(d1);
    n.d2 = R(D * D * (D + 3.0 * cp));
    n.e0 = R(d0 + 0.5 * d1);
    // sum_p h_cpp = (al + mcp c44) lin_c - (be + mcp c44) c1_c + (ga + 2 mcp D) x2_c
    const double t0 = c12 * (al + mcp * c44), t1 = -c12 * (be + mcp * c44), t2 = c12 * (ga + 2.0 * mcp * D);
    n.rc[0] = R(t0 + ydiag * al), n.rc[1] = R(t1 - ydiag * be), n.rc[2] = R(t2 + ydiag * ga);
    n.rn[0] = R(t0), n.rn[1] = R(t1), n.rn[2] = R(t2 + ydiag * mcp * D), n.rn[3] = R(ydiag * mcp * c44);
    n.re[0] = R(c44 * mcp * (2.0 * c44 + D)), n.re[1] = R(-c44 * mcp * D);
    n.rs[0] = R(c44 * al), n.rs[1] = R(c44 * mcp * D), n.rs[2] = R(c44 * (mcp * c44 - be)), n.rs[3] = R(c44 * ga);
    n.y12 = R(c12);
    n.ydiag = R(ydiag);
    n.y44 = R(c44);
    static const int PV[6] = {0, 1, 2, 1, 0, 0}, PP[6] = {0, 1, 2, 2, 2, 1};
    auto C = [&m, iu](int i, int j, int k, int l) { return iu * m.C[((i * 3 + j) * 3 + k) * 3 + l]; };
    for (int a = 0; a < 6; ++a)
        for (int x = 0; x < 6; ++x) {
            n.C[6 * a + x] = R(iu * m.V[6 * a + x]);
            // (zz)_jk = z_i C_ijkl z_l
            const int j = PV[a], k = PP[a], i = PV[x], l = PP[x];
            n.Z[6 * a + x] = R(C(i, j, k, l) + (i != l ? C(l, j, k, i) : 0.0));
            n.Z2[6 * a + x] = make_float2(float(n.Z[6 * a + x]), float(n.Z[6 * a + x]));
        }
    return n;
}

// rows and items that a pass may use: functions of the network's size alone (near_plan).  An
// undivided plan needs 15 rows a point (forward one, 14 leaves hold it in their lists) and one
// item per occupied leaf; the rest is room to divide the work.
static int64_t rows_sym(int64_t N) { return 32 * N + std::min<int64_t>(int64_t(1) << 20, N * N / 8 + 64); }
static int64_t rows_free(int64_t n) { return 4 * n + (int64_t(1) << 18); }
static int64_t items_cap(int64_t n, int64_t nl) { return n / 2 + std::min(n, nl) + 65536; }

// buffers of the pair kernel for n targets (records of the targets only when they are free)
static int pairs_alloc(gbfmm_ctx *ctx, int64_t n, bool free_targets) {
    NearWork &W = ctx->ws().nw;
    const bool f32 = ctx->opt.precision != GBFMM_FP64;
    const int64_t nl = ctx->n_leaves, rows = free_targets ? rows_free(n) : rows_sym(n), it = items_cap(n, nl);
    const size_t point = f32 ? 4 * sizeof(float4) : 5 * sizeof(double2), target = 2 * sizeof(float4);
    if (int rc = grow_dev(ctx, W.rec_cap, ctx->N, {{&W.rec, size_t(ctx->N) * point}}, "near-field points")) return rc;
    if (free_targets)
        if (int rc = grow_dev(ctx, W.trec_cap, n, {{&W.trec, size_t(n) * target}}, "near-field targets")) return rc;
    if (int rc = grow_dev(ctx, W.plan_cap, nl,
                          {{(void **)&W.plan, size_t(nl) * sizeof(NearPlan)}, {(void **)&W.lp, size_t(nl) * 27 * sizeof(int)}},
                          "near-field plan"))
        return rc;
    if (int rc = grow_dev(ctx, W.item_cap, it, {{(void **)&W.pitems, size_t(it) * sizeof(NearItem)}}, "near-field items"))
        return rc;
    if (int rc = grow_dev(ctx, W.row_cap, rows, {{(void **)&W.rows, size_t(rows) * 6 * sizeof(double)}}, "near-field sums"))
        return rc;
    if (!W.pcnt) CK(cudaMalloc(&W.pcnt, kCnt * sizeof(unsigned long long)));
    return GBFMM_OK;
}

int near_alloc(gbfmm_ctx *ctx) { return pairs_alloc(ctx, ctx->N, false); }

// the records of the source points
int near_prepare(gbfmm_ctx *ctx) {
    const int64_t N = ctx->N;
    ++ctx->launches;
    GaussWeights gw{};
    gw.n = ctx->opt.n_gauss;
    for (int i = 0; i < gw.n; ++i) gw.w[i] = ctx->gauss_w[i];
    const double fac = near_factor(ctx->mat);
    if (ctx->opt.precision == GBFMM_FP64)
        k_near_records<double><<<nblk(N, 256), 256, 0, ctx->stream>>>(N, ctx->L, ctx->d_box, ctx->d_y, ctx->d_perm,
                                                                       ctx->d_pleaf, ctx->d_segv, gw, fac, ctx->ws().nw.rec);
    else
        k_near_records<float><<<nblk(N, 256), 256, 0, ctx->stream>>>(N, ctx->L, ctx->d_box, ctx->d_y, ctx->d_perm,
                                                                      ctx->d_pleaf, ctx->d_segv, gw, fac, ctx->ws().nw.rec);
    CK(cudaGetLastError());
    return GBFMM_OK;
}

template <typename R, int HM, bool SYM, bool LEARN>
static int launch_pairs(gbfmm_ctx *ctx, const NearTree &tr, const NearMedium<R> &md, const NearLearned &ln) {
    size_t table = 0;
    if (HM == HM_POINTS) table = md.Q <= kPointMax ? size_t((md.Q + 1) / 2) * sizeof(float4) : 0;
    else if (HM != HM_ISO) table = md.np <= kMomMax ? size_t(md.np) * kMomRow * sizeof(R) : 0;
    const size_t smem = near_warps<R>() * sizeof(WarpShared<R, SYM, LEARN>) + table;
    auto kern = k_near_pairs<R, HM, SYM, LEARN>;
    CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
    ++ctx->launches;
    kern<<<unsigned(ctx->sm_count * near_blocks<R>()), near_warps<R>() * 32, smem, ctx->stream>>>(tr, md, ln);
    CK(cudaGetLastError());
    return GBFMM_OK;
}

template <bool SYM, typename SR>
static int launch_combine(gbfmm_ctx *ctx, const NearTree &tr, const int *tleaf, const double *xt, const SR *S, double *sig,
                          const int *pfine, const SR *S7) {
    const NodeTab<SR> nt = make_nodes<SR>(ctx->opt.p, ctx->opt.nodes);
    ++ctx->launches;
    if (tr.n_t <= kCombinePoints)
        k_near_combine<SYM, 8, SR><<<nblk(tr.n_t * 8, 256), 256, 0, ctx->stream>>>(ctx->opt.p, nt, tr, ctx->d_mat->V, tleaf,
                                                                                    xt, S, sig, pfine, S7);
    else
        k_near_combine<SYM, 1, SR><<<nblk(tr.n_t, 256), 256, 0, ctx->stream>>>(ctx->opt.p, nt, tr, ctx->d_mat->V, tleaf, xt,
                                                                               S, sig, pfine, S7);
    CK(cudaGetLastError());
    return GBFMM_OK;
}

template <typename R, bool SYM>
static int run_pairs(gbfmm_ctx *ctx, const int *tstart, const double *xt, int64_t n_t, const int *tleaf, double *sig) {
    if (int rc = pairs_alloc(ctx, n_t, !SYM)) return rc;
    NearWork &W = ctx->ws().nw;
    cudaStream_t st = ctx->stream;
    const int64_t nl = ctx->n_leaves;
    // adaptive tree (nodal forces): split leaves, their children's ranges and local values
    const bool fine = SYM && ctx->rf.on;
    NearTree tr{};
    tr.L = ctx->L;
    tr.N = ctx->N;
    tr.n_t = n_t;
    tr.box = ctx->d_box;
    tr.tstart = tstart;
    tr.sstart = ctx->d_leaf_start;
    tr.ref_start = fine ? ctx->rf.ref_start : nullptr;
    tr.child_start = fine ? ctx->rf.child_start : nullptr;
    tr.trec = SYM ? W.rec : W.trec;
    tr.srec = W.rec;
    tr.plan = static_cast<const NearPlan *>(W.plan);
    tr.lp = W.lp;
    tr.items = static_cast<const NearItem *>(W.pitems);
    tr.cnt = W.pcnt;
    tr.rows = W.rows;
    CK(cudaMemsetAsync(W.pcnt, 0, kCnt * sizeof(unsigned long long), st));
    if (!SYM) {
        ++ctx->launches;
        k_near_targets<R><<<nblk(n_t, 256), 256, 0, st>>>(n_t, ctx->L, ctx->d_box, xt, tleaf, W.trec);
    }
    ctx->launches += 2;
    k_near_totals<SYM><<<nblk(nl, 256), 256, 0, st>>>(nl, ctx->L, tstart, ctx->d_leaf_start, tr.ref_start, W.pcnt);
    k_near_plan<SYM><<<nblk(nl, 256), 256, 0, st>>>(nl, ctx->L, ctx->sm_count * near_blocks<R>() * near_warps<R>(),
                                                    SYM ? rows_sym(n_t) : rows_free(n_t), items_cap(n_t, nl), tstart,
                                                    ctx->d_leaf_start, tr.ref_start, W.pcnt,
                                                    static_cast<NearPlan *>(W.plan), W.lp,
                                                    static_cast<NearItem *>(W.pitems));
    CK(cudaGetLastError());
    const NearMedium<R> md = near_medium<R>(ctx->mat);
    NearLearned ln{};
    // The cubic form's FP32 rounding grows for Zener ratios below one (RMS of K, pointwise rule
    // from C / cubic moments: A = 3.2, 2.1 / 1.6e-7; A = 0.48, 0.9 / 1.2e-7; A = 0.17, 0.8 /
    // 2.6e-7): such media take the general rule.
    const bool cubic = ctx->mat.cubic && (sizeof(R) == 8 || ctx->mat.cd <= 1e-6 * ctx->mat.c44);
    int rc = GBFMM_OK;
    if (ctx->mat.mode == GBFMM_H_ISO) {
        rc = launch_pairs<R, HM_ISO, SYM, false>(ctx, tr, md, ln);
    } else if (near_learned(ctx)) {
        if constexpr (sizeof(R) == 4) {
            // pairs closer than near_fp64 segment lengths take the plain rule whatever mlp_min_dist is
            const double rmin = std::max(ctx->opt.mlp_min_dist > 0.0 ? ctx->opt.mlp_min_dist : 8.0, ctx->opt.near_fp64);
            ln.binmask = ctx->mlp.d_binmask;
            ln.poly = reinterpret_cast<const float4 *>(ctx->mlp.poly);
            ln.rmin2 = float(rmin * rmin);
            ln.m2 = mlp_poly_m2();
            ln.fac = float(near_unit(ctx->mat) / near_factor(ctx->mat));
            rc = cubic ? launch_pairs<R, HM_CUBIC, SYM, true>(ctx, tr, md, ln)
                       : launch_pairs<R, HM_GENERAL, SYM, true>(ctx, tr, md, ln);
        }
    } else if (cubic) {
        rc = launch_pairs<R, HM_CUBIC, SYM, false>(ctx, tr, md, ln);
    } else {
        if constexpr (sizeof(R) == 4)
            rc = launch_pairs<R, HM_POINTS, SYM, false>(ctx, tr, md, ln);
        else
            rc = launch_pairs<R, HM_GENERAL, SYM, false>(ctx, tr, md, ln);
    }
    if (rc) return rc;
    const int *pfine = fine ? ctx->rf.pfine : nullptr;
    if (ctx->opt.precision == GBFMM_MIXED) return launch_combine<SYM, float>(ctx, tr, tleaf, xt, ctx->d_Sf, sig, pfine, ctx->rf.S7);
    return launch_combine<SYM, double>(ctx, tr, tleaf, xt, ctx->d_S, sig, nullptr, nullptr);  // FP64 local values
}

// Near field and L2P of a pass, into sig (sorted order).  free_targets: the n_t sorted free
// points, else the Gauss points themselves.
int near_run(gbfmm_ctx *ctx, bool free_targets, int64_t n_t, double *sig) {
    const int *tstart = free_targets ? ctx->d_t_start : ctx->d_leaf_start;
    const double *xt = free_targets ? ctx->d_t_x : ctx->d_y;
    if (!free_targets) n_t = ctx->N;
    if (near_learned(ctx) && (!ctx->mlp.trained || !ctx->mlp.d_binmask))
        return set_err(ctx, GBFMM_ERR_INVALID_ARG, "GBFMM_H_MLP: train (or set) and calibrate the network first");
    const int *tleaf = free_targets ? ctx->d_t_leaf : ctx->d_pleaf;
    if (ctx->opt.precision == GBFMM_FP64)
        return free_targets ? run_pairs<double, false>(ctx, tstart, xt, n_t, tleaf, sig)
                            : run_pairs<double, true>(ctx, tstart, xt, n_t, tleaf, sig);
    return free_targets ? run_pairs<float, false>(ctx, tstart, xt, n_t, tleaf, sig)
                        : run_pairs<float, true>(ctx, tstart, xt, n_t, tleaf, sig);
}
