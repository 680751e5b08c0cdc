// libtula_ags: the AGS optimizer step (Tula, arXiv 2603.18112) for sm_103a.
//
// Per step, three kernels on the caller's stream, chained by programmatic
// dependent launch so that each one's launch and prologue overlap the tail of
// the one before:
//
//   k_reduce   (pass 1)  K-way replica mean (Eq. 1c) written over replica 0; each
//                        tile's sums of |gbar|^2, |g_0|^2 [, |w|^2] are added
//                        exactly into per-tensor accumulators (and |gbar|^2 into
//                        the step's |G|^2 accumulator) by L2 atomics.
//   k_update   (pass 2)  the branch of Algorithm 1 from |G|^2 (Eq. 5), then
//                        d = c gbar + wd w; m = mu m + d; w = w - lr m (Eq. 7b with
//                        the wrapped SGD); |w|^2 per tile for the statistics.
//   k_finish             per tensor, the norms rounded from its accumulators, its
//                        statistics and, when asked, the refreshed gradscale
//                        (UpdateGradScale, Algorithm 1); one more warp writes the
//                        step record (|G|^2, Delta, the branch).
//
// A LARS step has k_lars between the passes: its coefficients are ratios of this
// step's norms.
//
// The streaming passes: each tensor is cut into tiles of T elements (T fixed
// per pass by how many tensors it streams, so that one tile of every stream
// fills one shared-memory stage: 36 KB in pass 1, 24 KB in pass 2).  One
// persistent CTA per SM, whose warps each stream tiles through a stage of their
// own with TMA bulk copies (cp.async.bulk ... mbarrier::complete_tx), one copy per
// stream issued by one lane each, and claim tiles from a global counter (SMs
// stream at unequal rates).  Tile partials are fp32 sums within a tile
// (float-float pairs per lane in the precise mode for norms that feed a
// coefficient, triples for misaligned tensors), range-checked per tile, and leave
// the tile only as exact integer additions into the accumulators.
//
// Every mbarrier wait is bounded; a wait that runs out sets an error word in
// the workspace (tula_ags_workspace_error) and the CTA drains its copies in
// flight and returns.  The streaming kernels are HBM-bound (a few flops per
// 20-70 bytes); nothing here is a contraction, so no tensor cores.  The tile
// table, pointers and sizes travel in the kernel parameter block
// (__grid_constant__, up to ~31 KB per launch): no host-to-device copy,
// allocation or host sync is ever needed.  Integer addition does not depend on
// the order in which tiles land, so results are bitwise reproducible and
// independent of the grid and of which CTA took which tile.
#include "tula_ags.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <type_traits>
#include <utility>
#include <vector>

namespace {

// Tensors off a 16-byte boundary: a stream's tile starts up to 12 bytes into its part of the
// stage, which is kShiftBytes longer; the stages have room for that.
constexpr int kShiftBytes = 16;
// The stages of a streaming kernel's CTA: one per warp, each holding one tile of every stream.  A
// warp refills its own stage (see "Streaming warps" below), so a CTA is nothing but warps that
// stream for themselves.
template <int StageKB, int Warps, int Pad>
struct Ring {
    static constexpr int kTileBytes = StageKB * 1024;  // one aligned tile of every stream
    static constexpr int kStageBytes = kTileBytes + Pad;
    static constexpr int kWarps = Warps;
    static constexpr int kThreads = 32 * Warps;
    static constexpr int kSmemBytes = Warps * (kStageBytes + 8);
    static_assert(kSmemBytes <= 227 * 1024 && kStageBytes % 16 == 0, "one CTA per SM");
    // Elements per tile when `streams` tensors share one stage (multiple of 128).
    __host__ __device__ static constexpr int tile_elems(int streams) {
        return (kTileBytes / (4 * streams)) / 128 * 128;
    }
    // Whether the shifted tiles (see issue_edge_tile) of `streams` tensors fit, too.
    static constexpr bool shifted_fits(int streams) {
        return streams * (4 * tile_elems(streams) + kShiftBytes) <= kStageBytes;
    }
};
template <typename R>
constexpr bool shifted_fits_up_to(int streams) {
    for (int ns = 1; ns <= streams; ++ns)
        if (!R::shifted_fits(ns)) return false;
    return true;
}
// Pass 1 streams K (+1, +2) tensors through 36 KB stages.
// SH: with room for shifted tiles, in the kernels of launches that have any.
template <bool SH>
using Ring1 = Ring<36, 6, SH ? 256 : 0>;
static_assert(shifted_fits_up_to<Ring1<true>>(TULA_MAX_K), "shifted tiles fit a stage");
// Pass 1 when it also reads w (LARS, tula_layer_stats): five 45 KB stages.  No more padding than
// the stream count needs: beside the CTA, an SM must have the 1 KB of shared memory left that any
// other CTA takes, or the small kernels around it cannot be resident while it runs (a ResNet-50
// LARS step with 256 bytes more a stage took 251 us instead of 236).
template <int KT, bool SH>
using Ring1W = Ring<45, 5, !SH ? 0 : KT == 0 ? 240 : (KT + 1) * kShiftBytes>;
static_assert(shifted_fits_up_to<Ring1W<0, true>>(TULA_MAX_K + 1) &&
                  Ring1W<1, true>::shifted_fits(2) && Ring1W<2, true>::shifted_fits(3) &&
                  Ring1W<4, true>::shifted_fits(5) && Ring1W<8, true>::shifted_fits(9) &&
                  Ring1W<16, true>::shifted_fits(17),
              "shifted tiles fit a stage");
template <int KT, bool RW, bool SH>
using Ring1Of = std::conditional_t<RW, Ring1W<KT, SH>, Ring1<SH>>;
// Pass 2: eight 24 KB stages.
template <bool SH>
using Ring2 = Ring<24, 8, SH ? 256 : 0>;
static_assert(shifted_fits_up_to<Ring2<true>>(4), "shifted tiles fit a stage");
constexpr int kPend = 4;                // tiles whose warp reductions run together
constexpr int kFinWarps = 4;            // k_finish: one warp per tensor, 4 per CTA
constexpr int kParamBudget = 31 * 1024; // kernel parameter bytes per launch (limit 32764)
constexpr int kAcc = 3;                 // partial sums per pass-1 tile: |gbar|^2, |g_0|^2, |w|^2
constexpr int kPrecCols = 1;            // float4 columns per step of the precise path's tile loop
constexpr int kSpare = 32;              // unused bytes per tensor in the workspace's layout
constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kSpinLimit = 1u << 19;  // bound on every mbarrier wait (~2 s on GB300)

enum Mode { kModeStep = 0, kModeStats = 1, kModeScale = 2 };


// ----------------------------------------------------------------------------
// Launch tables (kernel parameters)
// ----------------------------------------------------------------------------

// One launch's tensors: sizes, first tiles and pointers, in a parameter block of Bytes bytes.  The
// arrays lie one after the other in `raw`, `np` pointers per tensor: a pointer is its role's base
// plus a 32-bit offset in fp32 elements (a 16 GB window), with 16 more bits when some role's
// tensors lie farther apart (`wide`).  6 bytes per tensor and 4 per pointer put 4096 tensors with
// K = 16 through 10 launches of pass 1 (whole pointers and sizes: 21), and leave less of the block
// to miss the constant cache on.
constexpr int kHints = 160;
constexpr int kMaxRoles = TULA_MAX_K + 1;
struct TableHead {
    int n;        // tensors in this launch
    int t0;       // global index of its first tensor
    int nc;       // tiles in this launch
    int chunk;    // elements per tile
    int seq;      // 0, 1, ... in the order of the pass's launches
    int shifted;  // 1: some tensor has a stream off a 16-byte boundary
    int np, wide;
    int o_last, o_lo, o_hi;  // byte offsets in raw
    int hint_shift;
    unsigned long long base[kMaxRoles];
    unsigned short hint[kHints + 2];  // tensor of tile min(i << hint_shift, nc - 1)
};
template <int Bytes>
struct Table : TableHead {
    static constexpr int kRaw = Bytes - (int)sizeof(TableHead);
    alignas(8) unsigned char raw[kRaw];  // cstart[n + 1], last[n], lo[n][np] [, hi[n][np]]
    static constexpr int bytes_for(int n, int np, bool wide) {
        return 4 * (n + 1) + (2 * n + 3) / 4 * 4 + 4 * n * np + (wide ? 2 * n * np : 0);
    }
    // First tile of tensor t (t = n: nc).
    __host__ __device__ int cstart(int t) const { return reinterpret_cast<const int *>(raw)[t]; }
    // Elements of its last tile.
    __host__ __device__ int last(int t) const {
        return reinterpret_cast<const unsigned short *>(raw + o_last)[t];
    }
    __host__ __device__ long long numel(int t) const {
        return (long long)(cstart(t + 1) - cstart(t) - 1) * chunk + last(t);
    }
    __host__ __device__ float *ptr(int t, int role) const { return ptr(t, role, base[role]); }
    __host__ __device__ float *ptr(int t, int role, unsigned long long base_of_role) const {
        const int i = t * np + role;
        unsigned long long e = reinterpret_cast<const unsigned *>(raw + o_lo)[i];
        if (wide)
            e |= (unsigned long long)reinterpret_cast<const unsigned short *>(raw + o_hi)[i] << 32;
        return reinterpret_cast<float *>(base_of_role + 4ull * e);
    }
};
// A tensor's pointers by role.
template <typename Tab>
struct Row {
    const Tab &tab;
    int t;
    __host__ __device__ float *operator[](int role) const { return tab.ptr(t, role); }
};
// A launch of few tensors passes a smaller block: three launches with 31 KB each cost the host
// 8.0 us, with 8 KB 5.6 us, and a call that waits for them 17.0 and 13.2 us.
template <bool Small>
using TableOf = Table<Small ? 8 * 1024 : kParamBudget>;
static_assert(sizeof(TableOf<true>) == 8 * 1024 && sizeof(TableOf<false>) == kParamBudget, "as sized");

struct Scalars {
    int K, rule, force, refresh, mode, n_total, read_w;
    int evict_first, early_w, keep_w;  // evict_first: TMA loads ask L2 to drop their lines first,
                                       // keep_w: but not pass 1's of w; early_w: the update
                                       // follows this call's pass 1
    float delta, eps, s_max, static_s, lars_trust, lr, mu, wd, invK, Kf;
    float *scale;
    double *state;
    double *stats;
    unsigned *err;             // [0]: bounded waits that ran out (sticky until read)
    unsigned long long *acc1;  // [tensor][kAcc][kTCopies][kAccWords]: |gbar|^2, |g_0|^2, |w|^2
    unsigned long long *gacc;  // [kGCopies][kAccWords]: |G|^2 = every tensor's |gbar|^2
    unsigned long long *acc2;  // [tensor][kTCopies][kAccWords]: |w|^2, pass 2
    float *cand;               // [tensor]: c_p of a LARS step
    unsigned *tiles;           // [2 * (seq & 1) + pass]: claims made
    unsigned claim_base;       // of them, by the pass's launches before this one on this counter
    const unsigned long long *g2ext;  // a sharded step's |G|^2: the ranks' shares summed (or NULL)
};

// ----------------------------------------------------------------------------
// Device helpers: memory, arithmetic
// ----------------------------------------------------------------------------

__device__ __forceinline__ void st_stream(float *p, float4 v) {
    __stcs(reinterpret_cast<float4 *>(p), v);
}
__device__ __forceinline__ void st_keep(float *p, float4 v) {
    *reinterpret_cast<float4 *>(p) = v;
}
// 16-byte load from shared memory (a shared-window address).
__device__ __forceinline__ float4 lds4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr));
    return v;
}

__device__ __forceinline__ float lds1(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

// fp32 sum of squares into a running fp32 partial, one FFMA per term
__device__ __forceinline__ float sq4(float acc, float4 v) {
    acc = __fmaf_rn(v.x, v.x, acc);
    acc = __fmaf_rn(v.y, v.y, acc);
    acc = __fmaf_rn(v.z, v.z, acc);
    acc = __fmaf_rn(v.w, v.w, acc);
    return acc;
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z),
                       __fadd_rn(a.w, b.w));
}

// Eq. 1c: divide the k-ascending sum by K (exact reciprocal when K is a power of 2).  K by value,
// for the same reason as Sgd.
struct MeanK {
    float invK, Kf;
};
__device__ __forceinline__ MeanK mean_k(const Scalars &sc) { return {sc.invK, sc.Kf}; }
template <int KT>
__device__ __forceinline__ float mean1(float s, const MeanK &sc) {
    static_assert((KT & (KT - 1)) == 0, "a power of two, or 0: known at run time");
    return KT > 0 ? __fmul_rn(s, 1.0f / (float)(KT > 0 ? KT : 1)) : __fdiv_rn(s, sc.Kf);
}
// s / K for a K known only at run time, correctly rounded (Markstein, IBM J. Res. Dev. 34, 1990):
// with y = fl(1 / K) and q = fl(s y), the remainder r = s - K q is exact in one fused operation and
// fl(q + r y) is the quotient.  It scales with powers of two, so that every significand of one
// binade decides it; the tests run them all for every K.  Only for |s| in [2^-90, inf): below, the
// remainder may leave fp32's range.  A ResNet-50 step with K = 6 spent 29 of 213 us on divisions.
__device__ __forceinline__ bool mean_in_range(float s) {
    return __float_as_uint(fabsf(s)) - __float_as_uint(0x1p-90f) <
           0x7f800000u - __float_as_uint(0x1p-90f);
}
__device__ __forceinline__ float mean_fast(float s, const MeanK &sc) {
    const float q = __fmul_rn(s, sc.invK);
    return __fmaf_rn(__fmaf_rn(-sc.Kf, q, s), sc.invK, q);
}
template <int KT>
__device__ __forceinline__ float4 mean4(float4 s, const MeanK &sc) {
    if (KT == 0 && mean_in_range(s.x) && mean_in_range(s.y) && mean_in_range(s.z) &&
        mean_in_range(s.w))
        return make_float4(mean_fast(s.x, sc), mean_fast(s.y, sc), mean_fast(s.z, sc),
                           mean_fast(s.w, sc));
    return make_float4(mean1<KT>(s.x, sc), mean1<KT>(s.y, sc), mean1<KT>(s.z, sc),
                       mean1<KT>(s.w, sc));
}


// Warp reduce-scatter of R values per lane (R a power of two, <= 32): each of log2(R) halving
// steps sends half of a lane's values to the lane `off` away and keeps the sums of the other
// half; the remaining steps add the one value left across the lanes still sharing it.
// Afterwards every lane holds the warp total of value `index` (bits of the lane id reversed):
// with R = 16, lanes 2i and 2i + 1 hold the same one.  16 + 1 shuffles for R = 16 instead of
// the 5 R of a tree per value, so the owners of R sums can store them at once.  The order of
// the additions is fixed (results do not depend on timing), and the two lanes that end with
// the same sum add the same two terms.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
template <int R, typename T>
__device__ __forceinline__ T warp_reduce_scatter(T (&v)[R], int &index) {
    static_assert(R >= 1 && R <= 32 && (R & (R - 1)) == 0, "R: a power of two <= 32");
    const int lane = threadIdx.x & 31;
    int idx = 0, off = 16;
#pragma unroll
    for (int h = R / 2; h >= 1; h >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const T send = up ? v[j] : v[j + h];
            const T keep = up ? v[j + h] : v[j];
            v[j] = add_rn(keep, __shfl_xor_sync(kFull, send, off));
        }
        if (up) idx += h;
    }
#pragma unroll
    for (; off >= 1; off >>= 1) v[0] = add_rn(v[0], __shfl_xor_sync(kFull, v[0], off));
    index = idx;
    return v[0];
}

// Float-float numbers (hi, lo as a float2, value hi + lo, |lo| <= ulp(hi) / 2)
// carry the precise path's per-lane sums: they hold ~48 significant bits and
// add on the FP32 pipes, where an fp64 add costs ~64x more on this part.
// Knuth's TwoSum: s + e == a + b exactly.
__device__ __forceinline__ float2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return make_float2(s, e);
}
// a + b for float-float a, b: TwoSum of the high parts, the low parts added to
// the error, then Dekker's Fast2Sum to renormalise.  All terms here are sums of
// squares (no cancellation): relative error below 2^-46 per addition.
__device__ __forceinline__ float2 ff_add(float2 a, float2 b) {
    const float2 s = two_sum(a.x, b.x);
    const float e = __fadd_rn(s.y, __fadd_rn(a.y, b.y));
    const float hi = __fadd_rn(s.x, e);
    return make_float2(hi, __fsub_rn(e, __fsub_rn(hi, s.x)));
}
__device__ __forceinline__ double ff_to_double(float2 v) {
    return __dadd_rn((double)v.x, (double)v.y);
}

// Precise sums of squares on the FP32 pipes.  x*x == p + e exactly, with
// p = fl(x*x) and e = fma(x, x, -p), unless p overflows or e underflows.  p
// joins the running high part by TwoSum, both error terms join the low part,
// and Fast2Sum renormalises the pair, so each addition errs by at most ~2u^2 of
// the running sum (u = 2^-24) with no fp64 instruction; one pair per float4
// component keeps four independent chains in flight.  The streaming loop has no
// range test (a branch there would cost more than the arithmetic): an overflow
// shows as a non-finite pair, and an underflowed e errs by at most 2^-149, so a
// lane sum of at least 2^-77 is as good as exact; dw_lane_ok tests both once
// per tile, and the tile is redone in fp64 when a lane fails.
struct Dw4 {
    float hi[4], lo[4];
};
__device__ __forceinline__ void dw_zero(Dw4 &a) {
#pragma unroll
    for (int c = 0; c < 4; ++c) a.hi[c] = a.lo[c] = 0.f;
}
__device__ __forceinline__ void dw_sq(float &hi, float &lo, float x) {
    const float p = __fmul_rn(x, x);
    const float e = __fmaf_rn(x, x, -p);
    const float2 t = two_sum(hi, p);
    const float l = __fadd_rn(lo, __fadd_rn(t.y, e));
    hi = __fadd_rn(t.x, l);
    lo = __fsub_rn(l, __fsub_rn(hi, t.x));
}
__device__ __forceinline__ void dw_sq4(Dw4 &a, float4 v) {
    dw_sq(a.hi[0], a.lo[0], v.x);
    dw_sq(a.hi[1], a.lo[1], v.y);
    dw_sq(a.hi[2], a.lo[2], v.z);
    dw_sq(a.hi[3], a.lo[3], v.w);
}
// The four pairs added in a fixed tree.
__device__ __forceinline__ float2 dw_pair(const Dw4 &a) {
    const float2 c01 = ff_add(make_float2(a.hi[0], a.lo[0]), make_float2(a.hi[1], a.lo[1]));
    const float2 c23 = ff_add(make_float2(a.hi[2], a.lo[2]), make_float2(a.hi[3], a.lo[3]));
    return ff_add(c01, c23);
}
__device__ __forceinline__ bool dw_lane_ok(float hi) {
    return hi >= 0x1p-77f && hi <= 3.0e38f;  // false for 0, tiny sums, inf and NaN
}

// Triples: the same sum with the errors of its high parts added exactly, too, for tiles whose norms
// hold fp64's precision (misaligned tensors).  Each error joins the middle part by TwoSum, and what
// that rounds off is added up in the low part, so N squares err by at most about (N u)^3 of their
// sum (cascaded summation: Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26, 2005): 4 (N u)^3 with the
// low part's own roundings, 2^-51.4 for the four chains of N <= 72 of the longest tile, where an
// fp64 sum of a lane's 288 squares errs by up to 2^-45.  (72 random squares, the worst of 200 draws:
// triples 2^-53, fp64 2^-50, pairs 2^-46.)  22 fp32 operations a square instead of the pairs' 13:
// 125 us a step of packed buckets (17.3 M elements, K = 4), 118 with pairs.  Overflow and underflow
// show as for pairs.
struct Tw4 {
    float hi[4], md[4], lo[4];
};
__device__ __forceinline__ void tw_zero(Tw4 &a) {
#pragma unroll
    for (int c = 0; c < 4; ++c) a.hi[c] = a.md[c] = a.lo[c] = 0.f;
}
__device__ __forceinline__ void tw_sq(Tw4 &a, int c, float x) {
    const float p = __fmul_rn(x, x);
    const float2 t = two_sum(a.hi[c], p);
    const float2 m = two_sum(a.md[c], t.y);
    const float2 e = two_sum(m.x, __fmaf_rn(x, x, -p));
    a.hi[c] = t.x;
    a.md[c] = e.x;
    a.lo[c] = __fadd_rn(a.lo[c], __fadd_rn(m.y, e.y));
}
// The four triples added in a fixed tree into the first; then as a double, with the high part for
// dw_lane_ok.
__device__ __forceinline__ void tw_add(Tw4 &a, int c, int d) {
    const float2 t = two_sum(a.hi[c], a.hi[d]);
    const float2 m = two_sum(a.md[c], a.md[d]);
    const float2 e = two_sum(m.x, t.y);
    a.hi[c] = t.x;
    a.md[c] = e.x;
    a.lo[c] = __fadd_rn(__fadd_rn(a.lo[c], a.lo[d]), __fadd_rn(m.y, e.y));
}
__device__ __forceinline__ double tw_total(Tw4 &a, float &high) {
    tw_add(a, 0, 1);
    tw_add(a, 2, 3);
    tw_add(a, 0, 2);
    high = a.hi[0];
    return __dadd_rn((double)a.hi[0], __dadd_rn((double)a.md[0], (double)a.lo[0]));
}

// Exact powers of two (k within the normal range of the type).
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

// Range of a tile's fp32 sums of squares, decided for the whole warp from the largest lane
// sum v (>= 0, or NaN): 0 when every lane sum is safe as it stands, else the exponent e of a
// power-of-two scaling 2^e to apply to the elements before squaring them again.
//  * max in [2^-100, 2^120]: nothing overflows (32 lanes add to < 2^125), and squares or partial
//    sums that fell below fp32's normal range err by at most 2^-150 each, < 2^-38 of the tile
//    sum: kept.
//  * max above 2^120, inf or NaN: a square or a sum reached fp32's top.  Scaled by 2^-72 every
//    finite element is below 2^56, its square below 2^112, a lane's sum of up to 288 squares
//    below 2^121 and the tile's below 2^126; what the scaling pushes below 2^-149 has a square
//    under 2^-254 of the tile sum.  Inf and NaN stay inf and NaN.
//  * max below 2^-100 (zero included): every element is below 2^-50 in magnitude (a sum of
//    squares is at least its largest term), so 2^100 x is exact, below 2^50, and its square is a
//    normal number unless x is 0.
constexpr int kScaleUp = 100, kScaleDown = -72;
// Two-bit codes of those exponents, for the partial sums a batch of tiles carries.
__device__ __forceinline__ unsigned scale_code(int e) { return e == 0 ? 0u : (e > 0 ? 1u : 2u); }
__device__ __forceinline__ int scale_exp(unsigned code) {
    return code == 0u ? 0 : (code == 1u ? kScaleUp : kScaleDown);
}
__device__ __forceinline__ bool sq_in_range(float v) {
    return v >= 0x1p-100f && v <= 0x1p120f;  // false for NaN
}
__device__ __forceinline__ int sq_range_exp(float v) {
    const unsigned m = __reduce_max_sync(kFull, __float_as_uint(v));
    if (m > __float_as_uint(0x1p120f)) return kScaleDown;
    if (m < __float_as_uint(0x1p-100f)) return kScaleUp;
    return 0;
}
__device__ __forceinline__ float4 mul4(float4 v, float f) {
    return make_float4(__fmul_rn(v.x, f), __fmul_rn(v.y, f), __fmul_rn(v.z, f), __fmul_rn(v.w, f));
}

// ----------------------------------------------------------------------------
// Exact accumulation of the squared norms
// ----------------------------------------------------------------------------
//
// The partial sums of squares (one per tile and norm, all >= 0) are added up exactly, in
// integers: an accumulator is a fixed-point number of kAccDigits 32-bit digits, digit i of
// weight 2^(32 i + kAccBase), each held in the low half of a 64-bit word whose high half
// collects carries.  A partial m * 2^E (m an fp32 or fp64 significand) touches two or three
// consecutive words, each by an atomic add that nothing waits for (red.global.add.u64).
// Integer addition is associative, so the sum does not depend on the order the tiles land in:
// norms are bitwise reproducible for any grid and any claim order, and they are the exact sums
// of the tile partials, rounded once to fp64 when read (acc_to_double).
//
// Range: the partials are fp32 tile sums scaled by 2^k (k in {0, -200, 144}, sq_range_exp) or
// fp64 sums of exact squares of fp32 numbers, so their bits lie within 2^-352 .. 2^273; a tensor
// of up to 2^31 tiles, or all tensors together, stays below 2^305; 21 digits from 2^-352 cover
// 2^-352 .. 2^320.  To one word a tile adds less than 2 * 2^32: one partial adds to a word once,
// less than 2^32, and the three limbs of a shifted tile's sum together no more than two such adds
// (limbs_max_add).  Only the last tile of a tensor of n % 4 != 0 elements may add up to 4 * 2^32,
// its fp32 sum and the squares of up to three tail elements.  A word therefore stays below 2^64
// while tiles and such tensors together number at most 2^31 (valid_numels).  A partial that is inf
// or NaN (an inf or NaN element) sets a flag in the last word instead: the norm is then inf, or NaN.
//
// Copies: the tiles of one tensor land close together in time, and every tile of a step adds
// into |G|^2, so one word would take an atomic every few ns, about what an L2 slice can do for
// one address.  Each accumulator therefore has copies, picked by the CTA, that the reading warp
// adds up (exact: the bound on a word holds for all copies together).
constexpr int kAccDigits = 21;
constexpr int kAccWords = 24;             // digits, two spare words, the flags
constexpr int kAccFlags = kAccWords - 1;  // bit 0: an inf partial, bit 1: a NaN partial
constexpr int kAccBase = -352;
constexpr int kTCopies = 2;               // copies of each per-tensor accumulator
constexpr int kGCopies = 8;               // copies of the |G|^2 accumulator
static_assert(kAccDigits <= kAccFlags && kAccWords <= 32, "one word per lane");
static_assert((kTCopies & (kTCopies - 1)) == 0 && (kGCopies & (kGCopies - 1)) == 0, "powers of 2");

// Adds m * 2^E (m < 2^53, kAccBase <= E, E + 53 <= 2^32 weight of the top digit) to A.
__device__ __forceinline__ void acc_add(unsigned long long *A, unsigned long long m, int E) {
    if (m == 0ull) return;
    const int s = E - kAccBase;
    const int i = s >> 5, r = s & 31;
    const unsigned long long lo = m << r;
    const unsigned long long hi = r ? (m >> (64 - r)) : 0ull;
    if (lo & 0xffffffffull) atomicAdd(A + i, lo & 0xffffffffull);
    if (lo >> 32) atomicAdd(A + i + 1, lo >> 32);
    if (hi) atomicAdd(A + i + 2, hi);
}
// Adds f * 2^k for an fp32 f >= 0 (or inf, NaN).
__device__ __forceinline__ void acc_add_f32(unsigned long long *A, float f, int k) {
    const unsigned u = __float_as_uint(f);
    const unsigned e = (u >> 23) & 0xffu;
    if (e == 0xffu) {
        atomicOr(A + kAccFlags, (u & 0x7fffffu) ? 2ull : 1ull);
        return;
    }
    const unsigned long long m = e ? ((u & 0x7fffffu) | 0x800000u) : (u & 0x7fffffu);
    acc_add(A, m, (e ? (int)e : 1) - 150 + k);
}
// Adds an fp64 d >= 0 (or inf, NaN).
__device__ __forceinline__ void acc_add_f64(unsigned long long *A, double d) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    const unsigned e = (unsigned)(u >> 52) & 0x7ffu;
    const unsigned long long f = u & 0xfffffffffffffull;
    if (e == 0x7ffu) {
        atomicOr(A + kAccFlags, f ? 2ull : 1ull);
        return;
    }
    acc_add(A, e ? (f | (1ull << 52)) : f, (e ? (int)e : 1) - 1075);
}

// The values of R accumulators rounded to the nearest double (ties to even), by the whole
// warp: lane i passes word i of each (any value for lanes >= kAccWords).  Carries first move up
// one word (each high half, < 2^32, into the next digit), which leaves at most one carry per
// digit; those ripple through runs of all-ones digits, found for all 32 digits at once with two
// votes and one integer addition (the carry-lookahead of an adder).  Then the top three digits
// give the 53-bit significand, its round bit and, with every digit below, its sticky bit.  The
// R conversions go stage by stage together, so their shuffle and vote latencies overlap.
template <int R>
__device__ __forceinline__ void acc_to_double(const unsigned long long (&wi)[R], double (&out)[R]) {
    const int lane = threadIdx.x & 31;
    unsigned long long flags[R], v[R];
    unsigned d[R], nz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) flags[r] = __shfl_sync(kFull, wi[r], kAccFlags);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const unsigned long long w = lane < kAccDigits ? wi[r] : 0ull;
        const unsigned long long up = __shfl_up_sync(kFull, w >> 32, 1);
        v[r] = (w & 0xffffffffull) + (lane > 0 ? up : 0ull);  // < 2^33
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const unsigned G = __ballot_sync(kFull, (v[r] >> 32) != 0ull);
        const unsigned P = __ballot_sync(kFull, (v[r] & 0xffffffffull) == 0xffffffffull);
        const unsigned carries = ((G | P) + G) ^ (G | P) ^ G;  // bit i: a carry into digit i
        d[r] = (unsigned)(v[r] + ((carries >> lane) & 1u));
    }
#pragma unroll
    for (int r = 0; r < R; ++r) nz[r] = __ballot_sync(kFull, d[r] != 0u);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int top = nz[r] ? 31 - __clz(nz[r]) : 0;
        const unsigned d0 = __shfl_sync(kFull, d[r], top);
        const unsigned d1 = __shfl_sync(kFull, d[r], top > 0 ? top - 1 : 0);
        const unsigned d2 = __shfl_sync(kFull, d[r], top > 1 ? top - 2 : 0);
        if (flags[r] & 2ull) {
            out[r] = __longlong_as_double(0x7ff8000000000000ll);  // NaN
        } else if (flags[r] & 1ull) {
            out[r] = __longlong_as_double(0x7ff0000000000000ll);  // +inf
        } else if (nz[r] == 0u) {
            out[r] = 0.0;
        } else {
            const unsigned m1 = top > 0 ? d1 : 0u, m2 = top > 1 ? d2 : 0u;
            const bool below = top > 2 && (nz[r] & ((1u << (top - 2)) - 1u)) != 0u;
            const int L = 32 - __clz(d0);  // bit length of the top digit
            const int z = 32 - L;          // shift that puts its leading 1 at bit 63
            const unsigned long long hi = ((unsigned long long)d0 << 32) | m1;
            const unsigned long long T = (hi << z) | (z ? ((unsigned long long)m2 >> (32 - z)) : 0ull);
            const bool rest = (m2 & (0xffffffffu >> z)) != 0u;  // bits of m2 below T
            unsigned long long mant = T >> 11;
            const bool round = (T >> 10) & 1ull;
            const bool sticky = (T & 0x3ffull) != 0ull || rest || below;
            int ex = 32 * top + kAccBase + L - 1;  // weight of the leading bit
            if (round && (sticky || (mant & 1ull))) {
                if (++mant == (1ull << 53)) {
                    mant >>= 1;
                    ++ex;
                }
            }
            out[r] = __longlong_as_double(
                (long long)(((unsigned long long)(ex + 1023) << 52) | (mant & 0xfffffffffffffull)));
        }
    }
}

// ----------------------------------------------------------------------------
// Device helpers: programmatic dependent launch, mbarrier, TMA (inline PTX)
// ----------------------------------------------------------------------------

// Wait for the grids this one depends on to complete and their memory to be
// visible, then let the next grid in the stream begin launching.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits for the phase of `bar` with this parity to complete; gives up after
// kSpinLimit tries (returns false).  try_wait suspends the thread in hardware
// until the phase completes or a short time limit passes; only a wait that is
// already far too long backs off with a sleep.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (mbar_test(bar, parity)) return true;
        if (i >= (1u << 16)) __nanosleep(256);
    }
    return false;
}
// One TMA bulk copy global -> shared, completing `bytes` of `bar`'s transaction count.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes,
                                         uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(dst),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
// The same with an L2 cache policy for the source lines.
__device__ __forceinline__ void bulk_g2s_hint(uint32_t dst, const void *src, uint32_t bytes,
                                              uint64_t *bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1], %2, [%3], %4;" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
        : "memory");
}
// Fetches `bytes` from src into L2: a hint, which reads nothing into the kernel.
__device__ __forceinline__ void bulk_prefetch(const void *src, uint32_t bytes, bool hint,
                                              uint64_t policy) {
    if (hint)
        asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(src),
                     "r"(bytes), "l"(policy));
    else
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes));
}
// One fp32 global -> shared, asynchronously, by this lane; cp_async_wait() waits for every such
// copy of this lane.
__device__ __forceinline__ void cp_async4(uint32_t dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void fence_async_proxy() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// L2 policy: these lines are the first to go.
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}


__device__ __forceinline__ void report_timeout(const Scalars &sc) {
    atomicOr(sc.err, 1u);
}

// ----------------------------------------------------------------------------
// Tile table lookups
// ----------------------------------------------------------------------------

template <typename Tab>
__device__ __forceinline__ int find_tensor(const Tab &tab, int lo, int hi, int c) {
    // cstart(lo) <= c < cstart(hi)
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (tab.cstart(mid) <= c) lo = mid; else hi = mid;
    }
    return lo;
}

// Follows the tensor index along one warp's tiles, which ascend.  A kernel finds the table outside
// the constant cache, and each step of a search through it is a miss (a search from scratch took
// 2 us before a warp's first copy), so the hints narrow it to the tensors of a few tiles.
struct Walker {
    int t = -1;
    template <typename Tab>
    __device__ __forceinline__ int to(const Tab &tab, int c) {
        if (t >= 0 && c < tab.cstart(t + 1)) return t;
        const int h = c >> tab.hint_shift;
        return t = find_tensor(tab, tab.hint[h], tab.hint[h + 1] + 1, c);
    }
};

// A tile: its tensor, its element range.
struct TilePos {
    int t, tg, c_in_t;
    long long begin, end;
};

template <typename Tab>
__device__ __forceinline__ TilePos locate(const Tab &tab, int c, int t, int chunk) {
    TilePos q;
    q.t = t;
    q.tg = tab.t0 + t;
    q.c_in_t = c - tab.cstart(t);
    q.begin = (long long)q.c_in_t * chunk;
    q.end = min(q.begin + (long long)chunk, tab.numel(t));
    return q;
}

// Float4 a tile moves by TMA: its 16-byte body when every stream of the tensor
// is 16-byte aligned (lane i < ns holds stream i's pointer), else none.
__device__ __forceinline__ int tile_vecs(const float *mine, int ns, const TilePos &q) {
    if (q.end <= q.begin) return 0;
    const unsigned low = (threadIdx.x & 31) < ns ? (unsigned)(reinterpret_cast<uintptr_t>(mine) & 15u)
                                                 : 0u;
    return __reduce_or_sync(kFull, low) == 0u ? (int)((q.end - q.begin) >> 2) : 0;
}

// The tensor of the previous tile, kept while the next tile stays in it: its
// index, its streams' alignment and the lane's stream pointer, so a tile in
// the same tensor needs no table look-up.
template <bool SH>
struct TensorCache {
    Walker walk;
    int t = -1;
    long long numel = 0;
    const float *mine = nullptr;
    unsigned long long base = 0;  // of the lane's role
    bool aligned = !SH;    // every stream at a 16-byte boundary
    int nv = 0;            // whole float4 columns of the last tile asked for (0: a shifted tile)
    template <typename Tab>
    __device__ __forceinline__ TilePos at(const Tab &tab, int c, int chunk, int role, int ns) {
        const int tn = walk.to(tab, c);
        if (tn != t) {
            t = tn;
            numel = tab.numel(t);
            if (base == 0ull) base = tab.base[role];
            mine = (threadIdx.x & 31) < ns ? tab.ptr(t, role, base) : nullptr;
            if constexpr (SH) {
                const unsigned low =
                    (threadIdx.x & 31) < ns ? (unsigned)(reinterpret_cast<uintptr_t>(mine) & 15u) : 0u;
                aligned = __reduce_or_sync(kFull, low) == 0u;
            }
        }
        TilePos q;
        q.t = t;
        q.tg = tab.t0 + t;
        q.c_in_t = c - tab.cstart(t);
        q.begin = (long long)q.c_in_t * chunk;
        q.end = min(q.begin + (long long)chunk, numel);
        nv = (aligned && q.end > q.begin) ? (int)((q.end - q.begin) >> 2) : 0;
        return q;
    }
    // Stream i's pointer, from the lane that holds it (the table may miss the constant cache).
    __device__ __forceinline__ float *stream(int i) const {
        return reinterpret_cast<float *>(
            __shfl_sync(kFull, (unsigned long long)reinterpret_cast<uintptr_t>(mine), i));
    }
};

// ----------------------------------------------------------------------------
// Streaming warps: TMA bulk copies of each tile's streams into a warp's own stage
// ----------------------------------------------------------------------------
//
// Each warp streams for itself: it has one stage of shared memory and one mbarrier, waits for the
// tile in it, computes, and issues its next tile into the same stage as soon as every lane has read
// the last one, before it adds that tile's sums up.  Lane i < ns fetches stream i's pointer (role
// i) and issues that stream's copy to offset i * chunk floats of the stage.  While one warp
// of a CTA computes, the others' copies are in flight; nothing is handed from warp to warp.
// One producer warp for all of them would bound the passes: a warp issues a bulk copy every ~27 ns
// (the lanes of one instruction go in turn), so 16 streams of 2 KB would take 0.83 us of a 36 KB
// stage's 0.80 us at the HBM rate, and 8 streams delay every refill.  Streams read this way alone
// run at 6.95-6.99 TB/s whatever the copy size (512 B to 18 KB), against 6.09 TB/s with one
// producer warp and 16 copies of 2 KB.
//
// Dealing: a launch has V = gridDim.x * kWarps streaming warps; warp v first takes tile v, then,
// when there are more tiles than warps, tiles claimed one at a time from a global counter
// (ctr[0]), the claim made a whole tile ahead so that its round trip passes while the tile issued
// before it is on its way (claim()).  SMs stream at unequal rates; with 36 KB tiles claims run at
// 7.19-7.25 TB/s where a fixed deal runs at 6.95.  (Tiles under ~18 KB would be bound by the
// counter: one atomic every 1.5-2.8 ns.)  A launch of nc tiles that claims makes exactly nc claims
// (nc - V tiles and one past the end for each warp), so the host knows where the next launch on the
// counter begins, and nobody waits at the end of a launch to re-arm it: the update does that for
// pass 1 (k_share in a sharded step), k_finish for pass 2 and for the calls without an update.  (A
// fence and a ticket per warp would take about 1 us at the end of each pass.)  Where a tile is
// processed never changes its result: each tile's partial sums are added exactly, in integers,
// into its tensor's accumulators.
//
// Any 4-byte aligned tensor moves this way.  When some stream of a tensor lies off a 16-byte
// boundary (views into a flat bucket, say), its tiles are shifted: stream i's part of the stage
// starts at i * (4 * chunk + kShiftBytes) and holds the 16-byte granules that the tile touches and
// that lie wholly inside the tensor, so element j of the tile sits addr & 12 bytes plus 4 j in,
// whatever the streams' alignments are to one another.  (The first and last granule may bring
// elements of the neighbouring tiles along, which another warp may be updating; nobody reads
// them.)  The up to three elements at each end of a tensor outside those granules, and the last
// n % 4 elements of an aligned tensor, come by 4-byte cp.async into the same places.  Only the
// kernels for launches with such a tensor (SH) hold this code: in the others it would cost 0.4 %
// (ResNet-50) to 5 % (1024 small layers) of a step, and they load an aligned tensor's tail
// directly.  17.3 M elements in 128 tensors, K = 4, the gradients packed, take 125 us a step,
// against 101 us aligned, and 548 loaded one element at a time and squared in fp64.

// A shifted tile, or the last tile of an aligned tensor of n % 4 != 0 elements: this lane's stream
// (mine; nullptr: none) of n elements from `begin` of a tensor with `rest` elements from there on.
// part: the lane's part of the stage.  The bytes of all streams are armed by lane 0 when `arm`.
// Out of line, so that the path of ordinary tiles stays short.
__device__ __noinline__ void issue_edge_tile(uint32_t part, const float *mine, bool aligned,
                                             long long begin, int n, long long rest, bool arm,
                                             bool copy, uint64_t *bar, bool hint, uint64_t policy) {
    // Elements [lo, hi) of this lane's stream, counted from the tile's first, come in bulk.
    int lo = 0, hi = n & ~3;
    if (!aligned) {
        const int phi = (int)(reinterpret_cast<uintptr_t>(mine) & 15u) >> 2;
        const long long inside = rest - ((phi + rest) & 3);
        const int up = (4 - phi) & 3;
        lo = begin == 0 ? up : -phi;
        hi = (int)min((long long)(n + up), inside);
        if (hi < lo) hi = lo;
        part += (uint32_t)(4 * phi);
    }
    if (!mine) hi = lo;
    const uint32_t bytes = 4u * (uint32_t)(hi - lo);
    const uint32_t expect = __reduce_add_sync(kFull, bytes);
    if (arm && (threadIdx.x & 31) == 0) mbar_arrive_tx(bar, expect);
    __syncwarp();
    if (!mine || !copy) return;
    const float *src = mine + begin;
    if (bytes) {
        const uint32_t to = part + 4u * (uint32_t)lo;  // lo may be negative: modulo 2^32
        if (hint) bulk_g2s_hint(to, src + lo, bytes, bar, policy);
        else bulk_g2s(to, src + lo, bytes, bar);
    }
    const int head = bytes ? max(lo, 0) : n, tail = bytes ? min(hi, n) : n;
    for (int e = 0; e < head; ++e) cp_async4(part + 4u * (uint32_t)e, src + e);
    for (int e = tail; e < n; ++e) cp_async4(part + 4u * (uint32_t)e, src + e);
}

template <typename R, bool SH>
struct Stream {
    uint32_t stage;  // shared-memory address of this warp's stage
    uint64_t *bar;   // its mbarrier: one arrival, which arms the bytes of all streams
    uint32_t phase = 0;
    unsigned nc, V, base;
    bool claims;
    unsigned *ctr;
    unsigned pend = 0;  // lane 0: the claim in flight
    uint64_t policy;
    bool hint;
    TensorCache<SH> tc;  // of the tile in the stage (or on its way there)
    bool edges = false;  // SH: it came partly by cp.async

    // Barrier init; returns this warp's first tile (-1: none).  Called by the whole CTA.
    __device__ __forceinline__ int start(unsigned char *smem, int n_tiles, unsigned *counter,
                                         const Scalars &sc) {
        const int warp = threadIdx.x >> 5;
        stage = smem_addr(smem) + (uint32_t)warp * R::kStageBytes;
        bar = reinterpret_cast<uint64_t *>(smem + R::kWarps * R::kStageBytes) + warp;
        if ((threadIdx.x & 31) == 0) {
            mbar_init(bar, 1);
            mbar_fence_init();
        }
        __syncwarp();
        nc = (unsigned)n_tiles;
        V = gridDim.x * (unsigned)R::kWarps;
        claims = nc > V;
        ctr = counter;
        base = sc.claim_base;
        hint = sc.evict_first != 0;
        policy = policy_evict_first();
        const unsigned v = (unsigned)warp * gridDim.x + blockIdx.x;
        return v < nc ? (int)v : -1;
    }
    // cp.async (the ends of shifted tiles) reads through L1, 32 bytes at a time, which bring the
    // neighbouring elements along: whatever L1 holds from before a wait is given up by a fence after
    // it, before elements that another kernel has written meanwhile are read this way.
    __device__ __forceinline__ void forget_l1() const {
        if constexpr (SH) __threadfence();
    }
    // Claims the tile after the one just issued: after, because the warp may stop for the
    // atomic's round trip here (its tile is on its way meanwhile; claimed before the copies, it
    // kept every stage empty for about 1500 of a tile's 10,500 cycles).
    __device__ __forceinline__ void claim() {
        if (claims && (threadIdx.x & 31) == 0) pend = atomicAdd(ctr, 1u);
    }
    // The tile claimed last (-1: none left).
    __device__ __forceinline__ int next() {
        if (!claims) return -1;
        const unsigned c = __shfl_sync(kFull, pend, 0) - base + V;
        return c < nc ? (int)c : -1;
    }
    // Issues tile c, or of it only streams `from` .. ns - 1, the rest left to issue_below();
    // every lane has read what the stage held (a __syncwarp ago).
    template <typename Tab>
    __device__ __forceinline__ TilePos issue(const Tab &tab, int c, int chunk, int role,
                                             int ns, int from = 0) {
        const int lane = threadIdx.x & 31;
        const TilePos q = tc.at(tab, c, chunk, role, ns);
        if constexpr (SH) {
            const int n = (int)(q.end - q.begin);
            if (edges) fence_async_proxy();  // cp.async wrote the stage: before bulk copies do
            edges = n > 0 && !(tc.aligned && (n & 3) == 0);
            if (edges) {
                edge(q, lane, lane >= from && lane < ns, lane < ns, chunk, true);
                return q;
            }
        }
        if (lane == 0) mbar_arrive_tx(bar, 16u * (uint32_t)(tc.nv * ns));
        __syncwarp();
        if (lane >= from && lane < ns) copy(q, lane, chunk);
        return q;
    }
    __device__ __forceinline__ void issue_below(const TilePos &q, int from, int ns, int chunk) {
        const int lane = threadIdx.x & 31;
        if (SH && edges) edge(q, lane, lane < from, lane < ns, chunk, false);
        else if (lane < from) copy(q, lane, chunk);
    }
    __device__ __forceinline__ void edge(const TilePos &q, int lane, bool mine, bool stream,
                                         int chunk, bool arm) {
        const uint32_t part = (uint32_t)(4 * chunk + (tc.aligned ? 0 : kShiftBytes));
        issue_edge_tile(stage + (uint32_t)lane * part, stream ? tc.mine : nullptr, tc.aligned,
                        q.begin, (int)(q.end - q.begin), tc.numel - q.begin, arm, mine, bar, hint,
                        policy);
    }
    // Has L2 fetch tile c, to be issued later; of a shifted one what lies between its first and
    // last 16-byte boundary.
    template <typename Tab>
    __device__ __forceinline__ void prefetch(const Tab &tab, int c, int chunk, int role, int ns) {
        const TilePos q = tc.at(tab, c, chunk, role, ns);
        if ((int)(threadIdx.x & 31) >= ns) return;
        int n = (int)(q.end - q.begin);
        const float *src = tc.mine + q.begin;
        if constexpr (SH) {
            const int up = (int)(-(reinterpret_cast<uintptr_t>(src) >> 2) & 3u);
            src += up;
            n -= up;
        }
        if (n >= 4) bulk_prefetch(src, 16u * (uint32_t)(n >> 2), hint, policy);
    }
    __device__ __forceinline__ void copy(const TilePos &q, int lane, int chunk) {
        const uint32_t bytes = 16u * (uint32_t)tc.nv;
        if (bytes) {
            const uint32_t dst = stage + (uint32_t)(lane * chunk * 4);
            if (hint) bulk_g2s_hint(dst, tc.mine + q.begin, bytes, bar, policy);
            else bulk_g2s(dst, tc.mine + q.begin, bytes, bar);
        }
    }
    // Waits for the tile in the stage.  false: the wait ran out (reported); the copies are then
    // given as long again to land, so that the CTA does not end with them in flight, and the
    // warp must stop.  The same in every lane.
    __device__ __forceinline__ bool arrived(const Scalars &sc) {
        const bool ok = __all_sync(kFull, mbar_wait(bar, phase));
        if (!ok) {
            if ((threadIdx.x & 31) == 0) report_timeout(sc);
            mbar_wait(bar, phase);
            claims = false;
        }
        phase ^= 1u;
        if (SH && edges) {  // each lane's cp.async copies, then every lane's are there
            cp_async_wait();
            __syncwarp();
        }
        return ok;
    }
};

// ----------------------------------------------------------------------------
// Pass 1: replica mean + per-tile squared norms
// ----------------------------------------------------------------------------
//
// Template: KT = replicas known at compile time (0: runtime K <= 16);
// WM = write the mean over replica 0; RW = also reduce |w|^2;
// SS = g_small is a separate stream instead of replica 0;
// PR = precise norms: every square is split exactly into two fp32 parts and
// added as a float-float pair (Dw4), each lane's pairs go to fp64 once per tile,
// and the tile's lanes are added in an fp64 tree (relative error ~1e-14), for
// norms that feed a per-tensor coefficient (UpdateGradScale, LARS).  Otherwise the tile's sum
// stays in fp32: each lane adds <= 16 squares per group of 4 columns, then the
// group sums, then a 5-level tree across lanes, a relative error below 71 ulp
// (4e-6) of the tile's sum; tiles are added exactly into the tensor's
// accumulator.  That is what the
// variability metric and the statistics need, and it keeps GB300's slow FP64
// pipe out of the streaming loop.  One warp vote per tile (sq_range_exp) keeps
// it valid over the whole fp32 range: a tile whose fp32 sums would overflow or
// lose precision to underflow is summed again from shared memory with its
// elements scaled by an exact power of two, and the scaling is undone in fp64.
// Pointer roles per tensor: [0, K) replicas, K = w (RW) or g_small (SS).
// Stage streams: replicas 0..K-1, then w (RW), then g_small (SS).

// Whether there is more than one replica: K = 1 has a kernel of its own, so that this is known at
// compile time for a K that is not.  (Tested at run time, it kept the four elements' chains of a
// step apart: a shifted tile with K = 3 took 21,000 cycles, and 16,600 so.)
template <int KT>
constexpr bool kMulti = KT != 1;

// One float4 column of a tile: mean, squares.  x0 = replica 0, s = sum.
template <int KT, bool WM, bool RW, bool SS, bool PR>
__device__ __forceinline__ void column1(float4 x0, float4 s, float4 wv, float4 sv, float *out,
                                        const Scalars &sc, Dw4 &ag, Dw4 &as, Dw4 &aw,
                                        float &pg, float &ps, float &pw) {
    if (kMulti<KT>) {
        s = mean4<KT>(s, mean_k(sc));
        if (WM) st_keep(out, s);
    }
    if (PR) {
        dw_sq4(ag, s);
        if (kMulti<KT>) dw_sq4(as, x0);
        if (SS) dw_sq4(as, sv);
        if (RW) dw_sq4(aw, wv);
    } else {
        pg = sq4(pg, s);
        if (kMulti<KT>) ps = sq4(ps, x0);
        if (SS) ps = sq4(ps, sv);
        if (RW) pw = sq4(pw, wv);
    }
}

// A tile's shared-memory columns again, every square exact in fp64 and added
// in fp64: the precise path's fallback when a lane's float-float sum is not
// finite or too small to hold its error (dw_lane_ok).  Out of line, so that
// the streaming loop keeps its shape.
struct D3 {
    double g, s, w;
};
template <int KT, bool RW, bool SS>
__device__ __noinline__ D3 tile_cols_fp64(uint32_t stage, int chunk, int nv, const Scalars &sc) {
    const int lane = threadIdx.x & 31;
    const int K = KT > 0 ? KT : sc.K;
    const uint32_t sw_s = stage + (uint32_t)(K * chunk * 4);
    const uint32_t ss_s = stage + (uint32_t)((K + (RW ? 1 : 0)) * chunk * 4);
    D3 r = {0.0, 0.0, 0.0};
    for (int v = lane; v < nv; v += 32) {
        const float4 x0 = lds4(stage + (uint32_t)(16 * v));
        float4 s = x0;
        for (int k = 1; k < K; ++k) s = add4(s, lds4(stage + (uint32_t)((k * chunk + 4 * v) * 4)));
        if (kMulti<KT>) s = mean4<KT>(s, mean_k(sc));
        const float gs[4] = {s.x, s.y, s.z, s.w};
        const float g0[4] = {x0.x, x0.y, x0.z, x0.w};
        float4 wv = make_float4(0.f, 0.f, 0.f, 0.f), sv = wv;
        if (RW) wv = lds4(sw_s + (uint32_t)(16 * v));
        if (SS) sv = lds4(ss_s + (uint32_t)(16 * v));
        const float ws[4] = {wv.x, wv.y, wv.z, wv.w};
        const float ss[4] = {sv.x, sv.y, sv.z, sv.w};
        for (int c = 0; c < 4; ++c) {
            r.g = __fma_rn((double)gs[c], (double)gs[c], r.g);
            if (kMulti<KT>) r.s = __fma_rn((double)g0[c], (double)g0[c], r.s);
            if (SS) r.s = __fma_rn((double)ss[c], (double)ss[c], r.s);
            if (RW) r.w = __fma_rn((double)ws[c], (double)ws[c], r.w);
        }
    }
    return r;
}

// A tile's shared-memory columns again in fp32, every element multiplied by an exact power of
// two first (sq_range_exp): the default path's fallback when a tile's fp32 sums of squares
// would overflow or lose their precision to underflow.  Returns this lane's sums of the scaled
// squares.  Out of line, so that the streaming loop keeps its shape.
struct F3 {
    float g, s, w;
};
template <int KT, bool RW, bool SS>
__device__ __noinline__ F3 tile_cols_scaled(uint32_t stage, int chunk, int nv, const Scalars &sc,
                                            float fg, float fs, float fw) {
    const int lane = threadIdx.x & 31;
    const int K = KT > 0 ? KT : sc.K;
    const uint32_t sw_s = stage + (uint32_t)(K * chunk * 4);
    const uint32_t ss_s = stage + (uint32_t)((K + (RW ? 1 : 0)) * chunk * 4);
    F3 r = {0.f, 0.f, 0.f};
    for (int v = lane; v < nv; v += 32) {
        const float4 x0 = lds4(stage + (uint32_t)(16 * v));
        float4 s = x0;
        for (int k = 1; k < K; ++k) s = add4(s, lds4(stage + (uint32_t)((k * chunk + 4 * v) * 4)));
        if (kMulti<KT>) s = mean4<KT>(s, mean_k(sc));
        r.g = sq4(r.g, mul4(s, fg));
        if (kMulti<KT>) r.s = sq4(r.s, mul4(x0, fs));
        if (SS) r.s = sq4(r.s, mul4(lds4(ss_s + (uint32_t)(16 * v)), fs));
        if (RW) r.w = sq4(r.w, mul4(lds4(sw_s + (uint32_t)(16 * v)), fw));
    }
    return r;
}

// A tile of a tensor off a 16-byte boundary (see issue_edge_tile() for where its elements lie):
// lane l takes elements l, l + 32, ..., four at a time, with conflict-free 4-byte loads from shared
// memory and coalesced 4-byte stores of the mean.  The squares are added as triples in either
// mode, so that these norms hold fp64's precision.  Returns the lane's sums; out of line, so that
// the streaming loop of aligned tensors keeps its shape.
template <int KT, bool WM, bool RW, bool SS, typename Tab>
__device__ __noinline__ D3 tile_shifted(uint32_t stage, int chunk, const Tab &tab, int t,
                                        long long begin, int n, const Scalars &sc) {
    const Row<Tab> ptr{tab, t};
    const MeanK mk = mean_k(sc);
    const int lane = threadIdx.x & 31;
    const int K = KT > 0 ? KT : sc.K;
    const uint32_t part = (uint32_t)(4 * chunk + kShiftBytes);
    // The streams' places within 16 bytes, two bits each (roles and streams are the same here): a
    // look-up in the table for every load costs more than the load.
    constexpr bool kExtra = RW || SS;
    unsigned long long phases = 0ull;
    for (int i = 0; i < K + (kExtra ? 1 : 0); ++i)
        phases |= (unsigned long long)((reinterpret_cast<uintptr_t>(ptr[i]) >> 2) & 3u) << (2 * i);
    auto at = [&](int i) {
        return stage + (uint32_t)i * part + ((uint32_t)(phases >> (2 * i)) & 3u) * 4u;
    };
    uint32_t at_k[KT > 0 ? KT : 1];
#pragma unroll
    for (int k = 0; k < (KT > 0 ? KT : 1); ++k) at_k[k] = at(k);
    static_assert(!(RW && SS), "one of them is role K");
    const uint32_t at_w = RW ? at(K) : 0u;
    const uint32_t at_s = SS ? at(K) : 0u;
    float *out = ptr[0] + begin;
    // Four elements per lane and step: their independent chains hide one another's latency.
    constexpr int U = 4;
    Tw4 ag, as, aw;
    tw_zero(ag);
    tw_zero(as);
    tw_zero(aw);
    // One step from element j0 on; the elements past the end count as 0.
    auto step = [&](int j0, auto whole) {
        constexpr bool kWhole = decltype(whole)::value;
        uint32_t o[U];  // byte offsets; past the end, the last element's
        bool in[U];
        float x0[U], s[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            in[u] = kWhole || j0 + 32 * u < n;
            o[u] = 4u * (uint32_t)(kWhole ? j0 + 32 * u : min(j0 + 32 * u, n - 1));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) s[u] = x0[u] = lds1(at_k[0] + o[u]);
        if constexpr (KT > 0) {
#pragma unroll
            for (int k = 1; k < KT; ++k)
#pragma unroll
                for (int u = 0; u < U; ++u) s[u] = __fadd_rn(s[u], lds1(at_k[k] + o[u]));
        } else {
            for (int k = 1; k < K; ++k) {
                const uint32_t a = at(k);
#pragma unroll
                for (int u = 0; u < U; ++u) s[u] = __fadd_rn(s[u], lds1(a + o[u]));
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) y[u] = RW || SS ? lds1((RW ? at_w : at_s) + o[u]) : 0.f;
        if (kMulti<KT>) {
            const float4 m = mean4<KT>(make_float4(s[0], s[1], s[2], s[3]), mk);
            s[0] = m.x;
            s[1] = m.y;
            s[2] = m.z;
            s[3] = m.w;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (kMulti<KT> && WM && in[u]) out[j0 + 32 * u] = s[u];
            tw_sq(ag, u, in[u] ? s[u] : 0.f);
            if (kMulti<KT>) tw_sq(as, u, in[u] ? x0[u] : 0.f);
            if (SS) tw_sq(as, u, in[u] ? y[u] : 0.f);
            if (RW) tw_sq(aw, u, in[u] ? y[u] : 0.f);
        }
    };
    int j = lane;
#pragma unroll 1
    for (; j - lane + 32 * U <= n; j += 32 * U) step(j, std::true_type{});
    if (j - lane < n) step(j, std::false_type{});
    __syncwarp();
    float hg, hs, hw;
    D3 r = {tw_total(ag, hg), tw_total(as, hs), tw_total(aw, hw)};
    const bool bad = lane < n && !(dw_lane_ok(hg) && (!(kMulti<KT> || SS) || dw_lane_ok(hs)) &&
                                   (!RW || dw_lane_ok(hw)));
    if (__any_sync(kFull, bad)) {  // as tile_cols_fp64: again, every square exact in fp64
        r = {0.0, 0.0, 0.0};
        for (int j = lane; j < n; j += 32) {
            const uint32_t o = 4u * (uint32_t)j;
            const float x0 = lds1(at_k[0] + o);
            float s = x0;
            for (int k = 1; k < K; ++k) s = __fadd_rn(s, lds1(at(k) + o));
            if (kMulti<KT>) s = mean1<KT>(s, mk);
            r.g = __fma_rn((double)s, (double)s, r.g);
            if (kMulti<KT>) r.s = __fma_rn((double)x0, (double)x0, r.s);
            if (SS) {
                const double y = (double)lds1(at_s + o);
                r.s = __fma_rn(y, y, r.s);
            }
            if (RW) {
                const double y = (double)lds1(at_w + o);
                r.w = __fma_rn(y, y, r.w);
            }
        }
        __syncwarp();
    }
    return r;
}

// Per-lane partial sums of one tile (not yet reduced across the warp).  Precise mode (PR):
// accd holds the lane's fp64 sums.  Default mode: accf holds the lane's fp32 sums over the
// tile's float4 columns, scaled by 2^(2 e) with e coded in `ecode` (the same in every lane), accd
// the lane's fp64 sums over the elements taken one by one (tail, shifted tile).
template <int KT, bool WM, bool RW, bool SS, bool PR, bool SH, typename Tab>
__device__ __forceinline__ void reduce_tile(uint32_t stage, int chunk, const Row<Tab> ptr,
                                            float *out0, const TilePos &q, int nv, bool aligned,
                                            const Scalars &sc, double (&accd)[kAcc], float (&accf)[kAcc],
                                            unsigned &ecode, bool &tail) {
    const int lane = threadIdx.x & 31;
    const int K = KT > 0 ? KT : sc.K;
    const uint32_t sw_s = stage + (uint32_t)(K * chunk * 4);
    const uint32_t ss_s = stage + (uint32_t)((K + (RW ? 1 : 0)) * chunk * 4);
    float *out = out0 + q.begin;
    Dw4 ag, as, aw;                       // precise (PR) sums of the shared-memory columns
    dw_zero(ag);
    dw_zero(as);
    dw_zero(aw);
    double rg = 0.0, rs = 0.0, rw = 0.0;  // exact fp64 sums of the tail
    const int ncols = nv;                 // the float4 columns (nv is reused below)
    tail = false;                         // the tile has elements taken one by one
    ecode = 0u;                           // scale_code of sum a's exponent in bits 2a, 2a + 1
    if (SH && !aligned) {
        const D3 d = tile_shifted<KT, WM, RW, SS>(stage, chunk, ptr.tab, ptr.t, q.begin,
                                                         (int)(q.end - q.begin), sc);
        accd[0] = d.g;
        accd[1] = (kMulti<KT> || SS) ? d.s : d.g;  // K = 1: replica 0 is the mean
        accd[2] = d.w;
        accf[0] = accf[1] = accf[2] = 0.f;
        tail = true;
        return;
    }
    float fg = 0.f, fs = 0.f, fw = 0.f;   // fp32 sums (not PR)

    if constexpr (KT > 0) {
        constexpr int CH = Ring1Of<KT, RW, SH>::tile_elems(KT + (RW ? 1 : 0) + (SS ? 1 : 0));
        constexpr int COLS = CH / 128;  // float4 columns per lane of a full tile
        if (nv == CH / 4) {
            // Full tile: every lane has COLS columns; all loads of a column issue together.
            // The loop over groups of G columns stays rolled: unrolled over the tile (and
            // again for each of the kPend tiles), the body outgrows the instruction cache.
            // The precise path's float-float arithmetic takes kPrecCols columns per group.
            constexpr int G = PR ? kPrecCols : 4;
#pragma unroll 1
            for (int c0 = 0; c0 < COLS; c0 += G) {
                float pg = 0.f, ps = 0.f, pw = 0.f;
#pragma unroll
                for (int u = 0; u < G; ++u) {
                    if (c0 + u < COLS) {
                        const int v = lane + 32 * (c0 + u);
                        float4 x[KT];
#pragma unroll
                        for (int k = 0; k < KT; ++k)
                            x[k] = lds4(stage + (uint32_t)((k * CH + 4 * v) * 4));
                        const float4 wv = RW ? lds4(sw_s + (uint32_t)(16 * v)) : x[0];
                        const float4 sv = SS ? lds4(ss_s + (uint32_t)(16 * v)) : x[0];
                        float4 s = x[0];
#pragma unroll
                        for (int k = 1; k < KT; ++k) s = add4(s, x[k]);
                        column1<KT, WM, RW, SS, PR>(x[0], s, wv, sv, out + 4 * v, sc, ag, as, aw,
                                                    pg, ps, pw);
                    }
                }
                if (!PR) {
                    fg = __fadd_rn(fg, pg);
                    if (kMulti<KT> || SS) fs = __fadd_rn(fs, ps);
                    if (RW) fw = __fadd_rn(fw, pw);
                }
            }
            nv = -1;  // done
        }
    }
    if (nv >= 0) {
        // Ragged tile, or K known only at run time.  The latter takes U columns together, replica
        // by replica, so that U loads are always in flight (ResNet-50, K = 6: 213 us a step, and
        // 234 one column at a time, each load waiting for the one before).
        constexpr int U = PR ? 2 : 4;
        // The tail's loads go first (not SH, K known: one lane per element), to land meanwhile.
        constexpr bool kTailFirst = !SH && KT > 0;
        constexpr int kTailRoles = kTailFirst ? KT + (RW || SS ? 1 : 0) : 1;
        const long long tail_at = q.begin + 4 * (long long)nv;
        float xt[kTailRoles] = {};
        if (kTailFirst && tail_at + lane < q.end) {
#pragma unroll
            for (int k = 0; k < kTailRoles; ++k) xt[k] = __ldcg(ptr[k] + tail_at + lane);
        }
        for (int v0 = lane; v0 < nv; v0 += 32 * 4) {
            float pg = 0.f, ps = 0.f, pw = 0.f;
            if constexpr (KT > 0) {
                for (int u = 0; u < 4; ++u) {
                    const int v = v0 + 32 * u;
                    if (v >= nv) break;
                    const float4 x0 = lds4(stage + (uint32_t)(16 * v));
                    float4 s = x0;
                    for (int k = 1; k < K; ++k)
                        s = add4(s, lds4(stage + (uint32_t)((k * chunk + 4 * v) * 4)));
                    const float4 wv = RW ? lds4(sw_s + (uint32_t)(16 * v)) : x0;
                    const float4 sv = SS ? lds4(ss_s + (uint32_t)(16 * v)) : x0;
                    column1<KT, WM, RW, SS, PR>(x0, s, wv, sv, out + 4 * v, sc, ag, as, aw, pg,
                                                ps, pw);
                }
            } else {
#pragma unroll 1
                for (int u0 = 0; u0 < 4 && v0 + 32 * u0 < nv; u0 += U) {
                    uint32_t o[U];  // byte offsets; past the end, the last column's (not used)
                    float4 x0[U], s[U], wv[U], sv[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        o[u] = 16u * (uint32_t)min(v0 + 32 * (u0 + u), nv - 1);
                        s[u] = x0[u] = lds4(stage + o[u]);
                    }
#pragma unroll 4
                    for (int k = 1; k < K; ++k) {
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            s[u] = add4(s[u], lds4(stage + (uint32_t)(k * chunk * 4) + o[u]));
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        wv[u] = RW ? lds4(sw_s + o[u]) : x0[u];
                        sv[u] = SS ? lds4(ss_s + o[u]) : x0[u];
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int v = v0 + 32 * (u0 + u);
                        if (v < nv)
                            column1<KT, WM, RW, SS, PR>(x0[u], s[u], wv[u], sv[u], out + 4 * v, sc,
                                                        ag, as, aw, pg, ps, pw);
                    }
                }
            }
            if (!PR) {
                fg = __fadd_rn(fg, pg);
                if (kMulti<KT> || SS) fs = __fadd_rn(fs, ps);
                if (RW) fw = __fadd_rn(fw, pw);
            }
        }
        // The last n % 4 elements, exact squares in fp64: from the stage (SH) or by plain loads.
        tail = tail_at < q.end;  // the same in every lane
        if (tail_at + lane < q.end) {
            const long long j = tail_at + lane;
            const uint32_t o = 4u * (uint32_t)(j - q.begin);
            const float x0 = SH ? lds1(stage + o) : kTailFirst ? xt[0] : __ldcg(ptr[0] + j);
            float s = x0;
            if constexpr (kTailFirst) {
#pragma unroll
                for (int k = 1; k < KT; ++k) s = __fadd_rn(s, xt[k]);
            } else {
                for (int k = 1; k < K; ++k)
                    s = __fadd_rn(s, SH ? lds1(stage + (uint32_t)(4 * k * chunk) + o)
                                        : __ldcg(ptr[k] + j));
            }
            if (kMulti<KT>) {
                s = mean1<KT>(s, mean_k(sc));
                if (WM) out0[j] = s;
            }
            if (kMulti<KT>) rs = __fma_rn((double)x0, (double)x0, rs);
            rg = __fma_rn((double)s, (double)s, rg);
            if (RW || SS) {  // role K
                const float y = SH ? lds1((RW ? sw_s : ss_s) + o)
                                   : kTailFirst ? xt[kTailRoles - 1] : __ldcg(ptr[K] + j);
                double &r = RW ? rw : rs;
                r = __fma_rn((double)y, (double)y, r);
            }
        }
    }
    if (PR) {
        // The warp is converged again here (the loops above end in every lane).
        const float2 pg = dw_pair(ag), ps = dw_pair(as), pw = dw_pair(aw);
        const bool bad = lane < ncols && !(dw_lane_ok(pg.x) &&
                                           (!(kMulti<KT> || SS) || dw_lane_ok(ps.x)) &&
                                           (!RW || dw_lane_ok(pw.x)));
        double cg, cs, cw;
        if (__any_sync(kFull, bad)) {
            const D3 f = tile_cols_fp64<KT, RW, SS>(stage, chunk, ncols, sc);
            cg = f.g;
            cs = f.s;
            cw = f.w;
        } else {
            cg = ff_to_double(pg);
            cs = ff_to_double(ps);
            cw = ff_to_double(pw);
        }
        accd[0] = __dadd_rn(cg, rg);
        accd[1] = (kMulti<KT> || SS) ? __dadd_rn(cs, rs) : accd[0];  // K = 1: replica 0 is the mean
        accd[2] = RW ? __dadd_rn(cw, rw) : 0.0;
    } else {
        // The warp is converged again here; ncols is the same in every lane.
        int eg = 0, es = 0, ew = 0;
        // One vote per tile; the warp maxima only when some lane is out of range.  A lane
        // without columns (lane >= ncols) has nothing to check.
        const bool lane_ok =
            lane >= ncols || (sq_in_range(fg) && (!(kMulti<KT> || SS) || sq_in_range(fs)) &&
                              (!RW || sq_in_range(fw)));
        if (ncols > 0 && !__all_sync(kFull, lane_ok)) {
            eg = sq_range_exp(fg);
            if (kMulti<KT> || SS) es = sq_range_exp(fs);
            if (RW) ew = sq_range_exp(fw);
            if (eg | es | ew) {
                const F3 r = tile_cols_scaled<KT, RW, SS>(stage, chunk, ncols, sc, pow2f(eg),
                                                          pow2f(es), pow2f(ew));
                if (eg) fg = r.g;
                if (es) fs = r.s;
                if (ew) fw = r.w;
                const bool own = kMulti<KT> || SS;
                ecode = scale_code(eg) | scale_code(own ? es : eg) << 2 | scale_code(ew) << 4;
            }
        }
        const bool own_s = kMulti<KT> || SS;  // K = 1: replica 0 is the mean
        accf[0] = fg;
        accd[0] = rg;
        accf[1] = own_s ? fs : fg;
        accd[1] = own_s ? rs : rg;
        accf[2] = fw;
        accd[2] = rw;
    }
}

static_assert(kPend == 4, "the owner lanes below pick one of four tiles");

// This CTA's copies of the accumulators: tensor tg's pass-1 norm a, |G|^2, tensor tg's |w|^2
// in pass 2.
__device__ __forceinline__ unsigned long long *acc1_of(const Scalars &sc, int tg, int a) {
    return sc.acc1 + (((size_t)tg * kAcc + a) * kTCopies + (blockIdx.x & (kTCopies - 1))) * kAccWords;
}
__device__ __forceinline__ unsigned long long *gacc_of(const Scalars &sc) {
    return sc.gacc + (size_t)(blockIdx.x & (kGCopies - 1)) * kAccWords;
}
__device__ __forceinline__ unsigned long long *acc2_of(const Scalars &sc, int tg) {
    return sc.acc2 + ((size_t)tg * kTCopies + (blockIdx.x & (kTCopies - 1))) * kAccWords;
}

// The fp64 squares of a default-mode tile's tail: the up to three lanes that hold an element each
// add it themselves, exactly, so that no warp-wide fp64 tree is needed.
__device__ __forceinline__ void add_tail(const Scalars &sc, int tg, const double (&accd)[kAcc]) {
    if (accd[0] == 0.0 && accd[1] == 0.0 && accd[2] == 0.0) return;  // (a NaN goes on)
#pragma unroll 1
    for (int a = 0; a < kAcc; ++a) {
        const double d = a == 0 ? accd[0] : a == 1 ? accd[1] : accd[2];
        acc_add_f64(acc1_of(sc, tg, a), d);
        if (a == 0 && sc.mode == kModeStep) acc_add_f64(gacc_of(sc), d);
    }
}
// The most that the limbs of add_shifted, at bits r, r + 26 and r + 52 of a word, add to any one
// word between them.
constexpr unsigned long long limbs_max_add() {
    unsigned long long most = 0;
    for (int r = 0; r < 32; ++r) {
        unsigned long long word[5] = {};
        for (int i = 0; i < 3; ++i) {
            const unsigned long long limb = 32ull * ((i == 2 ? 1ull << 27 : 1ull << 26) - 1ull);
            const int at = r + 26 * i, w = at >> 5, b = at & 31;
            const unsigned long long low = limb << b, top = (1ull << 32) - (1ull << b);
            word[w] += low < top ? low : top;
            word[w + 1] += low >> 32;
        }
        for (unsigned long long x : word) most = x > most ? x : most;
    }
    return most;
}
static_assert(limbs_max_add() <= 2ull << 32, "a shifted tile adds to a word as two partials do");

// The lanes' fp64 sums d[0 .. R) (>= 0, finite or not) of a shifted tile into R accumulators, and
// the first one into `also` as well (unless NULL).  An fp64 tree across the warp takes 4000 cycles
// of a tile's 13,000 on GB300's slow FP64 pipe, so the lanes are added as integers: relative to the
// warp's largest exponent a sum is a fixed-point number of 79 bits, limbs of 26, 26 and 27, and
// each limb's warp total (below 2^32) takes one instruction.  What lies below 2^-78 of the largest
// sum is cut off, less than an fp64 addition's own rounding.  The totals are exact integers and go
// to the accumulators by a lane each (the lowest limb is zero where its weight lies below the
// accumulators' 2^-352: squares of fp32 numbers are multiples of 2^-298).
template <int R>
__device__ __noinline__ void add_shifted(const double (&d)[R], unsigned long long *const (&A)[R],
                                         unsigned long long *also) {
    const int lane = threadIdx.x & 31;
    unsigned sum = 0u;  // lane 3 r + i: limb i of sum r; lanes 3 R + i: of sum 0, for `also`
    int ex = 0;
    unsigned long long *to = nullptr;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(d[r]);
        const int e = (int)(u >> 52) & 0x7ff;
        const int top = __reduce_max_sync(kFull, e);
        if (top == 0x7ff) {  // an inf or a NaN: its lanes flag it, and nothing else counts
            if (e == 0x7ff) {
                acc_add_f64(A[r], d[r]);
                if (r == 0 && also) acc_add_f64(also, d[r]);
            }
            continue;
        }
        // e == 0: zero (a square of an fp32 number is far above fp64's subnormal range)
        const unsigned long long m = e ? (u & 0xfffffffffffffull) | (1ull << 52) : 0ull;
        const int shift = top - e;
        // Bits 78 .. 26: m >> shift; bits 25 .. 0: the first 26 of those that cuts off.
        const unsigned long long hi = shift < 64 ? m >> shift : 0ull;
        const unsigned long long cut = shift == 0    ? 0ull
                                       : shift < 64  ? m << (64 - shift)
                                       : shift < 128 ? m >> (shift - 64)
                                                     : 0ull;
        const unsigned low = (unsigned)(cut >> 38);
        const unsigned l0 = __reduce_add_sync(kFull, low);
        const unsigned l1 = __reduce_add_sync(kFull, (unsigned)(hi & 0x3ffffffull));
        const unsigned l2 = __reduce_add_sync(kFull, (unsigned)(hi >> 26));
        const int i = lane - 3 * r, j = lane - 3 * R;
        if ((i >= 0 && i < 3) || (r == 0 && also && j >= 0 && j < 3)) {
            const int limb = i >= 0 && i < 3 ? i : j;
            sum = limb == 0 ? l0 : limb == 1 ? l1 : l2;
            ex = top - 1075 - 26 + 26 * limb;
            to = i >= 0 && i < 3 ? A[r] : also;
        }
    }
    if (to) acc_add(to, sum, ex);
}

template <int KT, bool WM, bool RW, bool SS, bool PR, bool SH, bool Small>
__global__ void __launch_bounds__(Ring1Of<KT, RW, SH>::kThreads, 1)
    k_reduce(const __grid_constant__ TableOf<Small> tab, const __grid_constant__ Scalars sc) {
    extern __shared__ __align__(128) unsigned char smem[];
    // The first launch of a pass reads and writes nothing before its wait: the kernel ahead of it
    // may be the caller's own, still writing the gradients, and may have let its dependents start.
    // Until then it sets up its barriers, finds its first tiles in the table and has L2 fetch them,
    // which puts no value into the kernel (ResNet-18, K = 4: 70.7 us a step, 71.6 without).  The
    // next kernel may start when that wait has passed; a later launch of the pass (more tensors than
    // one parameter block holds) therefore finds all but its predecessor in the pass complete.  It
    // shares no tensor with that one, and takes the other of two tile counters, so it only has to
    // complete after it: its warps wait once their first tile is done.
    const bool first = tab.seq == 0;
    const int lane = threadIdx.x & 31;
    const int K = KT > 0 ? KT : sc.K;
    const int chunk = tab.chunk;
    // Stage streams: replicas 0 .. K - 1, then w (RW), then g_small (SS).
    const int ns = K + (RW ? 1 : 0) + (SS ? 1 : 0);
    const int role = lane < ns ? lane : 0;
    Stream<Ring1Of<KT, RW, SH>, SH> st;
    int c = st.start(smem, tab.nc, sc.tiles + 2 * (tab.seq & 1), sc);
    TilePos q = {};
    if (RW && sc.keep_w && lane == K) st.hint = false;
    if (first) {
        if (c >= 0) st.prefetch(tab, c, chunk, role, ns);
        grid_wait();
        grid_launch_dependents();
    }
    st.forget_l1();
    if (c >= 0) q = st.issue(tab, c, chunk, role, ns);
    st.claim();
    bool to_wait = !first;
    const bool step_g2 = sc.mode == kModeStep;  // |gbar|^2 also goes into |G|^2
    // The partial sums of a batch of kPend tiles are reduced across the warp together
    // (reduce-scatter, kRS values with padding) and added into the accumulators by the lanes
    // that own them.
    constexpr int kRS = 16;
    static_assert(kPend * kAcc <= kRS, "one reduce-scatter per batch");
    while (c >= 0) {
        // PR: the lanes' fp64 sums.  Default: fp32 sums of the shared-memory columns, scaled by
        // 2^(2e) with e coded in two bits per value in `ecode` (same in every lane); a tail's fp64
        // squares, and a shifted tile's sums, are added at once instead.
        double pendd[PR ? kRS : 1];
        float pendf[PR ? 1 : kRS];
        unsigned ecode = 0u;
        int ptensor[kPend];  // global index of each pending tile's tensor, -1: none
#pragma unroll
        for (int i = 0; i < kRS; ++i) {
            if constexpr (PR) pendd[i] = 0.0;
            else pendf[i] = 0.f;
        }
#pragma unroll
        for (int p = 0; p < kPend; ++p) ptensor[p] = -1;
        // One copy of the tile's code for the whole batch: the sums go to their places by
        // predicated moves.
#pragma unroll 1
        for (int p = 0; p < kPend && c >= 0; ++p) {
            if (!st.arrived(sc)) {
                c = -1;
                break;
            }
            const Row<TableOf<Small>> ptr{tab, q.t};
            double accd[kAcc];
            float accf[kAcc];
            unsigned tcode;
            bool tile_tail;
            reduce_tile<KT, WM, RW, SS, PR, SH>(st.stage, chunk, ptr, st.tc.stream(0), q, st.tc.nv,
                                                st.tc.aligned, sc, accd, accf, tcode, tile_tail);
            __syncwarp();
            const int tg = q.tg;
            const bool shifted = SH && !st.tc.aligned;
            c = st.next();
            if (c >= 0) {
                q = st.issue(tab, c, chunk, role, ns);
                st.claim();
            }
            if (to_wait) {
                grid_wait();
                grid_launch_dependents();
                to_wait = false;
            }
            if constexpr (!PR) {
                if (tile_tail) {
                    if (SH && shifted) {
                        unsigned long long *const A[kAcc] = {acc1_of(sc, tg, 0), acc1_of(sc, tg, 1),
                                                             acc1_of(sc, tg, 2)};
                        add_shifted<kAcc>(accd, A, step_g2 ? gacc_of(sc) : nullptr);
                        continue;
                    }
                    add_tail(sc, tg, accd);
                }
            }
#pragma unroll
            for (int i = 0; i < kPend; ++i) {
                if (p == i) {
                    ptensor[i] = tg;
#pragma unroll
                    for (int a = 0; a < kAcc; ++a) {
                        if constexpr (PR) pendd[i * kAcc + a] = accd[a];
                        else pendf[i * kAcc + a] = accf[a];
                    }
                }
            }
            if constexpr (!PR) ecode |= tcode << (2 * kAcc * p);
        }
        int idx;
        double vd = 0.0;
        float vf = 0.f;
        if constexpr (PR) vd = warp_reduce_scatter<kRS>(pendd, idx);
        else vf = warp_reduce_scatter<kRS>(pendf, idx);
        // lanes 2i hold value i = p * kAcc + a of the batch
        if ((lane & 1) == 0 && idx < kPend * kAcc) {
            const int p = idx / kAcc, a = idx - p * kAcc;
            const int tg = p == 0 ? ptensor[0] : p == 1 ? ptensor[1] : p == 2 ? ptensor[2] : ptensor[3];
            if (tg >= 0) {
                unsigned long long *A = acc1_of(sc, tg, a);
                if constexpr (PR) {
                    acc_add_f64(A, vd);
                    if (a == 0 && step_g2) acc_add_f64(gacc_of(sc), vd);
                } else {
                    const int k = -2 * scale_exp((ecode >> (2 * idx)) & 3u);
                    acc_add_f32(A, vf, k);
                    if (a == 0 && step_g2) acc_add_f32(gacc_of(sc), vf, k);
                }
            }
        }
    }
    if (to_wait) grid_wait();
}

// ----------------------------------------------------------------------------
// k_finish: per-tensor results from the exact accumulators
// ----------------------------------------------------------------------------
//
// One warp per tensor reads its accumulators (one word per lane), rounds them to fp64
// (acc_to_double), puts them back to zero for the next call and writes the tensor's results: the
// last kernel of a step (statistics, UpdateGradScale), of tula_layer_stats and of a per-tensor
// tula_ags_update_scale.  In a step, one more warp forms |G|^2 from the global accumulator, then
// Delta (Eq. 5) and the branch of Algorithm 1 for the step record; the update has taken the same
// branch from the same accumulator (step_branch).  No warp waits for another.
//
// Between the passes it would keep the update waiting: 9.9 us from the end of the reduction to the
// update's first tile on ResNet-50, 3.7 of them the record's fp64 division.  Only LARS, whose
// coefficients are ratios of this step's norms, has a kernel there (k_lars).

// The square roots of three norms (lanes 0-2 in one fp64 sequence) and the two ratios of a
// tensor (lanes 0 and 1): UpdateGradScale's |g_s| / (|g_l| + eps) and |w| / |gbar| (LARS, the
// statistics).  GB300's FP64 pipe is slow, so the lanes share its latency instead of queueing
// behind it.  Called by the whole warp; every lane gets every result.
struct Norms {
    double ng, ns, nw, q_scale, q_w;
};
__device__ __forceinline__ Norms tensor_norms(const Scalars &sc, double sg, double ss, double sw) {
    const int lane = threadIdx.x & 31;
    const double r = sqrt(lane == 0 ? sg : (lane == 1 ? ss : sw));
    Norms o;
    o.ng = __shfl_sync(kFull, r, 0);
    o.ns = __shfl_sync(kFull, r, 1);
    o.nw = __shfl_sync(kFull, r, 2);
    const double q = (lane == 0 ? o.ns : o.nw) / (lane == 0 ? o.ng + (double)sc.eps : o.ng);
    o.q_scale = __shfl_sync(kFull, q, 0);
    o.q_w = __shfl_sync(kFull, q, 1);
    return o;
}

// Delta (Eq. 5): this step's |G|^2 against the last step's, +inf at the first step (no previous
// norm; the step is then unscaled, the sensitive phase).
__device__ __forceinline__ double variability(double g2, double g2_prev, double steps) {
    return steps == 0.0 ? (double)INFINITY : fabs((g2 - g2_prev) / g2_prev);
}
// The branch of Algorithm 1: scaled iff Delta < delta, unless forced.
__device__ __forceinline__ int branch_of(const Scalars &sc, double dv) {
    if (sc.force == TULA_BRANCH_SCALED) return 1;
    if (sc.force == TULA_BRANCH_UNSCALED) return 0;
    return dv < (double)sc.delta;
}
// The same branch without waiting for Eq. 5's fp64 division (1.8-3.7 us on GB300) unless it is
// close: with d = |g2 - g2_prev| as rounded and t = fl(delta * g2_prev), both far from underflow,
// d < t (1 - 2^-49) puts the exact quotient d / g2_prev below delta (1 - 2^-50) (t and the product
// err by 2^-53 each), so its rounding is below delta, and d > t (1 + 2^-49) puts it above.  NaN,
// infinite and zero norms fail both tests and divide.
__device__ __forceinline__ int branch_from(const Scalars &sc, double g2, double g2_prev,
                                           double steps) {
    if (sc.force == TULA_BRANCH_AUTO && steps != 0.0) {
        const double t = __dmul_rn((double)sc.delta, g2_prev);
        const double d = fabs(__dsub_rn(g2, g2_prev));
        if (t > 0x1p-900 && t < 0x1p900) {
            if (d < __dmul_rn(t, 1.0 - 0x1p-49)) return 1;
            if (d > __dmul_rn(t, 1.0 + 0x1p-49) && d < 0x1p1000) return 0;
        }
    }
    return branch_of(sc, variability(g2, g2_prev, steps));
}
// The step record from this step's |G|^2 (one lane).
__device__ void finalize_step(const Scalars &sc, double g2, double g2_prev, double steps) {
    const double dv = variability(g2, g2_prev, steps);
    const int scaled = branch_of(sc, dv);
    sc.state[TULA_STATE_G2_PREV] = g2;
    sc.state[TULA_STATE_STEPS] = steps + 1.0;
    sc.state[TULA_STATE_DELTA] = dv;
    sc.state[TULA_STATE_SCALED] = (double)scaled;
}

// This lane's word of the sum of R accumulators' Copies copies each (A[r] the first copy of
// accumulator r): digits and carries added, the flags or-ed.  Every load is issued before the
// first sum (one round trip); with `rearm`, the copies are put back to zero.
template <int R, int Copies>
__device__ __forceinline__ void acc_words(unsigned long long *const (&A)[R], bool rearm,
                                          unsigned long long (&w)[R]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < R; ++r) w[r] = 0ull;
    if (lane >= kAccWords) return;
    unsigned long long x[R][Copies];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < Copies; ++c) x[r][c] = __ldcg(A[r] + c * kAccWords + lane);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < Copies; ++c) w[r] = lane == kAccFlags ? (w[r] | x[r][c]) : (w[r] + x[r][c]);
    if (rearm) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < Copies; ++c) A[r][c * kAccWords + lane] = 0ull;
    }
}
// One accumulator's value (its copies summed), rounded to fp64 by the whole warp.
template <int Copies>
__device__ __forceinline__ double acc_read(unsigned long long *A, bool rearm) {
    unsigned long long *const a[1] = {A};
    unsigned long long w[1];
    acc_words<1, Copies>(a, rearm, w);
    double v[1];
    acc_to_double<1>(w, v);
    return v[0];
}

// A sharded step's share of |G|^2 (TULA_G2_SHARE_WORDS words): words 0 .. kAccDigits - 1 are the
// digits of the global accumulator with its copies added, word kAccDigits counts inf partials
// and the next one NaN partials, the rest are 0.  Every word adds as an integer, so the ranks'
// shares combine by any integer sum, in any order, to the share of the whole step.
static_assert(kAccDigits + 2 <= kAccWords && TULA_G2_SHARE_WORDS == kAccWords, "share layout");
__device__ __forceinline__ double share_to_double(const unsigned long long *share) {
    const int lane = threadIdx.x & 31;
    unsigned long long w = lane < kAccWords ? __ldcg(share + lane) : 0ull;
    const unsigned long long n_inf = __shfl_sync(kFull, w, kAccDigits);
    const unsigned long long n_nan = __shfl_sync(kFull, w, kAccDigits + 1);
    if (lane == kAccFlags) w = (n_nan ? 2ull : 0ull) | (n_inf ? 1ull : 0ull);
    else if (lane >= kAccDigits) w = 0ull;
    unsigned long long wi[1] = {w};
    double v[1];
    acc_to_double<1>(wi, v);
    return v[0];
}

// Pass 1 of a sharded step, after the reduction: this rank's share of |G|^2 out of the global
// accumulator, which is re-armed, as the reduction's tile counters are: the update may never come
// (a step dropped for its |G|^2).  One warp.
__global__ void __launch_bounds__(32) k_share(const __grid_constant__ Scalars sc,
                                              unsigned long long *share) {
    grid_wait();
    const int lane = threadIdx.x & 31;
    if (lane < 2) sc.tiles[2 * lane] = 0u;
    unsigned long long *const a[1] = {sc.gacc};
    unsigned long long w[1];
    acc_words<1, kGCopies>(a, true, w);
    const unsigned long long flags = __shfl_sync(kFull, w[0], kAccFlags);
    if (lane < kAccDigits) share[lane] = w[0];
    else if (lane == kAccDigits) share[lane] = (flags & 1ull) ? 1ull : 0ull;
    else if (lane == kAccDigits + 1) share[lane] = (flags & 2ull) ? 1ull : 0ull;
    else if (lane < kAccWords) share[lane] = 0ull;
}

// The step's |G|^2, by the whole warp: from the ranks' shares in a sharded step.
__device__ __forceinline__ double step_g2_of(const Scalars &sc, bool rearm) {
    return sc.g2ext ? share_to_double(sc.g2ext) : acc_read<kGCopies>(sc.gacc, rearm);
}
// The branch of this step for the update, by one warp, once the reduction has completed.
__device__ __forceinline__ int step_branch(const Scalars &sc) {
    const double g2_prev = __ldcg(sc.state + TULA_STATE_G2_PREV);
    const double steps = __ldcg(sc.state + TULA_STATE_STEPS);
    return branch_from(sc, step_g2_of(sc, false), g2_prev, steps);
}

// LARS (Sec. V-B), between the passes: c_p = trust * |w| / |gbar|, every step (1 when either norm
// is 0).  One warp per tensor; the accumulators stay as they are for k_finish.
__global__ void __launch_bounds__(32 * kFinWarps) k_lars(const __grid_constant__ Scalars sc) {
    const int lane = threadIdx.x & 31;
    const int t = (int)blockIdx.x * kFinWarps + (int)(threadIdx.x >> 5);
    grid_launch_dependents();  // the update's first w and m (see k_update)
    grid_wait();
    if (t >= sc.n_total) return;
    unsigned long long *A = sc.acc1 + (size_t)t * kAcc * kTCopies * kAccWords;
    unsigned long long *const a[2] = {A, A + 2 * kTCopies * kAccWords};
    unsigned long long w[2];
    acc_words<2, kTCopies>(a, false, w);
    double v[2];
    acc_to_double<2>(w, v);
    const Norms o = tensor_norms(sc, v[0], 0.0, v[1]);
    if (lane == 0)
        sc.cand[t] = (v[1] > 0.0 && v[0] > 0.0) ? (float)((double)sc.lars_trust * o.q_w) : 1.0f;
}

__global__ void __launch_bounds__(32 * kFinWarps) k_finish(const __grid_constant__ Scalars sc) {
    const int lane = threadIdx.x & 31;
    const int t = (int)blockIdx.x * kFinWarps + (int)(threadIdx.x >> 5);
    const int n = sc.n_total;
    const bool step = sc.mode == kModeStep;
    grid_wait();
    // The next call's first kernel may start now; it reads and writes nothing before its own wait.
    grid_launch_dependents();
    if (t == 0 && lane == 0) {
        const int pass = step ? 1 : 0;
        sc.tiles[pass] = sc.tiles[2 + pass] = 0u;
    }
    if (t > n || (t == n && !step)) return;
    if (t == n) {  // the step record
        const double g2_prev = sc.state[TULA_STATE_G2_PREV], steps = sc.state[TULA_STATE_STEPS];
        const double g2 = step_g2_of(sc, true);
        if (lane == 0) finalize_step(sc, g2, g2_prev, steps);
        return;
    }
    unsigned long long *A1 = sc.acc1 + (size_t)t * kAcc * kTCopies * kAccWords;
    unsigned long long *A2 = sc.acc2 + (size_t)t * kTCopies * kAccWords;
    // |w|^2 before the update comes from pass 1 when that read w, else from the update's own tiles.
    const bool have_sw2 = step && sc.stats && !sc.read_w;
    const float old = (step && sc.scale) ? sc.scale[t] : 0.0f;
    unsigned long long *const a[kAcc] = {A1, A1 + kTCopies * kAccWords,
                                         have_sw2 ? A2 : A1 + 2 * kTCopies * kAccWords};
    unsigned long long w[kAcc];
    acc_words<kAcc, kTCopies>(a, true, w);
    if (step && !sc.stats && !sc.refresh) return;  // re-armed, and nobody asks for the norms
    double v[kAcc];
    acc_to_double<kAcc>(w, v);
    const double sg = v[0], ss = v[1], sw = v[2];
    const Norms o = tensor_norms(sc, sg, ss, sw);
    if (lane != 0) return;
    float s_after = old;
    if (sc.mode == kModeScale || (step && sc.refresh && sc.scale)) {
        // UpdateGradScale: min(|g_small| / (|g_large| + eps), s_max); in a step g_small is replica
        // 0 and g_large the mean
        s_after = (float)fmin(o.q_scale, (double)sc.s_max);
        sc.scale[t] = s_after;
    }
    if (sc.stats) {
        double *row = sc.stats + (size_t)t * TULA_STATS_LEN;
        row[TULA_STAT_W_SQ] = sw;
        row[TULA_STAT_G_SQ] = sg;
        row[TULA_STAT_G0_SQ] = ss;
        row[TULA_STAT_W_NORM] = o.nw;
        row[TULA_STAT_G_NORM] = o.ng;
        row[TULA_STAT_RATIO] = sg > 0.0 ? o.q_w : 0.0;
        if (!step) row[TULA_STAT_COEF] = 0.0;  // a step's update has written its coefficient
        row[TULA_STAT_SCALE] = (double)s_after;
    }
}

// ----------------------------------------------------------------------------
// Pass 2: scaled momentum-SGD + weight-decay update (Eq. 7b, Algorithm 1)
// ----------------------------------------------------------------------------
// Pointer roles: 0 = gbar, 1 = w, then m (HM), then the per-element gradscale (PE).
// Stage streams: gbar, w, then m (HM), then the per-element scale (PE, scaled).

// The step's scalars by value: an out-of-line function that stores through float pointers would
// have to load them again after every store (the shifted update's tiles took 7000 cycles, and
// 5100 so).
struct Sgd {
    float lr, mu, wd;
};
__device__ __forceinline__ Sgd sgd_of(const Scalars &sc) { return {sc.lr, sc.mu, sc.wd}; }
__device__ __forceinline__ void sgd1(float g, float c, float &w, float &m, const Sgd &sc,
                                     bool has_m) {
    const float gt = __fmul_rn(c, g);
    const float d = __fadd_rn(gt, __fmul_rn(sc.wd, w));
    if (has_m) {
        m = __fadd_rn(__fmul_rn(sc.mu, m), d);
        w = __fsub_rn(w, __fmul_rn(sc.lr, m));
    } else {
        w = __fsub_rn(w, __fmul_rn(sc.lr, d));
    }
}

// One float4 column of the update; returns the squares of w (before the update).
template <bool HM>
__device__ __forceinline__ float update4(float4 g4, float4 w4, float4 m4, float4 cc, float *wp,
                                         float *mp, const Scalars &sc, float pw) {
    pw = sq4(pw, w4);
    sgd1(g4.x, cc.x, w4.x, m4.x, sgd_of(sc), HM);
    sgd1(g4.y, cc.y, w4.y, m4.y, sgd_of(sc), HM);
    sgd1(g4.z, cc.z, w4.z, m4.z, sgd_of(sc), HM);
    sgd1(g4.w, cc.w, w4.w, m4.w, sgd_of(sc), HM);
    st_stream(wp, w4);
    if (HM) st_stream(mp, m4);
    return pw;
}

// |w|^2 of a tile's shared-memory w columns in fp32, every element multiplied by the power of
// two f first (sq_range_exp): the statistics' fallback when the tile's fp32 sums would overflow
// or lose their precision to underflow.  Out of line, like tile_cols_scaled.
__device__ __noinline__ float w_cols_scaled(uint32_t w_stage, int nv, float f) {
    float a = 0.f;
    for (int v = threadIdx.x & 31; v < nv; v += 32)
        a = sq4(a, mul4(lds4(w_stage + (uint32_t)(16 * v)), f));
    return a;
}

// A tile of a tensor off a 16-byte boundary, as tile_shifted() of pass 1: four elements per lane
// and step.  Returns the lane's |w|^2 (triples, to fp64 once) when the statistics want it.
template <bool HM, bool PE, bool SW, typename Tab>
__device__ __noinline__ double update_shifted(uint32_t stage, const Tab &tab, int t,
                                              long long begin, int n, float ct, bool use_se,
                                              const Scalars &sc) {
    constexpr uint32_t part = (uint32_t)(4 * Ring2<false>::tile_elems(2 + (HM ? 1 : 0) + (PE ? 1 : 0)) +
                                         kShiftBytes);
    const int lane = threadIdx.x & 31;
    const Row<Tab> ptr{tab, t};
    auto at = [&](int role) {
        return stage + (uint32_t)role * part + ((uint32_t)reinterpret_cast<uintptr_t>(ptr[role]) & 12u);
    };
    const uint32_t at_g = at(0), at_w = at(1), at_m = HM ? at(2) : 0u;
    const uint32_t at_c = use_se ? at(HM ? 3 : 2) : 0u;
    float *wp = ptr[1] + begin;
    float *mp = HM ? ptr[2] + begin : nullptr;
    const Sgd sgd = sgd_of(sc);
    Tw4 aw;
    tw_zero(aw);
    // One step from element j0 on; the elements past the end count as 0.
    auto step = [&](int j0, auto whole) {
        constexpr bool kWhole = decltype(whole)::value;
        float g[4], w[4], m[4], c[4];
        bool in[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            in[u] = kWhole || j0 + 32 * u < n;
            const uint32_t o = 4u * (uint32_t)(kWhole ? j0 + 32 * u : min(j0 + 32 * u, n - 1));
            g[u] = lds1(at_g + o);
            w[u] = lds1(at_w + o);
            m[u] = HM ? lds1(at_m + o) : 0.f;
            c[u] = use_se ? lds1(at_c + o) : (PE ? 1.f : ct);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (SW) tw_sq(aw, u, in[u] ? w[u] : 0.f);
            sgd1(g[u], c[u], w[u], m[u], sgd, HM);
            if (in[u]) {
                __stcs(wp + j0 + 32 * u, w[u]);
                if (HM) __stcs(mp + j0 + 32 * u, m[u]);
            }
        }
    };
    int j0 = lane;
#pragma unroll 1
    for (; j0 - lane + 128 <= n; j0 += 128) step(j0, std::true_type{});
    if (j0 - lane < n) step(j0, std::false_type{});
    __syncwarp();
    if (!SW) return 0.0;
    float high;
    double r = tw_total(aw, high);
    if (__any_sync(kFull, lane < n && !dw_lane_ok(high))) {
        r = 0.0;
        for (int j = lane; j < n; j += 32) {
            const double y = (double)lds1(at_w + 4u * (uint32_t)j);
            r = __fma_rn(y, y, r);
        }
        __syncwarp();
    }
    return r;
}

template <bool HM, bool PE, bool SW, bool SH, bool Small>
__global__ void __launch_bounds__(Ring2<SH>::kThreads, 1)
    k_update(const __grid_constant__ TableOf<Small> tab, const __grid_constant__ Scalars sc) {
    extern __shared__ __align__(128) unsigned char smem[];
    // The first launch of the pass issues m (w when there is no m, w and m of shifted tiles) of its
    // first tiles at once: it starts only when this step's reduction (and k_lars) have started,
    // which let it once every kernel before them had completed, so both are final.  The rest
    // follows when the kernel before has completed.  (w and m together: ResNet-18 73.9 us instead
    // of 73.3, as the branch's reads queue behind them; neither: 74.5.)
    // The whole CTA waits per element (the stream count depends on the branch) and in a sharded
    // step (whatever ran between its two calls).  The next kernel may start when that wait has
    // passed: the next step's reduction reads the mean this step's has written.  A later launch of
    // the pass only has to complete after the one before, as in k_reduce; what it reads was final
    // when that one let it start, and it reads it from L2 (its own wait comes later): by TMA and
    // ld.cg, and the ends of shifted tiles through an L1 that it has given up (forget_l1).
    const bool first = tab.seq == 0;
    const bool early = !PE && first && sc.early_w;
    if (first && !early) {
        grid_wait();
        grid_launch_dependents();
    }
    // The reduction has completed: its tile counters for the next call.
    auto rearm_pass1 = [&]() {
        if (blockIdx.x == 0 && threadIdx.x == 0) sc.tiles[0] = sc.tiles[2] = 0u;
    };
    if (first && !early) rearm_pass1();
    __shared__ int branch;
    const bool gated = sc.rule == TULA_RULE_AGS || sc.rule == TULA_RULE_STATIC;
    // Called by the whole CTA after its wait: every CTA forms the branch from the accumulator for
    // itself, one warp each.
    auto take_branch = [&]() -> int {
        if (!gated) return 0;
        if (threadIdx.x < 32) {
            const int b = step_branch(sc);
            if (threadIdx.x == 0) branch = b;
        }
        __syncthreads();
        return branch;
    };
    int scaled = early ? 0 : take_branch();
    const int lane = threadIdx.x & 31;
    const int chunk = tab.chunk;
    const bool use_se = PE && scaled;
    const int ns = 2 + (HM ? 1 : 0) + (use_se ? 1 : 0);
    const int role = lane < ns ? lane : 0;
    constexpr int CH = Ring2<false>::tile_elems(2 + (HM ? 1 : 0) + (PE ? 1 : 0));
    constexpr int COLS = CH / 128;
    const uint32_t w_off = (uint32_t)(CH * 4);
    const uint32_t m_off = (uint32_t)(2 * CH * 4);
    const uint32_t se_off = (uint32_t)((HM ? 3 : 2) * CH * 4);
    constexpr int kEarlyFrom = HM && !SH ? 2 : 1;  // streams from here on are issued early
    Stream<Ring2<SH>, SH> st;
    int c = st.start(smem, tab.nc, sc.tiles + 2 * (tab.seq & 1) + 1, sc);
    TilePos q = {};
    st.forget_l1();
    if (c >= 0) q = st.issue(tab, c, chunk, role, ns, early ? kEarlyFrom : 0);
    st.claim();
    if (early) {
        grid_wait();
        grid_launch_dependents();
        st.forget_l1();  // a role's first tiles may share a sector with the mean's
        if (c >= 0) st.issue_below(q, kEarlyFrom, ns, chunk);
        rearm_pass1();
        scaled = take_branch();
    }
    bool to_wait = !first;
    const uint32_t stage = st.stage;
    // Where a tensor's coefficient comes from (per tensor): the gradscale or s when scaled, LARS's
    // ratio, else 1.
    const float *const cand_of = sc.rule == TULA_RULE_LARS ? sc.cand
                                 : (sc.rule == TULA_RULE_AGS && !PE && scaled) ? sc.scale : nullptr;
    const float c_all = sc.rule == TULA_RULE_STATIC && scaled ? sc.static_s : 1.0f;

    int cand_t = -1;
    float ct = c_all;
    while (c >= 0) {
        // fp32 |w|^2 of the tiles' shared-memory columns, scaled by 2^(2e) (e coded in `ecode`);
        // a tail's fp64 squares, and a shifted tile's sum, are added at once instead.
        float pend[kPend];
        unsigned ecode = 0u;
        int ptensor[kPend];  // global index of each pending tile's tensor, -1: none
#pragma unroll
        for (int i = 0; i < kPend; ++i) {
            ptensor[i] = -1;
            pend[i] = 0.f;
        }
#pragma unroll 1
        for (int p = 0; p < kPend && c >= 0; ++p) {
            if (q.tg != cand_t) {  // c_p changes only with the tensor
                if (cand_of) ct = __ldcg(cand_of + q.tg);
                cand_t = q.tg;
            }
            if (!st.arrived(sc)) {
                c = -1;
                break;
            }
            const Row<TableOf<Small>> ptr{tab, q.t};
            const int nv = st.tc.nv;
            if (sc.stats && q.c_in_t == 0 && lane == 0)
                sc.stats[(size_t)q.tg * TULA_STATS_LEN + TULA_STAT_COEF] =
                    PE ? (scaled ? (double)NAN : 1.0) : (double)ct;
            float *wp = st.tc.stream(1) + q.begin;
            float *mp = HM ? st.tc.stream(2) + q.begin : nullptr;
            const float4 cdef = PE ? make_float4(1.f, 1.f, 1.f, 1.f) : make_float4(ct, ct, ct, ct);
            float aw = 0.f;    // fp32 |w|^2 of the tile's columns (statistics only)
            double awt = 0.0;  // exact fp64 |w|^2 of its tail
            // The last n % 4 elements, one per lane: their loads go first, to land meanwhile (SH:
            // they are in the stage).
            const long long n = q.end - q.begin;
            const long long jj = 4 * (long long)nv + lane;
            const bool in_tail = jj < n && (!SH || st.tc.aligned);
            float g_t = 0.f, w_t = 0.f, m_t = 0.f, c_t = PE ? 1.f : ct;
            if (!SH && in_tail) {
                g_t = __ldcg(ptr[0] + q.begin + jj);
                w_t = __ldcg(wp + jj);
                if (HM) m_t = __ldcg(mp + jj);
                if (use_se) c_t = __ldcg(ptr[HM ? 3 : 2] + q.begin + jj);
            }
            if (nv == CH / 4) {
                // Two columns per step of a rolled loop (unrolled over the tile, the body
                // outgrew the instruction cache: 82.5 -> 75.5 us per ResNet-50 update pass).
#pragma unroll 1
                for (int c0 = 0; c0 < COLS; c0 += 2) {
                    float pw = 0.f;
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (c0 + u < COLS) {
                            const int v = lane + 32 * (c0 + u);
                            const float4 g4 = lds4(stage + (uint32_t)(16 * v));
                            const float4 w4 = lds4(stage + w_off + (uint32_t)(16 * v));
                            const float4 m4 = HM ? lds4(stage + m_off + (uint32_t)(16 * v)) : g4;
                            const float4 cc =
                                use_se ? lds4(stage + se_off + (uint32_t)(16 * v)) : cdef;
                            pw = update4<HM>(g4, w4, m4, cc, wp + 4 * v, mp + 4 * v, sc, pw);
                        }
                    }
                    if (SW) aw = __fadd_rn(aw, pw);
                }
            } else {
                for (int v0 = lane; v0 < nv; v0 += 32 * 4) {
                    float pw = 0.f;
                    for (int u = 0; u < 4; ++u) {
                        const int v = v0 + 32 * u;
                        if (v >= nv) break;
                        const float4 g4 = lds4(stage + (uint32_t)(16 * v));
                        const float4 w4 = lds4(stage + w_off + (uint32_t)(16 * v));
                        const float4 m4 = HM ? lds4(stage + m_off + (uint32_t)(16 * v)) : g4;
                        const float4 cc = use_se ? lds4(stage + se_off + (uint32_t)(16 * v)) : cdef;
                        pw = update4<HM>(g4, w4, m4, cc, wp + 4 * v, mp + 4 * v, sc, pw);
                    }
                    if (SW) aw = __fadd_rn(aw, pw);
                }
            }
            // The warp is converged again; nv is the same in every lane.  The stage still holds
            // the tile's w before the update.
            int ew = 0;
            if (SW && nv > 0 && !__all_sync(kFull, lane >= nv || sq_in_range(aw))) {
                ew = sq_range_exp(aw);
                if (ew) aw = w_cols_scaled(stage + w_off, nv, pow2f(ew));
            }
            if constexpr (SH) {
                if (!st.tc.aligned)
                    awt = update_shifted<HM, PE, SW>(stage, tab, q.t, q.begin,
                                                     (int)(q.end - q.begin), ct, use_se, sc);
            }
            const bool tile_tail = 4 * (long long)nv < n;  // the same in every lane
            if (in_tail) {
                if (SH) {
                    const uint32_t o = stage + 4u * (uint32_t)jj;
                    g_t = lds1(o);
                    w_t = lds1(o + w_off);
                    if (HM) m_t = lds1(o + m_off);
                    if (use_se) c_t = lds1(o + se_off);
                }
                if (SW) awt = __fma_rn((double)w_t, (double)w_t, awt);
                sgd1(g_t, c_t, w_t, m_t, sgd_of(sc), HM);
                wp[jj] = w_t;
                if (HM) mp[jj] = m_t;
            }
            __syncwarp();
            const int tg = q.tg;
            const bool shifted = SH && !st.tc.aligned;
            c = st.next();
            if (c >= 0) {
                q = st.issue(tab, c, chunk, role, ns);
                st.claim();
            }
            if (to_wait) {
                grid_wait();
                grid_launch_dependents();
                to_wait = false;
            }
            if (SW) {
                if (SH && shifted) {
                    const double d[1] = {awt};
                    unsigned long long *const A[1] = {acc2_of(sc, tg)};
                    add_shifted<1>(d, A, nullptr);
                    continue;
                }
                if (tile_tail && lane < 3) acc_add_f64(acc2_of(sc, tg), awt);  // as add_tail
#pragma unroll
                for (int i = 0; i < kPend; ++i) {
                    if (p == i) {
                        ptensor[i] = tg;
                        pend[i] = aw;
                    }
                }
                if (ew) ecode |= scale_code(ew) << (2 * p);
            }
        }
        if (SW) {
            // reduce-scatter: lanes 8p hold tile p's total
            int idx;
            const float f = warp_reduce_scatter<kPend>(pend, idx);
            if ((lane & 7) == 0) {
                const int tg = idx == 0   ? ptensor[0]
                               : idx == 1 ? ptensor[1]
                               : idx == 2 ? ptensor[2]
                                          : ptensor[3];
                if (tg >= 0)
                    acc_add_f32(acc2_of(sc, tg), f,
                                -2 * scale_exp((ecode >> (2 * idx)) & 3u));
            }
        }
    }
    if (to_wait) grid_wait();
}

// ----------------------------------------------------------------------------
// UpdateGradScale, element-wise (Algorithm 1): s = fminf(|gs / (gl + eps)|, s_max)
// ----------------------------------------------------------------------------
// A once-per-epoch call: plain 128-bit loads, one warp per tile.
// Pointer roles: 0 = g_small, 1 = g_large, 2 = s_out.

__device__ __forceinline__ float scale1(float gs, float gl, float eps, float s_max) {
    return fminf(fabsf(__fdiv_rn(gs, __fadd_rn(gl, eps))), s_max);
}

// The bounded wait itself, on an mbarrier that nothing ever arrives on: the
// wait runs out and the kernel reports it in the error word, the way every
// streaming kernel reports a stage that never fills.  (Failure detection is
// checked with this, not with a real fault.)
__global__ void __launch_bounds__(32) k_wait_check(unsigned *err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncwarp();
    if (threadIdx.x == 0 && !mbar_wait(&bar, 0u)) atomicOr(err, 1u);
}

// The elements from j0 on, one per lane: a tensor off a 16-byte boundary, or a tail.  Eight rows of
// 32 elements per step, every load issued before the first store (the output may not be assumed
// distinct, so the compiler would keep them in turn).  Out of line: inside, its registers cost the
// kernel CTAs per SM (ResNet-50: 57.5 us a call instead of 50.5).
__device__ __noinline__ void scale_rows(const float *a, const float *b, float *o, long long j0,
                                        long long n, float eps, float s_max) {
    for (; j0 < n; j0 += 8 * 32) {
        float x[8], y[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const long long j = j0 + 32 * u;
            if (j < n) {
                x[u] = __ldcs(a + j);
                y[u] = __ldcs(b + j);
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const long long j = j0 + 32 * u;
            if (j < n) o[j] = scale1(x[u], y[u], eps, s_max);
        }
    }
}

constexpr int kScaleThreads = 128;

template <bool Small>
__global__ void __launch_bounds__(kScaleThreads, 7)  // 73 registers: 28 warps an SM
    k_scale_elem(const __grid_constant__ TableOf<Small> tab, const __grid_constant__ Scalars sc) {
    grid_wait();  // no early start for the successor: it may overwrite what this kernel reads
    const int lane = threadIdx.x & 31;
    const int warp = (int)((blockIdx.x * (unsigned)kScaleThreads + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * (unsigned)kScaleThreads) >> 5);
    Walker walk;
    for (int c = warp; c < tab.nc; c += nwarps) {
        const TilePos q = locate(tab, c, walk.to(tab, c), tab.chunk);
        const Row<TableOf<Small>> ptr{tab, q.t};
        const int nv = tile_vecs(lane < 3 ? ptr[lane] : nullptr, 3, q);
        const float *a = ptr[0] + q.begin;
        const float *b = ptr[1] + q.begin;
        float *o = ptr[2] + q.begin;
        // Four float4 columns of each input per lane per step: eight 16-byte loads in flight
        // per lane, which a plain-load streaming kernel needs to cover HBM latency.
        for (int v0 = lane; v0 < nv; v0 += 4 * 32) {
            float4 x[4], y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int v = v0 + 32 * u;
                if (v < nv) {
                    x[u] = __ldcs(reinterpret_cast<const float4 *>(a) + v);
                    y[u] = __ldcs(reinterpret_cast<const float4 *>(b) + v);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int v = v0 + 32 * u;
                if (v < nv)
                    st_stream(o + 4 * v, make_float4(scale1(x[u].x, y[u].x, sc.eps, sc.s_max),
                                                     scale1(x[u].y, y[u].y, sc.eps, sc.s_max),
                                                     scale1(x[u].z, y[u].z, sc.eps, sc.s_max),
                                                     scale1(x[u].w, y[u].w, sc.eps, sc.s_max)));
            }
        }
        const long long n = q.end - q.begin;
        if (4 * (long long)nv < n) scale_rows(a, b, o, 4 * (long long)nv + lane, n, sc.eps, sc.s_max);
    }
}

// ----------------------------------------------------------------------------
// Host side
// ----------------------------------------------------------------------------

std::atomic<uint64_t> g_launches{0};
thread_local int g_last_cuda = 0;

inline long long tiles_of(int64_t n, int chunk) { return n <= 0 ? 1 : (n + chunk - 1) / chunk; }

// Tile sizes: the smallest a pass can use for K replicas sizes the workspace.
inline int chunk1(int K, bool rw, bool ss) {
    const int streams = K + (rw ? 1 : 0) + (ss ? 1 : 0);
    return rw ? Ring1W<0, false>::tile_elems(streams) : Ring1<false>::tile_elems(streams);
}
inline int chunk2(bool hm, bool pe) { return Ring2<false>::tile_elems(2 + (hm ? 1 : 0) + (pe ? 1 : 0)); }
// No pass-1 tile is smaller: K (+1 with g_small) streams in 36 KB, or K + 1 in 45 KB.
inline int chunk1_min(int K) { return Ring1<false>::tile_elems(K + 1 + (K == 1 ? 1 : 0)); }
inline int chunk2_min() { return chunk2(true, true); }

struct Plan {
    long long c1 = 0, c2 = 0;  // tiles of each pass (at the smallest tile sizes)
};

// Workspace layout.  Every counter and accumulator precedes `spare`, so zeroing [0, spare) clears
// all of them; the error word is the only one no call clears.  `flags` and `spare` hold nothing any
// more; they stay so that workspace sizes, and the longest list the static scratch takes, are what
// callers know.
struct WsLayout {
    size_t flags, err, tiles, acc1, gacc, acc2, spare, cand, total;
};

WsLayout ws_layout(int n_tensors, const Plan &) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = (off + bytes + 255) & ~size_t(255);
        return o;
    };
    const size_t acc = sizeof(unsigned long long) * kAccWords;
    WsLayout L;
    L.flags = take(sizeof(int) * 4);
    L.err = take(sizeof(unsigned) * 4);
    L.tiles = take(sizeof(unsigned) * 8);
    L.acc1 = take(acc * kAcc * kTCopies * (size_t)n_tensors);
    L.gacc = take(acc * kGCopies);
    L.acc2 = take(acc * kTCopies * (size_t)n_tensors);
    L.spare = take(kSpare * (size_t)n_tensors);
    L.cand = take(sizeof(float) * (size_t)n_tensors);
    L.total = off;
    return L;
}

// The tile index of either pass must fit an int; and the tiles and the tensors of n % 4 != 0
// elements together number at most 2^31, which keeps every accumulator word below 2^64.
bool valid_numels(const int64_t *numels, int n, int K, Plan *pl) {
    if (!numels || n < 1 || K < 1 || K > TULA_MAX_K) return false;
    const int t1 = chunk1_min(K), t2 = chunk2_min();
    Plan p;
    long long tails = 0;
    for (int i = 0; i < n; ++i) {
        if (numels[i] < 0) return false;
        p.c1 += tiles_of(numels[i], t1);
        p.c2 += tiles_of(numels[i], t2);
        tails += (numels[i] & 3) != 0;
        if (p.c1 >= (1LL << 31) || p.c2 >= (1LL << 31)) return false;
        if (std::max(p.c1, p.c2) + tails > (1LL << 31)) return false;
    }
    *pl = p;
    return true;
}

inline bool aligned4(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

// One wave of resident CTAs of `kernel` on the current device (cached); sets
// the kernel's dynamic shared memory limit on first use.
int resident_ctas(const void *kernel, int threads, int smem) {
    struct Entry { const void *k; int dev; int ctas; };
    static std::mutex mu;
    static std::vector<Entry> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    for (const Entry &e : cache)
        if (e.k == kernel && e.dev == dev) return e.ctas;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess)
        return 0;
    int sms = 0, per = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess)
        return 0;
    const int ctas = std::max(1, sms * std::max(per, 1));
    cache.push_back({kernel, dev, ctas});
    return ctas;
}

// L2 capacity of the current device in bytes (cached; 0 if unknown).
long long l2_bytes() {
    static std::mutex mu;
    static std::vector<std::pair<int, long long>> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    for (const auto &e : cache)
        if (e.first == dev) return e.second;
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, dev) != cudaSuccess) v = 0;
    cache.emplace_back(dev, (long long)v);
    return v;
}

// Launch with programmatic stream serialization: the kernel may begin while
// the previous kernel in the stream finishes; its griddepcontrol.wait orders
// what follows after that kernel's completion (what k_update and the later
// launches of a pass read before theirs is said there).
template <typename... KArgs, typename... Args>
int launch_pdl(void (*kernel)(KArgs...), int grid, int threads, int smem, cudaStream_t s,
               Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    return TULA_OK;
}

// The launch tables of a plan (tula_ags_plan_create): for each kernel instantiation and tile
// size, its parameter blocks, built by the first call that launches them and reused by every
// later one (they hold only sizes and pointers, which a plan fixes).
struct Blocks {
    bool small = false;  // TableOf<true>: one launch of few, aligned tensors
    std::vector<std::shared_ptr<const void>> tabs;
};
struct TableCache {
    struct Entry {
        const void *kernel;  // its instantiation for full blocks
        int chunk;
        Blocks blocks;
    };
    std::vector<Entry> entries;
    const Blocks *find(const void *kernel, int chunk) const {
        for (const Entry &e : entries)
            if (e.kernel == kernel && e.chunk == chunk) return &e.blocks;
        return nullptr;
    }
};

// What the tables of tensors [0, n) need: each role's lowest pointer, whether all of its pointers
// lie within 16 GB of that, and whether some non-empty tensor has a pointer off a 16-byte boundary.
// fill(p, ptrs) writes tensor p's np pointers.
struct Pointers {
    unsigned long long base[kMaxRoles] = {};
    bool wide = false, shifted = false;
};
template <typename Fill>
Pointers scan_pointers(int n, const int64_t *numels, int np, Fill fill) {
    Pointers r;
    unsigned long long low[kMaxRoles], high[kMaxRoles];
    for (int i = 0; i < np; ++i) {
        low[i] = ~0ull;
        high[i] = 0ull;
    }
    const float *ptr[kMaxRoles];
    for (int p = 0; p < n; ++p) {
        if (numels[p] <= 0) continue;
        fill(p, ptr);
        for (int i = 0; i < np; ++i) {
            const unsigned long long a = reinterpret_cast<uintptr_t>(ptr[i]);
            low[i] = std::min(low[i], a);
            high[i] = std::max(high[i], a);
            if (a & 15u) r.shifted = true;
        }
    }
    for (int i = 0; i < np; ++i) {
        if (low[i] > high[i]) continue;  // no non-empty tensor
        r.base[i] = low[i];
        if ((high[i] - low[i]) / 4 > 0xffffffffull) r.wide = true;
    }
    return r;
}

// Splits tensors [0, n) into parameter blocks of type Tab of tiles of `chunk` elements.
template <typename Tab, typename Fill>
void build_blocks(int n, const int64_t *numels, int chunk, int np, const Pointers &pts, Fill fill,
                  std::vector<std::shared_ptr<const void>> &tabs) {
    const float *ptr[kMaxRoles];
    for (int p = 0; p < n;) {
        int cnt = 1;
        while (p + cnt < n && Tab::bytes_for(cnt + 1, np, pts.wide) <= Tab::kRaw) ++cnt;
        std::shared_ptr<Tab> tab = std::make_shared<Tab>();
        std::memset(tab.get(), 0, sizeof(Tab));
        tab->t0 = p;
        tab->n = cnt;
        tab->chunk = chunk;
        tab->seq = (int)tabs.size();
        tab->np = np;
        tab->wide = pts.wide ? 1 : 0;
        tab->o_last = 4 * (cnt + 1);
        tab->o_lo = tab->o_last + (2 * cnt + 3) / 4 * 4;
        tab->o_hi = tab->o_lo + 4 * cnt * np;
        std::memcpy(tab->base, pts.base, sizeof(tab->base));
        int *cstart = reinterpret_cast<int *>(tab->raw);
        unsigned short *last = reinterpret_cast<unsigned short *>(tab->raw + tab->o_last);
        unsigned *lo = reinterpret_cast<unsigned *>(tab->raw + tab->o_lo);
        unsigned short *hi = reinterpret_cast<unsigned short *>(tab->raw + tab->o_hi);
        int nc = 0;
        for (int t = 0; t < cnt; ++t, ++p) {
            const long long tiles = tiles_of(numels[p], chunk);
            cstart[t] = nc;
            last[t] = (unsigned short)(numels[p] - (tiles - 1) * chunk);
            nc += (int)tiles;
            if (numels[p] <= 0) continue;  // its pointers may be NULL; nothing reads them
            fill(p, ptr);
            for (int i = 0; i < np; ++i) {
                const unsigned long long a = reinterpret_cast<uintptr_t>(ptr[i]);
                if (a & 15u) tab->shifted = 1;
                const unsigned long long e = (a - pts.base[i]) / 4;
                lo[t * np + i] = (unsigned)e;
                if (pts.wide) hi[t * np + i] = (unsigned short)(e >> 32);
            }
        }
        cstart[cnt] = nc;
        tab->nc = nc;
        while (((nc - 1) >> tab->hint_shift) >= kHints) ++tab->hint_shift;
        for (int i = 0, t = 0; i < kHints + 2; ++i) {
            while (t + 1 < cnt && ((long long)i << tab->hint_shift) >= cstart[t + 1]) ++t;
            tab->hint[i] = (unsigned short)t;
        }
        tabs.push_back(std::move(tab));
    }
}

// The instantiations of a streaming kernel: for launches whose tensors are all 16-byte aligned,
// with a small parameter block and with a full one, and for the others.
struct StreamKernels {
    void (*small)(TableOf<true>, Scalars);
    void (*full)(TableOf<false>, Scalars);
    void (*shifted)(TableOf<false>, Scalars);
    int smem, smem_shifted;
};
// base: claims made so far on the launch's tile counter.
template <typename Tab>
int launch_block(void (*fn)(Tab, Scalars), const void *block, int threads, int smem,
                 const Scalars &call, int grid_override, cudaStream_t stream, unsigned (&base)[2]) {
    const Tab &tab = *static_cast<const Tab *>(block);
    int grid = resident_ctas((const void *)fn, threads, smem);
    if (grid <= 0) {
        g_last_cuda = (int)cudaGetLastError();
        return TULA_ERR_CUDA;
    }
    if (grid_override > 0) grid = grid_override;
    grid = std::max(1, std::min(grid, tab.nc));
    Scalars sc = call;
    sc.claim_base = base[tab.seq & 1];
    if ((long long)tab.nc > (long long)grid * (threads / 32)) base[tab.seq & 1] += (unsigned)tab.nc;
    return launch_pdl(fn, grid, threads, smem, stream, tab, sc);
}
// Launches a streaming kernel once per parameter block.  With a cache, the blocks are taken from
// it, or built once and kept there.
template <typename Fill>
int launch_streaming(const StreamKernels &k, int n, const int64_t *numels, int chunk, int np,
                     int threads, const Scalars &sc, int grid_override, cudaStream_t stream,
                     Fill fill, TableCache *cache = nullptr) {
    using SmallTab = TableOf<true>;
    using FullTab = TableOf<false>;
    const Blocks *blocks = cache ? cache->find((const void *)k.full, chunk) : nullptr;
    Blocks built;
    if (!blocks) {
        const Pointers pts = scan_pointers(n, numels, np, fill);
        built.small = !pts.shifted && SmallTab::bytes_for(n, np, pts.wide) <= SmallTab::kRaw;
        try {
            if (built.small) build_blocks<SmallTab>(n, numels, chunk, np, pts, fill, built.tabs);
            else build_blocks<FullTab>(n, numels, chunk, np, pts, fill, built.tabs);
            if (cache) {
                cache->entries.push_back({(const void *)k.full, chunk, std::move(built)});
                blocks = &cache->entries.back().blocks;
            }
        } catch (const std::bad_alloc &) {
            return TULA_ERR_NO_MEMORY;
        }
        if (!blocks) blocks = &built;
    }
    unsigned base[2] = {0u, 0u};
    for (const auto &b : blocks->tabs) {
        int rc;
        if (blocks->small)
            rc = launch_block(k.small, b.get(), threads, k.smem, sc, grid_override, stream, base);
        else if (static_cast<const FullTab *>(b.get())->shifted)
            rc = launch_block(k.shifted, b.get(), threads, k.smem_shifted, sc, grid_override,
                              stream, base);
        else
            rc = launch_block(k.full, b.get(), threads, k.smem, sc, grid_override, stream, base);
        if (rc) return rc;
    }
    return TULA_OK;
}

// One warp per tensor (+ the step record's): k_lars, k_finish.
int launch_per_tensor(void (*kernel)(Scalars), int warps, const Scalars &sc, cudaStream_t s) {
    return launch_pdl(kernel, (warps + kFinWarps - 1) / kFinWarps, 32 * kFinWarps, 0, s, sc);
}
int launch_finish(int n, const Scalars &sc, cudaStream_t s) {
    return launch_per_tensor(k_finish, n + (sc.mode == kModeStep ? 1 : 0), sc, s);
}

Scalars make_scalars(const tula_ags_hparams *hp, int K, int n, void *ws, const WsLayout &L,
                     int mode) {
    Scalars sc;
    std::memset(&sc, 0, sizeof(sc));
    sc.K = K;
    sc.mode = mode;
    sc.n_total = n;
    sc.invK = 1.0f / (float)K;
    sc.Kf = (float)K;
    if (hp) {
        sc.rule = hp->rule;
        sc.force = hp->force_branch;
        sc.refresh = hp->refresh_scale;
        sc.delta = hp->delta;
        sc.eps = hp->eps;
        sc.s_max = hp->s_max;
        sc.static_s = hp->static_s;
        sc.lars_trust = hp->lars_trust;
        sc.scale = hp->scale;
        sc.state = hp->state;
        sc.stats = hp->layer_stats;
    }
    char *b = static_cast<char *>(ws);
    sc.err = reinterpret_cast<unsigned *>(b + L.err);
    sc.tiles = reinterpret_cast<unsigned *>(b + L.tiles);
    sc.acc1 = reinterpret_cast<unsigned long long *>(b + L.acc1);
    sc.gacc = reinterpret_cast<unsigned long long *>(b + L.gacc);
    sc.acc2 = reinterpret_cast<unsigned long long *>(b + L.acc2);
    sc.cand = reinterpret_cast<float *>(b + L.cand);
    return sc;
}

void record(void *ev, cudaStream_t s) {
    if (ev) cudaEventRecord(static_cast<cudaEvent_t>(ev), s);
}

// Pass 1 dispatched over the compile-time replica count.
template <int KT, bool WM, bool RW, bool SS, bool PR, typename Fill>
int run_reduce_k(int K, int n, const int64_t *numels, const Scalars &sc, int grid, cudaStream_t s,
                 Fill fill, TableCache *cache) {
    const int chunk = chunk1(K, RW, SS);
    using R = Ring1Of<KT, RW, false>;
    const StreamKernels k{k_reduce<KT, WM, RW, SS, PR, false, true>,
                          k_reduce<KT, WM, RW, SS, PR, false, false>,
                          k_reduce<KT, WM, RW, SS, PR, true, false>, R::kSmemBytes,
                          Ring1Of<KT, RW, true>::kSmemBytes};
    return launch_streaming(k, n, numels, chunk, K + (RW || SS ? 1 : 0), R::kThreads, sc, grid, s,
                            fill, cache);
}

template <bool WM, bool RW, bool SS, bool PR, typename Fill>
int run_reduce(int K, int n, const int64_t *numels, const Scalars &sc, int grid, cudaStream_t s,
               Fill fill, TableCache *cache = nullptr) {
    switch (K) {
    case 1: return run_reduce_k<1, false, RW, SS, PR>(K, n, numels, sc, grid, s, fill, cache);
    case 2: return run_reduce_k<2, WM, RW, SS, PR>(K, n, numels, sc, grid, s, fill, cache);
    case 4: return run_reduce_k<4, WM, RW, SS, PR>(K, n, numels, sc, grid, s, fill, cache);
    case 8: return run_reduce_k<8, WM, RW, SS, PR>(K, n, numels, sc, grid, s, fill, cache);
    case 16: return run_reduce_k<16, WM, RW, SS, PR>(K, n, numels, sc, grid, s, fill, cache);
    default: return run_reduce_k<0, WM, RW, SS, PR>(K, n, numels, sc, grid, s, fill, cache);
    }
}

int check_ws(void *ws, size_t bytes, int n, const Plan &pl) {
    if (!ws) return TULA_ERR_WORKSPACE;
    if (bytes < ws_layout(n, pl).total) return TULA_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return TULA_ERR_WORKSPACE;
    return TULA_OK;
}


}  // namespace

// ============================================================================
// C ABI
// ============================================================================

extern "C" {

void tula_ags_default_hparams(tula_ags_hparams *hp, int K) {
    if (!hp) return;
    std::memset(hp, 0, sizeof(*hp));
    hp->K = K;
    hp->rule = TULA_RULE_AGS;
    hp->granularity = TULA_SCALE_PER_TENSOR;
    hp->force_branch = TULA_BRANCH_AUTO;
    hp->refresh_scale = 0;
    hp->delta = 0.5f;
    hp->eps = 1e-8f;
    hp->s_max = std::sqrt((float)(K > 0 ? K : 1));
    hp->static_s = 1.0f;
    hp->lars_trust = 1.0f;
}

int tula_ags_workspace_size(const int64_t *numels, int n_tensors, int K, size_t *bytes) {
    Plan pl;
    if (!bytes || !valid_numels(numels, n_tensors, K, &pl)) return TULA_ERR_ARG;
    *bytes = ws_layout(n_tensors, pl).total;
    return TULA_OK;
}

int tula_ags_chunk_elems(int pass, int streams) {
    if (streams < 1 || streams > TULA_MAX_K + 2) return TULA_ERR_ARG;
    if (pass == 1) return Ring1<false>::tile_elems(streams);
    if (pass == 2 && streams <= 4) return Ring2<false>::tile_elems(streams);
    if (pass == 3) return Ring1W<0, false>::tile_elems(streams);
    return TULA_ERR_ARG;
}

int tula_ags_plan_chunks(const int64_t *numels, int n_tensors, int chunk_elems,
                         int64_t *chunk_start_out) {
    Plan pl;
    if (!chunk_start_out || chunk_elems < 1 || !valid_numels(numels, n_tensors, 1, &pl))
        return TULA_ERR_ARG;
    int64_t c = 0;
    for (int p = 0; p < n_tensors; ++p) {
        chunk_start_out[p] = c;
        c += tiles_of(numels[p], chunk_elems);
    }
    chunk_start_out[n_tensors] = c;
    return TULA_OK;
}

int tula_ags_check_wait_timeout(void *workspace, size_t workspace_bytes, void *stream) {
    const WsLayout L = ws_layout(1, Plan{});
    if (!workspace || workspace_bytes < L.err + sizeof(unsigned)) return TULA_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return TULA_ERR_WORKSPACE;
    unsigned *err = reinterpret_cast<unsigned *>(static_cast<char *>(workspace) + L.err);
    k_wait_check<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(err);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    return TULA_OK;
}

int tula_ags_workspace_error(const void *workspace, size_t workspace_bytes,
                             const int64_t *numels, int n_tensors, int K, int *error_out) {
    Plan pl;
    if (!workspace || !error_out || !valid_numels(numels, n_tensors, K, &pl)) return TULA_ERR_ARG;
    const WsLayout L = ws_layout(n_tensors, pl);
    if (workspace_bytes < L.total) return TULA_ERR_WORKSPACE;
    unsigned v = 0;
    unsigned *dev = reinterpret_cast<unsigned *>(static_cast<char *>(const_cast<void *>(workspace)) +
                                                 L.err);
    cudaError_t e = cudaMemcpy(&v, dev, sizeof(v), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && v) e = cudaMemset(dev, 0, sizeof(v));
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    *error_out = (int)v;
    return TULA_OK;
}

}  // extern "C"

namespace {

// The options of a step (hp apart from its workspace, and the momentum) against the buffers the
// step has: momentum buffers (has_mom) and per-element gradscales (has_se).
int check_step_options(const tula_ags_hparams *hp, float momentum, bool has_mom, bool has_se) {
    if (!hp || hp->K < 1 || hp->K > TULA_MAX_K) return TULA_ERR_ARG;
    if (hp->rule < TULA_RULE_AGS || hp->rule > TULA_RULE_STATIC) return TULA_ERR_ARG;
    if (hp->granularity != TULA_SCALE_PER_TENSOR && hp->granularity != TULA_SCALE_PER_ELEMENT)
        return TULA_ERR_ARG;
    if (hp->force_branch < TULA_BRANCH_AUTO || hp->force_branch > TULA_BRANCH_UNSCALED)
        return TULA_ERR_ARG;
    if (!hp->state) return TULA_ERR_ARG;
    const bool per_elem = hp->rule == TULA_RULE_AGS && hp->granularity == TULA_SCALE_PER_ELEMENT;
    if (hp->rule == TULA_RULE_AGS && !per_elem && !hp->scale) return TULA_ERR_ARG;
    if (per_elem && !has_se) return TULA_ERR_ARG;
    if (!has_mom && momentum != 0.0f) return TULA_ERR_ARG;
    if (hp->refresh_scale) {
        if (hp->K == 1 || !hp->scale) return TULA_ERR_ARG;
        if (hp->granularity != TULA_SCALE_PER_TENSOR) return TULA_ERR_UNSUPPORTED;
    }
    return TULA_OK;
}

// The tensors of a step: their sizes, and every pointer of a non-empty tensor non-NULL and
// 4-byte aligned (scale_elem: the per-element gradscales, or NULL when the step has none).
int check_step_tensors(float *const *param_ptrs, float *const *grad_ptrs, float *const *mom_ptrs,
                       float *const *scale_elem, const int64_t *numels, int n, int K, Plan *pl) {
    if (!param_ptrs || !grad_ptrs || !valid_numels(numels, n, K, pl)) return TULA_ERR_ARG;
    for (int p = 0; p < n; ++p) {
        if (numels[p] == 0) continue;
        if (!param_ptrs[p] || !aligned4(param_ptrs[p])) return TULA_ERR_ARG;
        if (mom_ptrs && (!mom_ptrs[p] || !aligned4(mom_ptrs[p]))) return TULA_ERR_ARG;
        if (scale_elem && (!scale_elem[p] || !aligned4(scale_elem[p]))) return TULA_ERR_ARG;
        for (int k = 0; k < K; ++k) {
            const float *g = grad_ptrs[(size_t)k * n + p];
            if (!g || !aligned4(g)) return TULA_ERR_ARG;
        }
    }
    return TULA_OK;
}

// Every host-side check of a step's arguments except the workspace: TULA_OK or the status
// tula_ags_step returns.  Nothing is enqueued before it passes.
int check_step_args(float *const *param_ptrs, float *const *grad_ptrs, float *const *mom_ptrs,
                    const int64_t *numels, int n_tensors, float momentum,
                    const tula_ags_hparams *hp, Plan *pl) {
    int rc = check_step_options(hp, momentum, mom_ptrs != nullptr, hp && hp->scale_elem);
    if (rc) return rc;
    const bool per_elem = hp->rule == TULA_RULE_AGS && hp->granularity == TULA_SCALE_PER_ELEMENT;
    return check_step_tensors(param_ptrs, grad_ptrs, mom_ptrs, per_elem ? hp->scale_elem : nullptr,
                              numels, n_tensors, hp->K, pl);
}

// Which part of a step run_step launches: all of it, or one half of a sharded step (pass 1 up to
// this rank's share of |G|^2; then, from the ranks' shares summed, the rest).
enum StepPart { kPartWhole = 0, kPartReduce = 1, kPartUpdate = 2 };

// The step's launches, once its arguments (check_step_args) and its scratch `ws` (the caller's
// workspace or the static array) have been accepted.
int run_step(float *const *param_ptrs, float *const *grad_ptrs, float *const *mom_ptrs,
             const int64_t *numels, int n, float lr, float momentum, float weight_decay,
             const tula_ags_hparams *hp, void *ws, const Plan &pl, void *stream,
             StepPart part = kPartWhole, unsigned long long *share_out = nullptr,
             const unsigned long long *g2_in = nullptr, TableCache *cache = nullptr) {
    const int K = hp->K;
    const bool per_elem = hp->rule == TULA_RULE_AGS && hp->granularity == TULA_SCALE_PER_ELEMENT;
    int rc = TULA_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const WsLayout L = ws_layout(n, pl);
    Scalars sc = make_scalars(hp, K, n, ws, L, kModeStep);
    const bool lars = hp->rule == TULA_RULE_LARS;
    sc.read_w = lars ? 1 : 0;
    // When the mean fits in L2, every bulk load is marked to leave L2 first, so
    // that the lines the step writes (the mean, w, m), which the update and the
    // next step read again, stay there instead (ResNet-18 K = 4: 103 -> 79 us per
    // step).  For larger models the mark only costs bandwidth.
    long long n_total = 0;
    for (int p = 0; p < n; ++p) n_total += numels[p];
    sc.evict_first = (K > 1 && 4 * n_total <= l2_bytes()) ? 1 : 0;
    // A LARS step's pass 1 reads w as the update will: that one stays when the mean and w fit L2
    // (ResNet-18, K = 4: 86.2 -> 83.1 us) and the step's buffers do not all fit anyway (4.3 M
    // elements, K = 2: 32.2 us with every load marked, 32.7 without w's).
    sc.keep_w = (8 * n_total <= l2_bytes() && 4 * n_total * (K + 2) > l2_bytes()) ? 1 : 0;
    sc.lr = lr;
    sc.mu = momentum;
    sc.wd = weight_decay;
    sc.early_w = part == kPartWhole ? 1 : 0;

    auto fill1 = [&](int p, const float **dst) {
        for (int k = 0; k < K; ++k) dst[k] = grad_ptrs[(size_t)k * n + p];
        dst[K] = param_ptrs[p];  // used by a pass that reads w
    };
    record(hp->trace_events[0], s);
    if (part == kPartUpdate) {
        // the ranks' shares summed give |G|^2; the local accumulators the tensors' norms
        sc.g2ext = g2_in;
    } else {
        // Norms feeding a coefficient (LARS, UpdateGradScale) are taken precisely.
        if (lars)
            rc = run_reduce<true, true, false, true>(K, n, numels, sc, hp->grid_ctas, s, fill1, cache);
        else if (hp->refresh_scale)
            rc = run_reduce<true, false, false, true>(K, n, numels, sc, hp->grid_ctas, s, fill1, cache);
        else
            rc = run_reduce<true, false, false, false>(K, n, numels, sc, hp->grid_ctas, s, fill1, cache);
        if (rc == TULA_OK && part == kPartReduce)
            return launch_pdl(k_share, 1, 32, 0, s, sc, share_out);
    }
    if (rc) return rc;
    record(hp->trace_events[1], s);
    if (lars) rc = launch_per_tensor(k_lars, n, sc, s);
    if (rc) return rc;
    record(hp->trace_events[2], s);

    auto fill2 = [&](int p, const float **dst) {
        dst[0] = grad_ptrs[p];
        dst[1] = param_ptrs[p];
        if (mom_ptrs) dst[2] = mom_ptrs[p];
        if (per_elem) dst[mom_ptrs ? 3 : 2] = hp->scale_elem[p];
    };
    const bool hm = mom_ptrs != nullptr;
    const bool sw = hp->layer_stats != nullptr && !lars;  // the update takes |w|^2
    const int c2 = chunk2(hm, per_elem);
#define TULA_UPD(HM, PE, SW)                                                                       \
    launch_streaming({k_update<HM, PE, SW, false, true>, k_update<HM, PE, SW, false, false>,  \
                            k_update<HM, PE, SW, true, false>, Ring2<false>::kSmemBytes,             \
                            Ring2<true>::kSmemBytes},                                                \
                     n, numels, c2, 2 + (HM) + (PE), Ring2<false>::kThreads, sc, hp->grid_ctas, s,  \
                     fill2, cache)
    if (hm) {
        if (per_elem) rc = sw ? TULA_UPD(true, true, true) : TULA_UPD(true, true, false);
        else rc = sw ? TULA_UPD(true, false, true) : TULA_UPD(true, false, false);
    } else {
        if (per_elem) rc = sw ? TULA_UPD(false, true, true) : TULA_UPD(false, true, false);
        else rc = sw ? TULA_UPD(false, false, true) : TULA_UPD(false, false, false);
    }
#undef TULA_UPD
    if (rc) return rc;
    record(hp->trace_events[3], s);
    rc = launch_finish(n, sc, s);
    if (rc) return rc;
    record(hp->trace_events[4], s);
    return TULA_OK;
}

}  // namespace

// A plan (tula_ags_plan_create): the step's sizes and pointer arrays, checked once, on one
// device, and the launch tables built from them by the first step of each kernel variant.
struct tula_ags_plan {
    int n = 0, K = 0, device = 0;
    Plan tiles;
    std::vector<int64_t> numels;
    std::vector<float *> params, grads, moms, scale_elem;
    TableCache tables;
};

extern "C" {

int tula_ags_step(float *const *param_ptrs, float *const *grad_ptrs, float *const *mom_ptrs,
                  const int64_t *numels, int n_tensors, float lr, float momentum,
                  float weight_decay, const tula_ags_hparams *hp, void *stream) {
    Plan pl;
    int rc = check_step_args(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, momentum, hp, &pl);
    if (rc) return rc;
    rc = check_ws(hp->workspace, hp->workspace_bytes, n_tensors, pl);
    if (rc) return rc;
    return run_step(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, lr, momentum,
                    weight_decay, hp, hp->workspace, pl, stream);
}

int tula_ags_plan_create(float *const *param_ptrs, float *const *grad_ptrs,
                         float *const *mom_ptrs, const int64_t *numels, int n_tensors,
                         const tula_ags_hparams *hp, tula_ags_plan **plan_out) {
    if (!plan_out) return TULA_ERR_ARG;
    *plan_out = nullptr;
    if (!hp || hp->K < 1 || hp->K > TULA_MAX_K) return TULA_ERR_ARG;
    Plan pl;
    int rc = check_step_tensors(param_ptrs, grad_ptrs, mom_ptrs, hp->scale_elem, numels,
                                n_tensors, hp->K, &pl);
    if (rc) return rc;
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    try {
        std::unique_ptr<tula_ags_plan> P(new tula_ags_plan);
        const size_t n = (size_t)n_tensors, K = (size_t)hp->K;
        P->n = n_tensors;
        P->K = hp->K;
        P->device = dev;
        P->tiles = pl;
        P->numels.assign(numels, numels + n);
        P->params.assign(param_ptrs, param_ptrs + n);
        P->grads.assign(grad_ptrs, grad_ptrs + K * n);
        if (mom_ptrs) P->moms.assign(mom_ptrs, mom_ptrs + n);
        if (hp->scale_elem) P->scale_elem.assign(hp->scale_elem, hp->scale_elem + n);
        *plan_out = P.release();
    } catch (const std::bad_alloc &) {
        return TULA_ERR_NO_MEMORY;
    }
    return TULA_OK;
}

int tula_ags_plan_step(tula_ags_plan *plan, float lr, float momentum, float weight_decay,
                       const tula_ags_hparams *hp, void *stream) {
    if (!plan || !hp || hp->K != plan->K) return TULA_ERR_ARG;
    int rc = check_step_options(hp, momentum, !plan->moms.empty(), !plan->scale_elem.empty());
    if (rc) return rc;
    rc = check_ws(hp->workspace, hp->workspace_bytes, plan->n, plan->tiles);
    if (rc) return rc;
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    if (dev != plan->device) return TULA_ERR_ARG;
    tula_ags_hparams h = *hp;
    h.scale_elem = plan->scale_elem.empty() ? nullptr : plan->scale_elem.data();
    return run_step(plan->params.data(), plan->grads.data(),
                    plan->moms.empty() ? nullptr : plan->moms.data(), plan->numels.data(),
                    plan->n, lr, momentum, weight_decay, &h, h.workspace, plan->tiles, stream,
                    kPartWhole, nullptr, nullptr, &plan->tables);
}

int tula_ags_plan_destroy(tula_ags_plan *plan) {
    delete plan;
    return TULA_OK;
}

int tula_ags_shard_reduce(float *const *param_ptrs, float *const *grad_ptrs,
                          float *const *mom_ptrs, const int64_t *numels, int n_tensors,
                          float momentum, const tula_ags_hparams *hp, uint64_t *g2_share,
                          void *stream) {
    Plan pl;
    int rc = check_step_args(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, momentum, hp, &pl);
    if (rc) return rc;
    if (!g2_share || (reinterpret_cast<uintptr_t>(g2_share) & 7u)) return TULA_ERR_ARG;
    rc = check_ws(hp->workspace, hp->workspace_bytes, n_tensors, pl);
    if (rc) return rc;
    return run_step(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, 0.f, momentum, 0.f, hp,
                    hp->workspace, pl, stream, kPartReduce,
                    reinterpret_cast<unsigned long long *>(g2_share), nullptr);
}

int tula_ags_shard_update(float *const *param_ptrs, float *const *grad_ptrs,
                          float *const *mom_ptrs, const int64_t *numels, int n_tensors, float lr,
                          float momentum, float weight_decay, const tula_ags_hparams *hp,
                          const uint64_t *g2_total, void *stream) {
    Plan pl;
    int rc = check_step_args(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, momentum, hp, &pl);
    if (rc) return rc;
    if (!g2_total || (reinterpret_cast<uintptr_t>(g2_total) & 7u)) return TULA_ERR_ARG;
    rc = check_ws(hp->workspace, hp->workspace_bytes, n_tensors, pl);
    if (rc) return rc;
    return run_step(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, lr, momentum,
                    weight_decay, hp, hp->workspace, pl, stream, kPartUpdate, nullptr,
                    reinterpret_cast<const unsigned long long *>(g2_total));
}

int tula_layer_stats(const float *const *param_ptrs, const float *const *grad_ptrs, int K,
                     const int64_t *numels, int n_tensors, double *stats_out, void *workspace,
                     size_t workspace_bytes, void *stream) {
    Plan pl;
    if (!param_ptrs || !grad_ptrs || !stats_out || !valid_numels(numels, n_tensors, K, &pl))
        return TULA_ERR_ARG;
    const int n = n_tensors;
    for (int p = 0; p < n; ++p) {
        if (numels[p] == 0) continue;
        if (!param_ptrs[p] || !aligned4(param_ptrs[p])) return TULA_ERR_ARG;
        for (int k = 0; k < K; ++k) {
            const float *g = grad_ptrs[(size_t)k * n + p];
            if (!g || !aligned4(g)) return TULA_ERR_ARG;
        }
    }
    int rc = check_ws(workspace, workspace_bytes, n, pl);
    if (rc) return rc;
    const WsLayout L = ws_layout(n, pl);
    Scalars sc = make_scalars(nullptr, K, n, workspace, L, kModeStats);
    sc.stats = stats_out;
    sc.read_w = 1;
    auto fill = [&](int p, const float **dst) {
        for (int k = 0; k < K; ++k) dst[k] = grad_ptrs[(size_t)k * n + p];
        dst[K] = param_ptrs[p];
    };
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    rc = run_reduce<false, true, false, false>(K, n, numels, sc, 0, s, fill);
    return rc ? rc : launch_finish(n, sc, s);
}

int tula_ags_update_scale(const float *const *g_small, const float *const *g_large,
                          const int64_t *numels, int n_tensors, const tula_ags_hparams *hp,
                          void *stream) {
    Plan pl;
    if (!hp || !g_small || !g_large || !valid_numels(numels, n_tensors, 1, &pl))
        return TULA_ERR_ARG;
    const int n = n_tensors;
    const bool per_elem = hp->granularity == TULA_SCALE_PER_ELEMENT;
    if (!per_elem && hp->granularity != TULA_SCALE_PER_TENSOR) return TULA_ERR_ARG;
    if (per_elem ? !hp->scale_elem : !hp->scale) return TULA_ERR_ARG;
    for (int p = 0; p < n; ++p) {
        if (numels[p] == 0) continue;
        if (!g_small[p] || !g_large[p] || !aligned4(g_small[p]) || !aligned4(g_large[p]))
            return TULA_ERR_ARG;
        if (per_elem && (!hp->scale_elem[p] || !aligned4(hp->scale_elem[p]))) return TULA_ERR_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (per_elem) {
        Scalars sc;
        std::memset(&sc, 0, sizeof(sc));
        sc.eps = hp->eps;
        sc.s_max = hp->s_max;
        auto fill = [&](int p, const float **dst) {
            dst[0] = g_small[p];
            dst[1] = g_large[p];
            dst[2] = hp->scale_elem[p];
        };
        return launch_streaming({k_scale_elem<true>, k_scale_elem<false>, k_scale_elem<false>, 0, 0}, n,
                                numels, 4096, 3, kScaleThreads, sc, hp->grid_ctas, s, fill);
    }
    int rc = check_ws(hp->workspace, hp->workspace_bytes, n, pl);
    if (rc) return rc;
    const WsLayout L = ws_layout(n, pl);
    Scalars sc = make_scalars(hp, 1, n, hp->workspace, L, kModeScale);
    sc.stats = nullptr;  // the rows of the steps that hp is also used for
    auto fill = [&](int p, const float **dst) {
        dst[0] = g_large[p];
        dst[1] = g_small[p];
    };
    rc = run_reduce_k<1, false, false, true, true>(1, n, numels, sc, hp->grid_ctas, s, fill, nullptr);
    return rc ? rc : launch_finish(n, sc, s);
}

const char *tula_ags_error_string(int code) {
    switch (code) {
    case TULA_OK: return "ok";
    case TULA_ERR_ARG: return "invalid argument";
    case TULA_ERR_WORKSPACE: return "workspace missing, too small or not 256-byte aligned";
    case TULA_ERR_CUDA: return "CUDA launch failed";
    case TULA_ERR_UNSUPPORTED: return "unsupported combination of options";
    case TULA_ERR_SCRATCH_LIMIT:
        return "tensor list needs more than the library's static scratch "
               "(TULA_STATIC_SCRATCH_BYTES); use tula_ags_step with a workspace";
    case TULA_ERR_NO_MEMORY: return "host memory allocation failed";
    default: return "unknown status";
    }
}

int tula_ags_last_cuda_error(void) { return g_last_cuda; }

uint64_t tula_ags_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

}  // extern "C"

// ============================================================================
// Allocation-free step: the scratch in a static device array
// ============================================================================
// For callers that cannot allocate device memory (see the header).  The step
// itself is tula_ags_step's; only where its scratch lives differs.

namespace {

constexpr size_t kStaticScratchBytes = TULA_STATIC_SCRATCH_BYTES;

// One copy per device, alive until the process exits.  In host code this name
// is only a handle: its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// Device address of g_static_scratch in the current device's context.  Looked up on every call
// (a host-side table lookup once the module is loaded): a cached address would go stale when the
// context is destroyed and re-created (cudaDeviceReset).
int static_scratch_address(void **out) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    *out = p;
    return TULA_OK;
}

// The static array's error word (its layout's `err` section does not depend on the tensors).
int static_scratch_error_word(unsigned **out) {
    void *base = nullptr;
    const int rc = static_scratch_address(&base);
    if (rc) return rc;
    *out = reinterpret_cast<unsigned *>(static_cast<char *>(base) + ws_layout(1, Plan{}).err);
    return TULA_OK;
}

}  // namespace

extern "C" int tula_ags_step_static_scratch(float *const *param_ptrs, float *const *grad_ptrs,
                                            float *const *mom_ptrs, const int64_t *numels,
                                            int n_tensors, float lr, float momentum,
                                            float weight_decay, const tula_ags_hparams *hp,
                                            void *stream) {
    Plan pl;
    int rc = check_step_args(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, momentum, hp, &pl);
    if (rc) return rc;
    const WsLayout L = ws_layout(n_tensors, pl);
    if (L.total > kStaticScratchBytes) return TULA_ERR_SCRATCH_LIMIT;
    void *scratch = nullptr;
    rc = static_scratch_address(&scratch);
    if (rc) return rc;
    // The array keeps the last call's contents: zero the tile counters and the accumulators before
    // this call's kernels.  The error word is left alone, so that a wait that ran out stays reported
    // until tula_ags_static_scratch_error reads it.
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char *b = static_cast<char *>(scratch);
    cudaError_t e = cudaMemsetAsync(b, 0, L.err, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b + L.tiles, 0, L.spare - L.tiles, s);
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    return run_step(param_ptrs, grad_ptrs, mom_ptrs, numels, n_tensors, lr, momentum,
                    weight_decay, hp, scratch, pl, stream);
}

extern "C" int tula_ags_static_scratch_error(void *stream, int *error_out) {
    if (!error_out) return TULA_ERR_ARG;
    unsigned *word = nullptr;
    int rc = static_scratch_error_word(&word);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, word, sizeof(v), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && v) e = cudaMemsetAsync(word, 0, sizeof(v), s);
    if (e == cudaSuccess && v) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    *error_out = (int)v;
    return TULA_OK;
}

extern "C" int tula_ags_static_scratch_check_wait_timeout(void *stream) {
    unsigned *word = nullptr;
    const int rc = static_scratch_error_word(&word);
    if (rc) return rc;
    k_wait_check<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(word);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return TULA_ERR_CUDA;
    }
    return TULA_OK;
}
