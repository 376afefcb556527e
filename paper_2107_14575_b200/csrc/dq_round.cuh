// The quantizer kernels: one pass over the gradients that takes the bucket norms (or reads
// them), encodes and packs (Eq. 5/6), and -- in the round kernels -- also forms the server's
// average (Algorithm 1) from the codes while they are still in registers.
//
// Modes (where the norms come from):
//   kWarpBuckets   buckets of 32 * 2^k <= 1024 elements: a warp tile is 1024 / bucket buckets
//   kOddBuckets    other buckets of up to 992 elements: a warp tile is as many buckets as 32 groups hold
//   kTeamBuckets   buckets of 2048 or 4096: a team of 2 or 4 warps of the CTA takes a bucket
//   kGivenNorms    any bucket length, whole-tensor layouts: norms are read, a tile is 32 groups
// B = 0: norms alone.  AVG = false: codes (and norms) of every worker.  AVG = true: a warp keeps its tile of the output
// while it goes through the M workers, whose words it writes as it goes; the averaged gradient (or
// the updated parameters) leaves at the end of the tile.
//
// Every WARP is a pipeline of its own: two 4 KB stages filled by TMA tensor copies with the 128-byte
// swizzle.  A lane owns one 128-byte row (32 elements, one group): it squares the row, the lanes of a
// bucket combine by shuffles, then the lane encodes its row against that norm; the words leave from
// registers or through the consumed stage, which is refilled.
// HBM traffic: 4 + b/8 bytes per element and worker, plus 4 (8 with the update) per output element.
// What bounds it: per tile of a worker a warp issues some 515 instructions at b = 4 (290 of them the codes,
// their draws and the sums; 65 are the wide multiplies of the generator, four cycles of the multiplier
// each), 60 % of the issue slots' and 67 % of the multiplier's time, beside loads that alone take 0.9 of
// the measured copy bandwidth.  Measured: 2^26 elements M = 32 b = 4 1.87 ms (5.3 TB/s; separate
// quantizer and average 2.29), ResNet-18 shape M = 8 88 us (5.1), VGG-16 shape M = 16 b = 5 with update 252 us.
// Rounds with few tiles: see tile_rounds.
#pragma once

#include "dq_common.cuh"
#include "dq_device.cuh"
#include "dq_rule.cuh"
#include "dq_tma.cuh"

#include <type_traits>

enum RoundMode { kWarpBuckets = 0, kTeamBuckets = 1, kGivenNorms = 2, kOddBuckets = 3 };

struct RoundArgs {
    LayoutView v;
    const float* grads;
    int64_t grad_stride;          // elements from a worker's gradient to the next
    float* norms;                 // written, or read (kGivenNorms)
    int32_t* dev_b;               // b of this call; with the rule attached, the next b when the kernel ends
    uint32_t* packed;
    int64_t packed_stride;
    float* out;                   // AVG: averaged gradient, or the parameters (update != 0)
    int32_t* status;
    PhiloxKeys keys;
    uint32_t step;
    uint32_t worker0;             // worker m of the call draws the uniforms of worker worker0 + m
    int32_t M;
    int32_t map_has_worker_dim;   // 0 when all workers read the same buffer (stride 0)
    int32_t gpb_shift;            // log2(groups per bucket) (kWarpBuckets, kTeamBuckets)
    uint32_t div_magic;           // groups_per_bucket as multiply-shift, or as a shift if a power of two
    int32_t div_shift;            //              (>= 0: the shift; < 0: use div_magic with a 33-bit shift)
    int32_t stream_reads;         // 1: more than 64 MB of gradients (see the L2 policy of the reads)
    int32_t linf;                 // norm kind (host: which kernel)
    int32_t update;               // AVG: out <- out + neg_lr * average instead of out <- average
    int32_t wide_words;           // packed rows start on 32-byte boundaries: 32-byte stores allowed
    int32_t wide_out;             // out starts on a 32-byte boundary
    uint32_t each, extra;         // list entries per warp (or team): `each`, one more for the first `extra` of them
    float neg_lr;
    int32_t with_rule;            // choose the next b from this call's norms (dev_b, in place)
    RuleArgs rule;
    WaitLimits wait;
};

// Launch of one of the kernels (each in a translation unit of its own): norms alone, or codes with or
// without the average.  `entries`: length of the list of work (see WarpFetch).
template <int MODE, bool LINF>
int dq_launch_norms(const RoundArgs& a, const CUtensorMap& map, int n_seg, int64_t entries, cudaStream_t st);
template <int MODE, bool AVG, bool LINF>
int dq_launch_round(const RoundArgs& a, const CUtensorMap& map, int n_seg, int64_t entries, cudaStream_t st);
// The round in which a CTA takes its tiles through the workers (buckets of 2048, of the teams').
template <int MODE, bool LINF>
int dq_launch_tile_round(const RoundArgs& a, int n_seg, int64_t entries, cudaStream_t st);

// CTAs per SM, i.e. registers per thread: 128 with the 32 sums (96 spill and run 4-6 % slower); 102 without them
// (codes of 2^24 elements, b = 6: 17.4 us with five CTAs, 18.1 with six of 80 registers, 18.7 with four; buckets of
// 4096, M = 16, b = 5: 251, 256 and 254 us).
template <bool AVG>
struct RoundShape {
    static constexpr int ctas_per_sm = AVG ? 4 : 5;
};

constexpr int kRoundThreads = 128;
constexpr int kRoundWarps = kRoundThreads / 32;
constexpr int kRoundMaxCtasPerSm = 6;            // of any of the kernels (the rule's workspace has a sum per CTA)

// Host, dq_norms.cu: geometry, gradients and tensor map of a launch over view `v` (not the norms, b, words, draws).
bool dq_fill_round(RoundArgs& a, CUtensorMap& map, const dq_layout_t* L, const LayoutView& v, const float* dev_grads,
                   int64_t worker_stride_elems, int32_t M, int32_t* dev_status);
// Whether the kernels take the norms of a layout's buckets themselves.
bool dq_norms_inside(const dq_layout_t* L);
// The norm kernel over the buckets `a` describes.
int dq_norms_of_buckets(const RoundArgs& a, const CUtensorMap& map, int n_seg, cudaStream_t st);
// Positions of a worker's tiles; given: those of kGivenNorms.
int64_t dq_tile_positions(const RoundArgs& a, bool given);

#ifdef DQ_ROUND_KERNELS

namespace {

constexpr int kTileBytes = 32 * 128;
constexpr int kMaxSmemSegs = 1023;

constexpr int kStages = 2;                          // per warp: a tile being encoded and one on its way

// Dynamic shared memory, addressed only through this symbol so that every access compiles to a
// shared-memory instruction:
//   [0, kWarps * kStages * 4 KB)  input tiles, warp-major (1024-byte aligned for the swizzle)
//   (a consumed tile doubles as the staging area of its words where they do not leave straight from
//   registers), then the stage barriers, the teams' exchange slots ([2 parities][4 warps] of {partial,
//   lost}), the rule's partial sums and its last-CTA word, and the tensor table
extern __shared__ __align__(1024) unsigned char smem[];
struct SmemMap {
    static constexpr int bars = kRoundWarps * kStages * kTileBytes;
    static constexpr int slots = bars + kRoundWarps * kStages * 8;
    static constexpr int sums = slots + 2 * kRoundWarps * 8;
    static constexpr int table = sums + kRoundWarps * 8 + 16;
};

__device__ __forceinline__ uint64_t* stage_bar(int warp, int st)
{
    return reinterpret_cast<uint64_t*>(smem + SmemMap::bars) + warp * kStages + st;
}
__device__ __forceinline__ unsigned char* stage_ptr(int warp, int st) { return smem + (warp * kStages + st) * kTileBytes; }

__device__ __forceinline__ uint32_t div_gpb(const RoundArgs& a, uint32_t n)
{
    if (a.div_shift >= 0) return n >> a.div_shift;
    return (uint32_t)(((uint64_t)n * a.div_magic) >> 33);     // exact for n < 2^26, divisor <= 128
}

// A norm load that stays where it is written (a volatile statement keeps its place among the other
// volatile statements, the barrier wait among them): the next worker's norm is requested before this
// one's encoding, not after it.
__device__ __forceinline__ float load_norm_early(const float* p)
{
    float x;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(p));
    return x;
}

// Elements 4c .. 4c + 3 of the row at byte offset `row` of the shared memory (swizzle phase folded in)
__device__ __forceinline__ ulonglong2 row_quad(const uint32_t row, const int c)
{
    return *reinterpret_cast<const ulonglong2*>(smem + (row ^ (uint32_t)(c << 4)));
}

// What a warp knows about a tile position: where it starts and what this lane's share of it is.
struct TilePos {
    int row0;        // first group of the tile
    int row;         // this lane's row of the tile (its group is row0 + row)
    int valid;       // elements of that group that count (0: nobody's row)
    int bucket;      // its bucket
    int span;        // groups of the tile that get words
    int len;         // kOddBuckets: elements of this lane's bucket
    bool regular;    // every lane owns its own full row
    bool writes;     // this lane writes the norm of its bucket
};

// Whether the lane speaks for its bucket where the warp asks for sums out of range.  A tile at the end of a layout has lanes
// without a bucket, whose sum of nothing is no reason to go and look (it was one: a round of 70,000 elements with 8 workers
// in one kernel took 19.4 us, now 14.8).  The warps of a team have the same sum and must agree, rows or not.
template <int MODE>
__device__ __forceinline__ bool has_say(const TilePos& t)
{
    return MODE == kTeamBuckets || t.valid > 0;
}

// Bucket reductions in the order of dq_bucket_norms: four accumulators over a full row's float4
// components (one over a tensor's last, partial row), a pairwise join.
__device__ __forceinline__ float row_sum_squares(const uint32_t row)
{
    uint64_t a01 = 0ull, a23 = 0ull;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const ulonglong2 x = row_quad(row, c);
        a01 = fma_pair(x.x, x.x, a01);
        a23 = fma_pair(x.y, x.y, a23);
    }
    float a0, a1, a2, a3;
    unpack_pair(a01, a0, a1);
    unpack_pair(a23, a2, a3);
    return (a0 + a1) + (a2 + a3);
}
__device__ __forceinline__ float row_max(const uint32_t row)
{
    float m0 = 0.0f, m1 = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const ulonglong2 x = row_quad(row, c);
        float u, w;
        unpack_pair(x.x, u, w);
        m0 = max_magnitude(m0, u, w);
        unpack_pair(x.y, u, w);
        m1 = max_magnitude(m1, u, w);
    }
    return max_nan(m0, m1);
}

// What a tile that touches a tensor's end needs more, out of line so that the others do not pay for
// its registers.  The tail of a partial row is padding: it is set to zero where it stands, and the
// row's sum runs through one accumulator (zeros leave it as it is).  Rows that are nobody's (valid = 0) are left alone and
// add nothing.  Thirty-two bytes at a time: element by element, every load waited for the one before (a round of 3000
// elements with 8 workers in one kernel took 22 us, one of 2048 17).
template <bool LINF>
__device__ __noinline__ float end_row(const uint32_t row, const int valid)
{
    float chain = 0.0f;
    if (valid > 0 && valid < 32) {
#pragma unroll 1
        for (int c = 0; c < 128; c += 32) {
            float4* p[2] = {reinterpret_cast<float4*>(smem + (row ^ (uint32_t)c)), reinterpret_cast<float4*>(smem + (row ^ (uint32_t)(c + 16)))};
            float4 x[2] = {*p[0], *p[1]};
            int here = valid - (c >> 2);               // elements of these eight and behind them that count
#pragma unroll
            for (int i = 0; i < 2; ++i, here -= 4) {
                if (here < 4) {
                    x[i] = make_float4(here < 1 ? 0.0f : x[i].x, here < 2 ? 0.0f : x[i].y, here < 3 ? 0.0f : x[i].z, 0.0f);
                    *p[i] = x[i];
                }
                if (LINF) {
                    chain = max_magnitude(chain, x[i].x, x[i].y);
                    chain = max_magnitude(chain, x[i].z, x[i].w);
                } else {
                    chain = fmaf(x[i].x, x[i].x, chain);
                    chain = fmaf(x[i].y, x[i].y, chain);
                    chain = fmaf(x[i].z, x[i].z, chain);
                    chain = fmaf(x[i].w, x[i].w, chain);
                }
            }
        }
    }
    __syncwarp();
    return chain;
}

// A norm that is an infinity or a NaN: the scale of the codes is 0, every code is s and every term of the average
// 0 * norm = NaN, but 0 times an entry that is not finite has no code (for b <= 4 its bits reach the codes of its
// neighbours).  Kernels with l2 norms set the row of such a bucket to zero beforehand, in the call that finds the norm,
// which costs the others nothing; the ones that have no such call set the words after the encoder.  (That in all of
// them: VGG-16 shape M = 16 with update 256 -> 264 us, codes of 1.6M elements M = 4 8.9 -> 9.3; clearing the row beside the
// encoder: l-inf rounds 25.9 -> 27.9.)
template <int MODE, bool LINF>
struct ClearsRow {
    static constexpr bool value = !LINF && MODE != kGivenNorms;
};
template <bool CLEAR>
__device__ __forceinline__ void clear_nonfinite_row(const uint32_t row, const int valid, const float nrm)
{
    if constexpr (CLEAR) {
        if (valid == 0 || isfinite(nrm)) return;                 // (valid = 0: the lane has no row of its own)
#pragma unroll 1
        for (int c = 0; c < 128; c += 16) *reinterpret_cast<float4*>(smem + (row ^ (uint32_t)c)) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// The lanes of a bucket combine their v; the result is the same in all of them.
template <int MODE, class Op>
__device__ __forceinline__ float join_lanes(float v, const int gpb, const Op& op)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float other = __shfl_xor_sync(0xffffffffu, v, o);
        if (MODE == kTeamBuckets || o < gpb) v = op(v, other);
    }
    return v;
}
// ... and so do the warps of a team.  A warp that lost a wait says so in its slot: `lost` is then set in
// every warp of the team.  slots: float2[2][kRoundWarps], the exchanges of even and of odd number.
template <int MODE, class Op>
__device__ __forceinline__ float join_team(float v, float2* slots, const int T_shift, uint32_t& exchanges, const bool landed,
                                           bool& lost, const Op& op)
{
    if constexpr (MODE == kTeamBuckets) {
        const int warp = threadIdx.x >> 5, T = 1 << T_shift;
        slots += (exchanges & 1u) * kRoundWarps;
        ++exchanges;
        if ((threadIdx.x & 31) == 0) slots[warp] = make_float2(v, landed ? 0.0f : 1.0f);
        // (numbers the assembler sees: a number from a register reserves all sixteen barriers for the CTA, and
        // only four such CTAs fit an SM)
        if (warp >> T_shift) asm volatile("bar.sync 2, %0;" ::"r"(32 << T_shift) : "memory");
        else asm volatile("bar.sync 1, %0;" ::"r"(32 << T_shift) : "memory");
        const float2* mine = slots + (warp & ~(T - 1));
        float any = mine[0].y;
        v = op(0.0f, mine[0].x);
        for (int i = 1; i < T; ++i) { v = op(v, mine[i].x); any += mine[i].y; }
        lost |= any != 0.0f;
    }
    return v;
}
struct AddOp { __device__ __forceinline__ float operator()(const float a, const float b) const { return a + b; } };
struct MaxOp { __device__ __forceinline__ float operator()(const float a, const float b) const { return max_nan(a, b); } };
template <bool LINF> struct JoinOp { using type = AddOp; };
template <> struct JoinOp<true> { using type = MaxOp; };

// kOddBuckets: the bucket sums (maxima) of a tile, in the order of the kernel that took such buckets before.
// The warp goes through the buckets one by one -- half warps two by two for buckets of 96 --, lane i taking
// the bucket's float4s i, i + 32, ...; a lane gets the result of its own bucket, r (1 if it has none).
// stage: byte offset of the tile; the buckets' first rows and lengths are with the lanes r * gpb.
__device__ __forceinline__ float4 stage_float4(const uint32_t stage, const int first, const int i)
{
    const int row = first + (i >> 3);
    return *reinterpret_cast<const float4*>(smem + stage + tma::swizzle128(row, i & 7));
}
__device__ __forceinline__ float stage_float(const uint32_t stage, const int first, const int e)
{
    const int row = first + (e >> 5);
    return *reinterpret_cast<const float*>(smem + stage + tma::swizzle128(row, (e >> 2) & 7) + ((e & 3) << 2));
}
template <int P, int UNROLL>
__device__ __forceinline__ float odd_share(const uint32_t stage, const int first, const int len, const int lane, const int lanes)
{
    const int n4 = len >> 2;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll UNROLL
    for (int i = lane; i < n4; i += lanes) {
        const float4 x = stage_float4(stage, first, i);
        a0 = take<P>(a0, x.x); a1 = take<P>(a1, x.y); a2 = take<P>(a2, x.z); a3 = take<P>(a3, x.w);
    }
    if (lane < (len & 3)) a0 = take<P>(a0, stage_float(stage, first, n4 * 4 + lane));
    return join<P>(join<P>(a0, a1), join<P>(a2, a3));
}
template <bool LINF>
__device__ __forceinline__ float odd_bucket_sums(const uint32_t stage, const int row, const int len, const int gpb, const int R, const int r)
{
    constexpr int P = LINF ? DQ_NORM_LINF : DQ_NORM_L2;
    const int lane = threadIdx.x & 31;
    float mine = 1.0f;
    if (gpb >= 4) {
#pragma unroll 1
        for (int k = 0; k < R; ++k) {
            const int first = __shfl_sync(0xffffffffu, row, k * gpb), n = __shfl_sync(0xffffffffu, len, k * gpb);
            float v = odd_share<P, 1>(stage, first, n, lane, 32);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) v = join<P>(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (r == k) mine = v;
        }
    } else {                                     // 96 elements: R = 10, an even number
        // (unrolled: five reductions in flight; ResNet-18 shape, M = 8, b = 4 222 -> 212 us.  The longer buckets' loop
        // loses 2 % when it is unrolled.)
#pragma unroll
        for (int k = 0; k < 10; k += 2) {
            const int src = (k + (lane >> 4)) * 3;
            const int first = __shfl_sync(0xffffffffu, row, src), n = __shfl_sync(0xffffffffu, len, src);
            float v = odd_share<P, 4>(stage, first, n, lane & 15, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v = join<P>(v, __shfl_xor_sync(0xffffffffu, v, o));
            const float lo = __shfl_sync(0xffffffffu, v, 0), hi = __shfl_sync(0xffffffffu, v, 16);
            if (r == k) mine = lo;
            if (r == k + 1) mine = hi;
        }
    }
    return mine;
}
// ... and the norms of those out of range, as rare_norm has them.  The largest magnitudes come from the lanes' own
// rows, of all buckets at once, which settles buckets of zeros, infinities and NaNs; the scaled squares of the others
// are added bucket by bucket (half warps two by two for buckets of 96).  own, valid: the lane's row and its elements.
// Sparse gradients are full of zero buckets: 2^25 elements M = 8 b = 4, 97 % of rows of 300 zero, a round with buckets
// of 96 1839 -> 441 us, 480 884 -> 292 (each bucket reduced twice, and encoded, before); entries of 1e-25, all out of
// range, 2045 -> 958 and 957 -> 685.
template <bool CLEAR>
__device__ __noinline__ float rare_norm_odd(const uint32_t stage, const int row, const int len, const int gpb, const int R, const int r,
                                            const float sum, const float nrm, const uint32_t own, const int valid)
{
    const int lane = threadIdx.x & 31;
    const bool again = r < R && !l2_sum_in_range(sum);
    // (as numbers, magnitudes are in the order of the floats, and a NaN is above them all)
    const uint32_t mine_max = valid > 0 ? __float_as_uint(row_max(own)) : 0u;
    float largest = 0.0f;
    for (int k = 0; k < R; ++k) {
        const uint32_t m = __reduce_max_sync(0xffffffffu, r == k ? mine_max : 0u);
        if (r == k) largest = __uint_as_float(m);
    }
    const uint32_t todo = __ballot_sync(0xffffffffu, again && magnitude_scalable(largest));
    float norm = again ? largest : nrm;
    const int lanes = gpb >= 4 ? 32 : 16, halves = gpb >= 4 ? 1 : 2;
    for (int k = 0; k < R; k += halves) {
        const int mine = k + (halves == 2 ? lane >> 4 : 0);            // (R = 10 buckets of 96: an even number)
        if ((todo >> (k * gpb) & 1u) == 0u && (halves == 1 || (todo >> ((k + 1) * gpb) & 1u) == 0u)) continue;
        const int first = __shfl_sync(0xffffffffu, row, mine * gpb), n = __shfl_sync(0xffffffffu, len, mine * gpb);
        // 2^-e in two steps, each a normal number (exact, or of no account where the product underflows)
        const int e = scale_exponent(__shfl_sync(0xffffffffu, largest, mine * gpb)), e1 = e / 2;
        const float f1 = __uint_as_float((uint32_t)(127 - e1) << 23), f2 = __uint_as_float((uint32_t)(127 - (e - e1)) << 23);
        float ss = 0.0f;
        for (int i = lane & (lanes - 1); i < n; i += lanes) {
            const float y = stage_float(stage, first, i) * f1 * f2;
            ss = fmaf(y, y, ss);
        }
        for (int o = lanes >> 1; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float got = __shfl_sync(0xffffffffu, ss, halves == 2 ? (r - k) << 4 & 16 : 0);
        if (r >= k && r < k + halves && (todo >> lane & 1u) != 0u) norm = rescaled_l2(largest, got, scale_exponent(largest));
    }
    clear_nonfinite_row<CLEAR>(own, valid, norm);
    return norm;
}

// The l2 norm of buckets whose sum of squares is out of range (see l2_sum_in_range): all zeros, tiny
// entries, an overflowed square.  Called by all lanes of the warp (by all warps of a team, which agree
// on the sum); zero buckets are settled by their largest magnitude, the others are reduced again with
// their entries scaled, and lanes whose own bucket was in range keep `nrm`.  Always two exchanges of a
// team.  Out of line: it is rare, and the common case does not pay for its registers.
template <int MODE, bool CLEAR>
__device__ __noinline__ float rare_norm(const uint32_t row, const int valid, const int gpb, float2* slots, const int T_shift,
                                        uint32_t exchanges, const float sum, const float nrm)
{
    bool lost = false;
    float mx = valid > 0 ? row_max(row) : 0.0f;          // (a partial row's tail is zero by now)
    mx = join_team<MODE>(join_lanes<MODE>(mx, gpb, MaxOp{}), slots, T_shift, exchanges, true, lost, MaxOp{});
    const bool again = !l2_sum_in_range(sum);
    float scaled = 0.0f;
    const int e = scale_exponent(mx);
    if (MODE == kTeamBuckets || __any_sync(0xffffffffu, again && magnitude_scalable(mx))) {
        const ScaledSquares red{e};
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f, chain = 0.f;
#pragma unroll 1
        for (int c = 0; c < 8; ++c) {
            const float4 x = *reinterpret_cast<const float4*>(smem + (row ^ (uint32_t)(c << 4)));
            a0 = red.take(a0, x.x); a1 = red.take(a1, x.y); a2 = red.take(a2, x.z); a3 = red.take(a3, x.w);
            chain = red.take(chain, x.x); chain = red.take(chain, x.y); chain = red.take(chain, x.z); chain = red.take(chain, x.w);
        }
        scaled = valid == 32 ? (a0 + a1) + (a2 + a3) : (valid > 0 ? chain : 0.0f);
        scaled = join_team<MODE>(join_lanes<MODE>(scaled, gpb, AddOp{}), slots, T_shift, exchanges, true, lost, AddOp{});
    }
    const float norm = again ? (magnitude_scalable(mx) ? rescaled_l2(mx, scaled, e) : mx) : nrm;
    clear_nonfinite_row<CLEAR>(row, valid, norm);
    return norm;
}

constexpr uint32_t kNoTile = 0x7fffffffu;

// Where the tiles of a worker lie.  table: byte offset of the tensor table in shared memory.
template <int MODE>
struct TileMap {
    static constexpr bool ODD = MODE == kOddBuckets;
    static constexpr bool TILES = MODE == kWarpBuckets || ODD;        // tiles of whole buckets
    const RoundArgs& a;
    const bool in_smem;
    const int32_t* const tbl_s;
    const int lane, n1, gpb;
    const int T_shift, sub;          // log2 of the warps that share a bucket, and this warp's place among them
    const int R;                     // buckets per warp tile
    const int r, l;                  // of a regular tile: the lane's bucket and its group in there (kOddBuckets: the last lanes may have none, r >= R)
    // the tensor looked at last: first bucket, first group, elements, end (in buckets), full buckets
    int c_b0, c_g0, c_n, c_end, c_full;

    __device__ __forceinline__ TileMap(const RoundArgs& args, const bool tbl_in_smem, const int table, const int warp_of_team)
        : a(args), in_smem(tbl_in_smem), tbl_s(reinterpret_cast<const int32_t*>(smem + table)), lane(threadIdx.x & 31),
          n1(args.v.n_seg + 1), gpb(ODD ? args.v.groups_per_bucket : 1 << args.gpb_shift),
          T_shift(MODE == kTeamBuckets ? args.gpb_shift - 5 : 0), sub(warp_of_team),
          R(ODD ? 32 / gpb : (MODE == kWarpBuckets ? 32 >> args.gpb_shift : 1)),
          r(ODD ? lane / gpb : lane >> args.gpb_shift), l(lane - (ODD ? r * gpb : r << args.gpb_shift))
    {
        c_b0 = 0;
        c_g0 = 0;
        c_n = a.v.seg0_elems;
        c_end = a.v.n_seg == 1 ? 0x7fffffff : 0;
        c_full = full_buckets(c_n);
    }
    __device__ __forceinline__ int full_buckets(const int n) const
    {
        return ODD ? (int)div_gpb(a, (uint32_t)n >> 5) : n >> (a.gpb_shift + 5);
    }
    __device__ __forceinline__ int tbl(const int i) const { return in_smem ? tbl_s[i] : __ldg(a.v.seg_group0 + i); }
    // Tile positions of one worker; a team takes bucket `pos`, each of its warps 1024 elements of it.
    __device__ __forceinline__ int positions() const
    {
        return TILES ? (a.v.nb + R - 1) / R : (MODE == kTeamBuckets ? a.v.nb : (a.v.total_groups + 31) / 32);
    }
    // last tensor whose first bucket (column 1) or group (column 0) is <= x
    __device__ __forceinline__ int find_seg(const int column, const int x) const
    {
        return last_not_above_by_warp(x, a.v.n_seg, [&](int i) { return tbl(column * n1 + i); });
    }
    // the same for an x of each lane's own, from tensor `from` on
    __device__ __forceinline__ int walk_seg(const int column, int from, const int x) const
    {
        while (x >= tbl(column * n1 + from + 1)) ++from;
        return from;
    }
    // kWarpBuckets, kTeamBuckets: first group of the warp's tile at position p, bit 31 set if every lane owns
    // a full row of it; kNoTile if a team's bucket ends before this warp's share.  kGivenNorms: the tensor of
    // the tile's first group. 
    __device__ __forceinline__ uint32_t describe(const int p)
    {
        const int k0 = MODE == kGivenNorms ? p * 32 : p * R;
        if constexpr (MODE == kGivenNorms) {
            return a.v.n_seg == 1 ? 0u : (uint32_t)find_seg(0, k0);
        } else {
            if (k0 < c_b0 || k0 >= c_end) {
                const int i = find_seg(1, k0);
                c_b0 = tbl(n1 + i);
                c_end = tbl(n1 + i + 1);
                c_g0 = tbl(i);
                c_n = tbl(2 * n1 + i);
                c_full = full_buckets(c_n);
            }
            const int local = k0 - c_b0;
            if constexpr (TILES) {
                return (uint32_t)(c_g0 + (ODD ? local * gpb : local << a.gpb_shift)) | (local + R <= c_full ? 0x80000000u : 0u);
            } else {
                const int share = (local << T_shift) + sub;              // 1024-element pieces of the tensor before it
                const int left = c_n - share * 1024;
                if (left <= 0) return kNoTile;
                return (uint32_t)(c_g0 + share * 32) | (left >= 1024 ? 0x80000000u : 0u);
            }
        }
    }
    __device__ __forceinline__ TilePos locate(const int p, const uint32_t desc) const
    {
        const int nb = a.v.nb, G = a.v.total_groups;
        TilePos t;
        t.row = lane; t.valid = 32; t.span = 32; t.bucket = p; t.writes = false;
        t.row0 = MODE == kGivenNorms ? p * 32 : (int)(desc & 0x7fffffffu);
        t.regular = (desc >> 31) != 0;
        t.len = gpb * 32;
        if constexpr (TILES) {
            const int k = p * R + r;
            const bool mine = k < nb && (!ODD || r < R);
            t.bucket = k;
            t.writes = l == 0 && mine;
            if (ODD) {
                t.valid = r < R ? 32 : 0;
                t.span = R * gpb;
            }
            if (!t.regular) {
                // the tile touches the end of a tensor: buckets may be short, rows may be nobody's
                int first = 0, len = 0;
                const int seg0 = a.v.n_seg > 1 ? find_seg(1, p * R) : 0;
                if (mine) {
                    int local = k, n = a.v.seg0_elems, g0 = 0;
                    if (a.v.n_seg > 1) {
                        const int i = walk_seg(1, seg0, k);
                        local = k - tbl(n1 + i);
                        n = tbl(2 * n1 + i);
                        g0 = tbl(i);
                    }
                    first = g0 + (ODD ? local * gpb : local << a.gpb_shift);
                    const int left = n - local * (gpb * 32);
                    len = left < gpb * 32 ? left : gpb * 32;
                }
                t.row = first - t.row0 + l;
                const int v = len - l * 32;
                t.valid = v < 0 ? 0 : (v > 32 ? 32 : v);
                t.len = len;
                if (t.valid == 0 && !(ODD && l == 0 && mine)) t.row = lane;
                t.span = __reduce_max_sync(0xffffffffu, t.valid > 0 ? t.row + 1 : 0);
            }
        } else if constexpr (MODE == kTeamBuckets) {
            t.writes = sub == 0 && lane == 0;
            if (!t.regular) {
                if (desc == kNoTile) {
                    t.row0 = -1; t.valid = 0; t.span = 0;
                } else {
                    int local = p, n = a.v.seg0_elems;
                    if (a.v.n_seg > 1) {
                        const int i = find_seg(1, p);
                        local = p - tbl(n1 + i);
                        n = tbl(2 * n1 + i);
                    }
                    const int v = n - ((local << T_shift) + sub) * 1024 - lane * 32;
                    t.valid = v < 0 ? 0 : (v > 32 ? 32 : v);
                    t.span = __reduce_max_sync(0xffffffffu, t.valid > 0 ? lane + 1 : 0);
                }
            }
        } else {
            const int g = t.row0 + lane;
            t.valid = 0;
            if (g < G) {
                int local = g, n = a.v.seg0_elems, b0 = 0;
                if (a.v.n_seg > 1) {
                    const int i = walk_seg(0, (int)desc, g);
                    local = g - tbl(i);
                    b0 = tbl(n1 + i);
                    n = tbl(2 * n1 + i);
                }
                const int k = (int)div_gpb(a, (uint32_t)local);
                t.bucket = b0 + k;
                t.writes = local == k * a.v.groups_per_bucket;       // (the lane that accounts for the bucket's norm)
                const int left = n - local * 32;
                t.valid = left < 32 ? left : 32;
            }
            t.regular = __all_sync(0xffffffffu, t.valid == 32);
            t.span = (G - t.row0) < 32 ? (G - t.row0) : 32;
        }
        return t;
    }
};

// A warp's list of work and its copies: tiles are fetched in the order they are consumed, two ahead.  The list: positions
// (AVG: every position goes through all workers), or the worker-major list of all tiles.  Each unit -- a warp, or a
// team -- takes every hop-th entry, `each` of them, the first `extra` units one more: dense and sparse stretches of a
// gradient then fall to all units alike (text shape, 97 % of the embedding's rows zero: 154 -> 145 us against contiguous
// ranges).
template <int MODE, bool AVG>
struct WarpFetch {
    static constexpr bool TEAM = MODE == kTeamBuckets;
    TileMap<MODE>& tiles;
    const CUtensorMap* map;
    const int n_pos, hop, positions;
    const int m_first, pos0;         // the first entry: worker (codes alone) and position
    int pos, m, left;                // AVG: position and worker of the next copy; copies to come
    int worker;                      // !AVG: worker of the next copy, as a coordinate
    uint32_t first;                  // what describe() says of its position
    // A team's warp has no tile of some buckets, so it keeps the parity of each stage's next copy and which
    // copies are on their way, a bit each; the others find the parity by counting.
    uint32_t parities, flying;
    // !AVG: descriptions of the positions fetched and not done with, the consumer's and at most two more
    uint32_t queue0, queue1, queue2;
    int queued;
    // L2 policy of the reads.  AVG: evict-normal.  The words are not read again by the call, and gradients
    // that leave the L2 ahead of them leave a cache full of dirty words: writing 1 GB beside 8.6 GB of reads
    // then costs twice its bytes (copy loop without the encoder, d = 2^26, M = 32, b = 4: 1706 us with
    // evict-first, 1585 normal; text shape 145 -> 134 us, whole-tensor norms 160 -> 155 us at b = 4).  Codes
    // alone: evict-first above 64 MB, the average reads them next (2^24 elements: 16.6 us, 17.3 normal).  For given norms it
    // is made once, before the loop: at every copy / once (us) 33.5M elements M = 4 b = 4 102.4 / 98.9, M = 8 b = 2 199.0 / 192.8.  Where
    // the norms are found as well it makes 1 or 2 % either way: 33.5M M = 4 b = 4 104.2 / 102.9, 16.8M M = 4 b = 8 l-infinity 59.7 / 61.0,
    // M = 1 b = 6 16.4 / 16.5; and AVG has no registers to keep it.
    static constexpr bool kKeepsPolicy = MODE == kGivenNorms && !AVG;
    uint64_t policy;

    __device__ __forceinline__ static uint64_t policy_of(const RoundArgs& a)
    {
        return (!AVG && a.stream_reads) ? tma::policy_evict_first() : tma::policy_evict_normal();
    }
    __device__ __forceinline__ static uint32_t unit_of(const RoundArgs& a)
    {
        return (blockIdx.x * kRoundWarps + (threadIdx.x >> 5)) >> (TEAM ? a.gpb_shift - 5 : 0);
    }
    __device__ __forceinline__ WarpFetch(TileMap<MODE>& where, const CUtensorMap* tensor_map)
        : tiles(where), map(tensor_map), n_pos((int)(where.a.each + (unit_of(where.a) < where.a.extra ? 1u : 0u))),
          hop((int)((gridDim.x * kRoundWarps) >> where.T_shift)), positions(where.positions()),
          m_first((AVG || where.a.M == 1) ? 0 : (int)((int64_t)unit_of(where.a) / positions)),
          pos0((int)((int64_t)unit_of(where.a) - (int64_t)m_first * positions)), pos(pos0), m(0),
          left(AVG ? n_pos * where.a.M : n_pos), worker(m_first * (where.a.map_has_worker_dim ? 1 : 0)), first(kNoTile),
          parities(0), flying(0), queue0(0), queue1(0), queue2(0), queued(0),
          policy(kKeepsPolicy ? policy_of(where.a) : 0)
    {
        if (left > 0) first = tiles.describe(pos);
    }
    __device__ __forceinline__ int items() const { return AVG ? n_pos * tiles.a.M : n_pos; }
    __device__ __forceinline__ void next(const int st)
    {
        if (left <= 0) return;
        --left;
        const RoundArgs& a = tiles.a;
        if (!AVG) {
            if (queued == 0) queue0 = first;
            else if (queued == 1) queue1 = first;
            else queue2 = first;
            ++queued;
        }
        if (TEAM && first != kNoTile) flying |= 1u << st;
        if ((threadIdx.x & 31) == 0 && (!TEAM || first != kNoTile))
            tma::fetch_tile(tma::smem_addr(stage_ptr(threadIdx.x >> 5, st)), map, tma::smem_addr(stage_bar(threadIdx.x >> 5, st)),
                            kTileBytes, MODE == kGivenNorms ? pos * 32 : (int)(first & 0x7fffffffu),
                            AVG ? (a.map_has_worker_dim ? m : 0) : worker,
                            kKeepsPolicy ? policy : policy_of(a));
        if (AVG) {
            if (++m == a.M) {
                m = 0; pos += hop;
                if (left > 0) first = tiles.describe(pos);
            }
        } else {
            pos += hop;
            while (pos >= positions) { pos -= positions; worker += a.map_has_worker_dim ? 1 : 0; }
            if (left > 0) first = tiles.describe(pos);
        }
    }
};

template <int B, int MODE, bool AVG, bool LINF>
__device__ __forceinline__ void round_tiles(const RoundArgs& a, TileMap<MODE>& tiles, WarpFetch<MODE, AVG>& copies, double& square_sum)
{
    using Join = typename JoinOp<LINF>::type;
    float2* slots = reinterpret_cast<float2*>(smem + SmemMap::slots);
    constexpr int s = B > 0 ? (1 << (B > 0 ? B - 1 : 0)) - 1 : 0;
    const float sf = (float)s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int M = a.M;
    const int nb = a.v.nb;
    const int G = a.v.total_groups;
    constexpr bool kClears = B != 0 && ClearsRow<MODE, LINF>::value;
    constexpr bool ODD = MODE == kOddBuckets;
    const int T_shift = tiles.T_shift;
    const int gpb = tiles.gpb, R = tiles.R, r = tiles.r;
    const int n_pos = copies.n_pos, hop = copies.hop, items = copies.items();
    int pos = copies.pos0;
    const uint32_t bar0 = tma::smem_addr(stage_bar(warp, 0));

    const float to_unit = (B <= 1) ? 0.0f : __fdiv_rn(1.0f, (float)s * (float)M);          // 1 / (s * M)
    uint32_t it = 0;                              // items consumed; item i travels through stage i & 1
    uint32_t exchanges = 0;
    bool timed_out = false, bad = false;
    // (test hook: the warp's first wait counts as lost, and the warp goes straight to what follows a time-out)
    const bool skip_all = a.wait.lose_first != 0u && items > 0;
    int m = copies.m_first;
    // Every lane polls the barrier itself; the verdict is made warp-uniform so that the warp-level
    // synchronisations are always reached by all lanes or by none.
    auto wait_for = [&](int stage) -> bool {
        const uint32_t par = MODE == kTeamBuckets ? (copies.parities >> stage) & 1u : (it >> 1) & 1u;
        const bool landed = __all_sync(0xffffffffu, tma::mbar_try_wait(bar0 + stage * 8, par)) ||
                            __all_sync(0xffffffffu, tma::mbar_wait(stage_bar(warp, stage), par, a.wait));
        if (MODE == kTeamBuckets && landed) { copies.parities ^= 1u << stage; copies.flying &= ~(1u << stage); }
        return landed;
    };

    for (int ip = 0; ip < n_pos && !skip_all; ++ip) {
        // (where the tile lies -- codes alone: worked out once, when the copies move there; AVG: twice, the second time from
        // the tensor looked at last as a rule)
        const TilePos t = tiles.locate(pos, AVG ? tiles.describe(pos) : copies.queue0);
        const bool has_tile = MODE != kTeamBuckets || t.row0 >= 0;
        // byte offset of the lane's row inside a stage, swizzle phase folded in: chunk c sits at own ^ (c << 4)
        const uint32_t own = (uint32_t)(t.row * 128 + ((t.row & 7) << 4));
        const uint32_t q0 = (uint32_t)(t.row0 + t.row) * 4u;
        uint64_t acc2[16];
        if constexpr (AVG) {
#pragma unroll
            for (int q = 0; q < 16; ++q) acc2[q] = 0ull;
        }
        // this lane's norm and the start of the tile's words, of the worker at hand
        float* norm_ptr = a.norms + (int64_t)m * nb + t.bucket;
        uint32_t* tile_words = a.packed + (int64_t)m * a.packed_stride + (int64_t)t.row0 * B;
        float norm_next = 0.0f;
        if constexpr (MODE == kGivenNorms) {
            if (t.valid > 0) norm_next = load_norm_early(norm_ptr);
        }

        // The norm of a tile: the lane's share from its row, ...
        auto row_share = [&](uint32_t row, const bool landed) -> float {
            float v = LINF ? row_max(row) : row_sum_squares(row);
            if (!t.regular) {
                const float end = has_tile && landed ? end_row<LINF>(row, t.valid) : 0.0f;
                if (t.valid != 32) v = end;
            }
            return v;
        };
        // ... the norm and its scale from the bucket's sum (or maximum) `v`, ...
        float nrm = 0.0f, inv = 0.0f;
        bool plain = false;                      // no zero bucket, no norm outside the normal range
        auto scale_of = [&](float v) {
            nrm = LINF ? v : sqrt_normal(v);
            inv = inv_scale_normal(sf, nrm);
        };
        // ... and what remains: the buckets out of range, and the norm written.  Rarely a bucket's sum of squares
        // is out of range (see l2_sum_in_range): all zeros, tiny entries, an overflowed square.
        auto settle = [&](float v, uint32_t row, float* dst) {
            plain = !__any_sync(0xffffffffu, has_say<MODE>(t) && (LINF ? !norm_is_plain(v) : !l2_sum_in_range(v)));
            if (!plain) {
                if constexpr (!LINF) {
                    if constexpr (ODD) {
                        nrm = rare_norm_odd<kClears>(row - own, t.row, t.len, gpb, R, r, v, nrm, row, t.valid);
                    } else {
                        nrm = rare_norm<MODE, kClears>(row, t.valid, gpb, slots, T_shift, exchanges, v, nrm);
                        exchanges += 2;
                    }
                }
                inv = inv_scale(sf, nrm);
                bad |= t.writes && !isfinite(nrm);
            }
            if (t.writes) {
                DQ_STORE(dst, nrm, a.norms, (int64_t)M * nb * 4, a.status);
                square_sum = fma((double)nrm, (double)nrm, square_sum);
            }
            __syncwarp();
        };

        const int workers = AVG ? M : 1;
#pragma unroll 1
        for (int j = 0; j < workers; ++j, norm_ptr += nb, tile_words += a.packed_stride) {
            const int mm = AVG ? j : m;
            const int st = (int)(it & 1u);
            const uint32_t row = (uint32_t)((warp * kStages + st) * kTileBytes) + own;
            const bool landed = !has_tile || wait_for(st);
            if (MODE != kTeamBuckets && !landed) { timed_out = true; break; }
            if constexpr (MODE == kGivenNorms || ODD) {
                if (!t.regular && landed) (void)end_row<LINF>(row, t.valid);
            }
            if constexpr (MODE == kGivenNorms) {
                nrm = norm_next;
                inv = inv_scale_normal(sf, nrm);
                plain = !__any_sync(0xffffffffu, !norm_is_plain(nrm));
                if (!plain) inv = inv_scale(sf, nrm);
                if (AVG && j + 1 < workers && t.valid > 0) norm_next = load_norm_early(norm_ptr + nb);
                if (t.writes) square_sum = fma((double)nrm, (double)nrm, square_sum);
            } else {
                bool lost = false;
                float v;
                if constexpr (ODD) v = odd_bucket_sums<LINF>(row - own, t.row, t.len, gpb, R, r);
                else v = join_team<MODE>(join_lanes<MODE>(row_share(row, landed), gpb, Join{}), slots, T_shift, exchanges, landed,
                                                lost, Join{});
                if (lost) { timed_out = true; break; }
                scale_of(v);
                settle(v, row, norm_ptr);
            }
            if (!has_tile) {
                copies.next(st);
            } else if constexpr (B == 0) {       // norms alone: the row has been read (see the refill below)
                tma::fence_proxy_async();
                __syncwarp();
                copies.next(st);
            } else {
                // ---- codes of the row against that norm, and the lane's share of the average
                uint32_t words[B];
                const float scale = nrm * to_unit;
                const uint64_t inv2 = pack_pair(__float_as_uint(inv), __float_as_uint(inv));
                const uint64_t scale2 = pack_pair(__float_as_uint(scale), __float_as_uint(scale));
                if constexpr (B == 1) {
                    words[0] = 0u;
                } else if (!plain && __all_sync(0xffffffffu, nrm == 0.0f || t.valid == 0)) {
                    // sparse gradients are full of zero buckets: every code is s, whatever the draw, and adds 0 to the
                    // average (lanes without a row have no say: a tile of odd buckets always has some)
                    zero_group_words<B>(words);
                } else {
                    encode_row<B, AVG>([row](int c) { return row_quad(row, c); }, inv2, scale2, acc2, words, q0,
                                       (uint32_t)mm + a.worker0, a.step, a.keys);
                    if constexpr (!kClears) {
                        if (!isfinite(nrm)) zero_group_words<B>(words);
                    }
                }

                // ---- words out, the stage refilled.  The fence orders the warp's accesses to the stage before the copy's
                // writes (they go through different proxies, and a read waits its turn in the load queue after it was issued).
                const int64_t extent = (int64_t)M * a.packed_stride * 4;
                if constexpr (StoresDirectly<B>::value) {
                    tma::fence_proxy_async();
                    __syncwarp();
                    copies.next(st);
                    if (t.valid > 0) store_words<B>(tile_words + t.row * B, words, a.wide_words != 0, a.packed, extent, a.status);
                } else {
                    __syncwarp();                // the warp has read all of its rows
                    uint32_t* out_words = reinterpret_cast<uint32_t*>(stage_ptr(warp, st));
                    // the staging area keeps the 16-byte phase of the output stream; whole quads move 16 bytes per
                    // lane, the ragged ends word by word
                    const int off = (int)(((int64_t)t.row0 * B) & 3);
                    uint32_t* aligned_dst = tile_words - off;
                    if (t.valid > 0) {
#pragma unroll
                        for (int i = 0; i < B; ++i) out_words[off + t.row * B + i] = words[i];
                    }
                    __syncwarp();
                    const int jend = off + t.span * B;
                    const int f0 = off ? 1 : 0, f1 = jend >> 2;          // full quads [f0, f1)
#pragma unroll
                    for (int i = 0; i < (8 * B + 31) / 32; ++i) {
                        const int q = lane + 32 * i;
                        if (q >= f0 && q < f1)
                            DQ_STORE(reinterpret_cast<uint4*>(aligned_dst) + q, reinterpret_cast<const uint4*>(out_words)[q],
                                     a.packed, extent, a.status);
                    }
                    if (off | (jend & 3)) {
                        if (off && lane >= off && lane < 4 && lane < jend)                                        // head
                            DQ_STORE(aligned_dst + lane, out_words[lane], a.packed, extent, a.status);
                        int ts = f1 * 4;                                                                          // tail
                        if (off && ts < 4) ts = 4;
                        if (lane < jend - ts) DQ_STORE(aligned_dst + (ts + lane), out_words[ts + lane], a.packed, extent, a.status);
                    }
                    tma::fence_proxy_async();
                    __syncwarp();
                    copies.next(st);
                }
                __syncwarp();
            }
            ++it;
        }
        if (timed_out) break;

        if constexpr (AVG) {
            if (t.valid > 0 && has_tile && !(B == 1 && a.update)) {
                float r[32];
#pragma unroll
                for (int q = 0; q < 16; ++q) unpack_pair(acc2[q], r[2 * q], r[2 * q + 1]);
                if (!t.regular) {
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (e >= t.valid) r[e] = 0.0f;
                }
                store_row(a.out + ((int64_t)t.row0 + t.row) * 32, r, a.update != 0, a.neg_lr, a.wide_out != 0, a.out, (int64_t)G * 128,
                          a.status);
            }
            pos += hop;
        } else {
            pos += hop;
            while (pos >= copies.positions) { pos -= copies.positions; ++m; }
            copies.queue0 = copies.queue1; copies.queue1 = copies.queue2; --copies.queued;
        }
    }
    if (bad) atomicOr(a.status, DQ_STAT_NONFINITE);
    if (timed_out || skip_all) {
        if (lane == 0) atomicOr(a.status, DQ_STAT_WAIT);
        // every copy the warp has issued and not seen land, the one whose wait ran out included, gets the
        // full limit before the CTA's shared memory is released
        if constexpr (MODE == kTeamBuckets) {
            for (int i = 0; i < kStages; ++i)
                if ((copies.flying >> i) & 1u) (void)tma::mbar_wait(stage_bar(warp, i), (copies.parities >> i) & 1u, a.wait);
        } else {
            for (uint32_t i = it; i < (uint32_t)(items - copies.left); ++i)
                (void)tma::mbar_wait(stage_bar(warp, (int)(i & 1u)), (i >> 1) & 1u, a.wait);
        }
    }
}

// The tensor table (true if it is in shared memory); behind it the CTA is in step.
__device__ __forceinline__ bool copy_table(const RoundArgs& a, const int table)
{
    const bool tbl_in_smem = a.v.n_seg > 1 && a.v.n_seg <= kMaxSmemSegs;
    if (tbl_in_smem) {
        int32_t* tbl_s = reinterpret_cast<int32_t*>(smem + table);
        for (int i = threadIdx.x; i < 3 * (a.v.n_seg + 1); i += kRoundThreads) tbl_s[i] = __ldg(a.v.seg_group0 + i);
    }
    __syncthreads();
    return tbl_in_smem;
}
// Barriers, tensor table, and the wait for the kernel before.
__device__ __forceinline__ bool set_up(const RoundArgs& a, const CUtensorMap& map)
{
    // (nothing up to the wait touches memory that an earlier kernel may still be writing)
    if (threadIdx.x == 0) {
        tma::prefetch_tensor_map(&map);
        for (int i = 0; i < kRoundWarps * kStages; ++i) tma::mbar_init(stage_bar(0, i), 1);
        tma::fence_barrier_init();
    }
    grid_dependency_wait();
    return copy_table(a, SmemMap::table);
}

template <int MODE>
__device__ __forceinline__ int warp_of_team(const RoundArgs& a)
{
    return MODE == kTeamBuckets ? (int)(threadIdx.x >> 5) & ((1 << (a.gpb_shift - 5)) - 1) : 0;
}
// The first two copies of a warp that will not look at them: the CTA's shared memory outlives them, or the call says that a
// wait ran out (beside what else is wrong with it).
template <int MODE, bool AVG>
__device__ __forceinline__ void drain_first(const WarpFetch<MODE, AVG>& copies)
{
    const RoundArgs& a = copies.tiles.a;
    const int issued = copies.items() - copies.left;
    bool lost = false;
#pragma unroll
    for (int st = 0; st < kStages; ++st) {
        if (MODE == kTeamBuckets ? ((copies.flying >> st) & 1u) != 0u : st < issued) {
            lost |= a.wait.lose_first != 0u;         // (test hook: the wait counts as lost, and the copy is waited for all the same)
            lost |= !tma::mbar_wait(stage_bar(threadIdx.x >> 5, st), 0u, a.wait);
        }
    }
    if (__any_sync(0xffffffffu, lost) && (threadIdx.x & 31) == 0) atomicOr(a.status, DQ_STAT_WAIT);
}

// Norms alone.  Bound by HBM, 4 bytes read per element.  Against a CTA-wide ring of 16 KB tiles with a barrier
// per tile (three CTAs of 128 threads per SM): ResNet-18 shape M = 8 72 -> 57 us (6.3 TB/s), VGG-16 shape M = 16,
// bucket 2048, 191 -> 150, text shape with its zero rows 407 -> 103, pieces of whole tensors 84 -> 60.
constexpr int kNormCtasPerSm = 6;
template <int MODE, bool LINF>
__global__ void __launch_bounds__(kRoundThreads, kNormCtasPerSm)
norms_kernel(const __grid_constant__ RoundArgs a, const __grid_constant__ CUtensorMap map)
{
    const bool tbl_in_smem = set_up(a, map);
    if (tma::smem_addr(smem) & 1023u) {          // the swizzled tiles need a 1024-byte aligned base
        if (threadIdx.x == 0) atomicOr(a.status, DQ_STAT_INTERNAL);
        return;
    }
    double square_sum = 0.0;
    TileMap<MODE> tiles(a, tbl_in_smem, SmemMap::table, warp_of_team<MODE>(a));
    WarpFetch<MODE, false> copies(tiles, &map);
    copies.next(0);
    copies.next(1);
    round_tiles<0, MODE, false, LINF>(a, tiles, copies, square_sum);
    if (a.with_rule)
        rule_at_end<kRoundThreads>(a.rule, square_sum, nullptr, 0, reinterpret_cast<double*>(smem + SmemMap::sums), a.dev_b, 0, a.status);
}

template <int MODE, bool AVG, bool LINF>
__global__ void __launch_bounds__(kRoundThreads, RoundShape<AVG>::ctas_per_sm)
round_kernel(const __grid_constant__ RoundArgs a, const __grid_constant__ CUtensorMap map)
{
    const bool tbl_in_smem = set_up(a, map);
    const int b = *reinterpret_cast<const volatile int32_t*>(a.dev_b);
    uint32_t trouble = 0;
    if (tma::smem_addr(smem) & 1023u) trouble = DQ_STAT_INTERNAL;          // the swizzled tiles need a 1024-byte aligned base
    auto look_at_b = [&] {
        if (b < 1 || b > DQ_MAX_BITS) trouble = DQ_STAT_BAD_BITS;
        else if ((int64_t)b * a.v.total_groups > a.packed_stride) trouble = DQ_STAT_CAPACITY;
    };
    auto give_up = [&] {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.status, (int)trouble);
        // nothing is written but the next b, which follows from the norms that are there
        if (a.with_rule)
            rule_at_end<kRoundThreads>(a.rule, 0.0, a.norms, (int64_t)a.M * a.v.nb, reinterpret_cast<double*>(smem + SmemMap::sums),
                                       a.dev_b, b, a.status);
    };
    double square_sum = 0.0;
    if constexpr (AVG && (MODE == kWarpBuckets || MODE == kTeamBuckets)) {
        if (!trouble) look_at_b();
        if (trouble) return give_up();
        switch (b) {
#define DQ_CASE(BB)                                                                          \
        case BB: {                                                                               \
            TileMap<MODE> tiles(a, tbl_in_smem, SmemMap::table, warp_of_team<MODE>(a));          \
            WarpFetch<MODE, AVG> copies(tiles, &map);                                            \
            copies.next(0);                                                                      \
            copies.next(1);                                                                      \
            round_tiles<BB, MODE, AVG, LINF>(a, tiles, copies, square_sum);                      \
            break;                                                                               \
        }
            DQ_CASE(1) DQ_CASE(2) DQ_CASE(3) DQ_CASE(4) DQ_CASE(5) DQ_CASE(6) DQ_CASE(7) DQ_CASE(8)
            DQ_CASE(9) DQ_CASE(10) DQ_CASE(11) DQ_CASE(12) DQ_CASE(13) DQ_CASE(14) DQ_CASE(15) DQ_CASE(16)
#undef DQ_CASE
            default: break;
        }
    } else {
        // The first copies are on their way before b is here and its code is fetched; a call that cannot run waits for
        // them.  Codes, b = 6, one worker (us): 16.8M elements 17.1 -> 15.6, 1M 3.7 -> 3.4.  (With the sums of the two modes
        // above there are no registers for what that keeps alive: ResNet-18 shape M = 8 78.0 us, 83.8 so.)
        if (trouble) return give_up();
        TileMap<MODE> tiles(a, tbl_in_smem, SmemMap::table, warp_of_team<MODE>(a));
        WarpFetch<MODE, AVG> copies(tiles, &map);
        copies.next(0);
        copies.next(1);
        look_at_b();
        if (trouble) {
            drain_first(copies);
            return give_up();
        }
        switch (b) {
#define DQ_CASE(BB) case BB: round_tiles<BB, MODE, AVG, LINF>(a, tiles, copies, square_sum); break;
            DQ_CASE(1) DQ_CASE(2) DQ_CASE(3) DQ_CASE(4) DQ_CASE(5) DQ_CASE(6) DQ_CASE(7) DQ_CASE(8)
            DQ_CASE(9) DQ_CASE(10) DQ_CASE(11) DQ_CASE(12) DQ_CASE(13) DQ_CASE(14) DQ_CASE(15) DQ_CASE(16)
#undef DQ_CASE
            default: break;
        }
    }
    if (a.with_rule)
        rule_at_end<kRoundThreads>(a.rule, square_sum, nullptr, 0, reinterpret_cast<double*>(smem + SmemMap::sums), a.dev_b, b, a.status);
}


// ---- rounds with few tiles: the CTA takes a tile through the workers together --------------------------
// A chunk is a tile position of up to four workers, a warp's stage each (with buckets of 2048, whose two tiles are two
// warps', the bucket of up to two workers).  First every warp takes the norm of its own tile, a lane a row (group), and
// leaves the scales of every row in shared memory.  Behind a barrier the CTA goes through the workers of the chunk, a
// thread an octet (eight elements, one Philox block) of the tile, two workers side by side, and keeps the octet's sums
// in registers from a position's first worker to its last.
// What bounds it: with a position per SM the chain of a chunk (20 tiles, M = 16, cycles: norm 710, codes of four workers 1090
// two by two, 1400 one after the other, two barriers 180; the rest copies and addresses), with many the instructions,
// 830 per tile and worker at b = 4 (2^19 elements, M = 8, set-up and the rule's end among them), 515 in a warp's own way:
// scales, notes and addresses come once per eight elements.  A capture, whose caches are cold, has waiting for instructions as its
// largest stall (2.9 of some 9 per issue, 0.25 by warps); with warm ones it is not measured.  Where the line between the two lies,
// and what both measured: dq_route.h.
// Five CTAs per SM (96 registers; buckets of 2048, l2, spill 632 bytes, the others next to nothing).  By five / four / six of them (us): bucket 512, 600k elements M = 8 b = 5 10.4 / 10.2 / 12.2
// (six spill); 610k, one turn of five, two of four, M = 8 b = 4 9.4 / 11.3; 1.3M M = 8 17.4 / 17.1 / 23.2; bucket 2048, 1.2M
// M = 16 31.4 / 29.6 / 38.1, 1.3M M = 8 21.6 / 23.0.  (Four for buckets of 2048 alone: 6 to 15 % less where the positions fill
// as many turns, 2 to 14 % more where they need another, 0.6M and 1.25M.)
constexpr int kTileCtasPerSm = 5;
constexpr int kSets = 2;                            // chunks in shared memory: the one at hand and one on its way
struct TileSmem {
    static constexpr int notes = kSets * kRoundWarps * kTileBytes;            // uint4[4]: worker_rounds, and whether all norms of the tile are plain
    static constexpr int scales = notes + kRoundWarps * 16;                   // float4[4][32]: scale of the codes, scale of the sums, twice each
    static constexpr int valid = scales + kRoundWarps * 512;                  // bytes[32], of an irregular tile
    static constexpr int slots = valid + 32;                                  // the teams' exchange slots
    static constexpr int sums = slots + 2 * kRoundWarps * 8;
    static constexpr int table = sums + kRoundWarps * 8 + 16;
};

// A row's scales, as they stand there: that of its codes is 0 and that of its sums finite.
__device__ __forceinline__ bool adds_zero(const ulonglong2 sc)
{
    return (uint32_t)sc.x == 0u && isfinite(__uint_as_float((uint32_t)sc.y));
}

// The warp's copies: its tile of every position and worker of the CTA, a chunk at a time, 16 bytes per lane and instruction
// straight to where a swizzled tensor copy would put them.  They complete as loads do: there is no barrier to poll, and
// WaitLimits does not apply (under its test hook a round is never sent here).  With one position per SM a chunk's chain is what counts, and
// a tensor copy costs that chain some 250 cycles to issue, 250 to find landed and 100 for the fence before its stage is refilled.
template <int MODE, int T>
struct TileFetch {
    static constexpr bool TEAM = MODE == kTeamBuckets;
    static constexpr int kWorkers = kRoundWarps / T;       // of a chunk
    TileMap<MODE>& tiles;
    int pos, m, left;                // next position and worker, positions not fetched yet
    uint32_t first;                  // where that position's tile lies

    __device__ __forceinline__ TileFetch(TileMap<MODE>& where, const int n_pos)
        : tiles(where), pos((int)blockIdx.x), m((int)(threadIdx.x >> 5) / T), left(n_pos),
          first(n_pos > 0 ? where.describe((int)blockIdx.x) : kNoTile)
    {
    }
    __device__ __forceinline__ void next(const int set)
    {
        if (left > 0) {
            const RoundArgs& a = tiles.a;
            if (m < a.M && (!TEAM || first != kNoTile)) {
                const int lane = threadIdx.x & 31, at = lane >> 3;                      // row of the first four, piece lane & 7
                const int row0 = MODE == kGivenNorms ? pos * 32 : (int)(first & 0x7fffffffu);
                const float* src = a.grads + (int64_t)m * a.grad_stride + (int64_t)(row0 + at) * 32 + (lane & 7) * 4;
                const uint32_t dst = tma::smem_addr(smem) + (set * kRoundWarps + (threadIdx.x >> 5)) * kTileBytes + at * 128;
                const uint32_t even = (uint32_t)((lane & 7) ^ at) << 4, odd = even ^ 64u;       // swizzled piece
                const int rows = a.v.total_groups - row0 - at;                          // (rows behind the last arrive as zeros)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int bytes = 4 * i < rows ? 16 : 0;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + i * 512 + (i % 2 ? odd : even)),
                                 "l"(bytes ? src + i * 128 : a.grads), "r"(bytes)
                                 : "memory");
                }
            }
            m += kWorkers;
            const int mine = (int)(threadIdx.x >> 5) / T;
            if (m - mine >= a.M) {
                m = mine;
                pos += (int)gridDim.x;
                if (--left > 0) first = tiles.describe(pos);
            }
        }
        // (an empty group where nothing is left to copy: the wait counts groups)
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // The chunk before the last one requested is there.
    __device__ __forceinline__ void wait() const
    {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
    }
    __device__ __forceinline__ void drain() const { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
};

template <int B, int MODE, bool LINF, int T>
__device__ __forceinline__ void tile_rounds(const RoundArgs& a, TileMap<MODE>& tiles, TileFetch<MODE, T>& copies, const int n_pos,
                                            double& square_sum)
{
    using Join = typename JoinOp<LINF>::type;
    constexpr bool ODD = MODE == kOddBuckets, TEAM = MODE == kTeamBuckets;
    constexpr int T_shift = T - 1;                  // (T is 1 or 2)
    constexpr int kWorkers = kRoundWarps / T;       // of a chunk
    constexpr int s = (1 << (B - 1)) - 1;
    const float sf = (float)s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int M = a.M, nb = a.v.nb;
    const int sub = warp & (T - 1), mine = warp / T;
    float2* slots = reinterpret_cast<float2*>(smem + TileSmem::slots);
    uint4* notes = reinterpret_cast<uint4*>(smem + TileSmem::notes);
    float4* scales = reinterpret_cast<float4*>(smem + TileSmem::scales);
    unsigned char* valids = smem + TileSmem::valid;
    const int hop = (int)gridDim.x;

    const float to_unit = (B <= 1) ? 0.0f : __fdiv_rn(1.0f, (float)s * (float)M);          // 1 / (s * M)
    bool bad = false;
    uint32_t exchanges = 0;

    // the thread's octet of a tile: row, place in the row, and where its two 16-byte pieces stand in a stage
    const int orow = threadIdx.x >> 2, oq = threadIdx.x & 3;
    const uint32_t opiece = (uint32_t)(orow * 128) + ((uint32_t)((2 * oq) ^ (orow & 7)) << 4);
    const int64_t extent = (int64_t)M * a.packed_stride * 4;

    uint32_t it = 0;
    int pos = (int)blockIdx.x;
    for (int ip = 0; ip < n_pos; ++ip, pos += hop) {
        // ---- the position: this lane's row of it, and the thread's octets
        TilePos t;
        int row0, span;                              // of the whole position
        {
            const uint32_t desc = tiles.describe(pos);
            if constexpr (TEAM) {
                const int local = pos - tiles.c_b0;
                row0 = tiles.c_g0 + (local << (T_shift + 5));
                const int rest = tiles.c_n - (local << (T_shift + 10));
                const int len = rest < T * 1024 ? rest : T * 1024;
                span = (len + 31) >> 5;
                const int v = len - sub * 1024 - lane * 32;
                t.row = lane; t.bucket = pos; t.writes = sub == 0 && lane == 0; t.len = len;
                t.valid = v < 0 ? 0 : (v > 32 ? 32 : v);
                t.row0 = desc == kNoTile ? -1 : row0 + 32 * sub;
                t.regular = (desc >> 31) != 0;
                t.span = 0;
            } else {
                t = tiles.locate(pos, desc);
                row0 = t.row0;
                span = t.span;
                if (!t.regular && t.valid > 0) valids[t.row] = (unsigned char)t.valid;       // (all warps write the same)
            }
        }
        const bool has_tile = !TEAM || t.row0 >= 0;
        const uint32_t own = (uint32_t)(t.row * 128 + ((t.row & 7) << 4));
        float* norm_ptr = a.norms + (int64_t)mine * nb + t.bucket;
        float given = 0.0f;
        if constexpr (MODE == kGivenNorms) {
            if (mine < M && t.valid > 0) given = load_norm_early(norm_ptr);
        }
        unsigned char* words = reinterpret_cast<unsigned char*>(a.packed + (int64_t)row0 * B) +
                               (OctetDirect<B>::value ? (int)threadIdx.x * B : (warp * 8 * B + lane) * 4);
        OctetRounds oct[T];
        uint64_t sums[T][4];
#pragma unroll
        for (int k = 0; k < T; ++k) {
            oct[k] = octet_rounds((uint32_t)(row0 + 32 * k) * 4u + threadIdx.x, a.step, a.keys);
#pragma unroll
            for (int q = 0; q < 4; ++q) sums[k][q] = 0ull;
        }

#pragma unroll 1
        for (int m0 = 0; m0 < M; m0 += kWorkers, ++it) {
            const int set = (int)(it & 1u);
            // ---- the norm of the warp's own tile
            copies.wait();
            if (m0 + mine < M) {
                const uint32_t row = (uint32_t)((set * kRoundWarps + warp) * kTileBytes) + own;
                float nrm = 0.0f, inv = 0.0f;
                bool plain = false;
                if constexpr (MODE == kGivenNorms || ODD) {
                    if (!t.regular) (void)end_row<LINF>(row, t.valid);
                }
                if constexpr (MODE == kGivenNorms) {
                    nrm = given;
                    inv = inv_scale_normal(sf, nrm);
                    plain = !__any_sync(0xffffffffu, t.valid > 0 && !norm_is_plain(nrm));
                    if (!plain) {
                        inv = inv_scale(sf, nrm);
                        clear_nonfinite_row<true>(row, t.valid, nrm);
                    }
                    if (t.writes) square_sum = fma((double)nrm, (double)nrm, square_sum);
                    if (m0 + mine + kWorkers < M && t.valid > 0) given = load_norm_early(norm_ptr + (int64_t)kWorkers * nb);
                } else {
                    bool lost = false;           // (of teams; not here)
                    float v;
                    if constexpr (ODD) {
                        v = odd_bucket_sums<LINF>(row - own, t.row, t.len, tiles.gpb, tiles.R, tiles.r);
                    } else {
                        v = LINF ? row_max(row) : row_sum_squares(row);
                        if (!t.regular) {
                            const float end = has_tile ? end_row<LINF>(row, t.valid) : 0.0f;
                            if (t.valid != 32) v = end;
                        }
                        v = join_team<MODE>(join_lanes<MODE>(v, tiles.gpb, Join{}), slots, T_shift, exchanges, true, lost, Join{});
                    }
                    nrm = LINF ? v : sqrt_normal(v);
                    inv = inv_scale_normal(sf, nrm);
                    plain = !__any_sync(0xffffffffu, has_say<MODE>(t) && (LINF ? !norm_is_plain(v) : !l2_sum_in_range(v)));
                    if (!plain) {
                        if constexpr (LINF) {
                            clear_nonfinite_row<true>(row, t.valid, nrm);
                        } else if constexpr (ODD) {
                            nrm = rare_norm_odd<true>(row - own, t.row, t.len, tiles.gpb, tiles.R, tiles.r, v, nrm, row, t.valid);
                        } else {
                            nrm = rare_norm<MODE, true>(row, t.valid, tiles.gpb, slots, T_shift, exchanges, v, nrm);
                            exchanges += 2;
                        }
                        inv = inv_scale(sf, nrm);
                        bad |= t.writes && !isfinite(nrm);
                    }
                    if (t.writes) {
                        DQ_STORE(norm_ptr, nrm, a.norms, (int64_t)M * nb * 4, a.status);
                        square_sum = fma((double)nrm, (double)nrm, square_sum);
                    }
                }
                norm_ptr += (int64_t)kWorkers * nb;
                if (t.valid > 0) scales[warp * 32 + t.row] = make_float4(inv, inv, nrm * to_unit, nrm * to_unit);
                uint4 note = worker_rounds((uint32_t)(m0 + mine) + a.worker0, a.keys);
                note.w = plain ? 1u : 0u;
                if (lane == 0) notes[warp] = note;
            }
            __syncthreads();

            // ---- the codes of the chunk, a thread an octet of each tile
            const int slots_used = (M - m0 < kWorkers ? M - m0 : kWorkers) * T;
            auto emit = [&](const int slot, const int k, const uint32_t (&w)[OctetWords<B>::n], unsigned char* to) {
                if constexpr (OctetDirect<B>::value) {
                    if (32 * k + orow < span) store_octet<B>(to, w, a.packed, extent, a.status);
                } else {
                    // through the warp's eight rows of the stage, which it has read
                    unsigned char* staged = smem + (set * kRoundWarps + slot) * kTileBytes + warp * 1024;
                    __syncwarp();
                    stage_octet<B>(staged + lane * B, w);
                    __syncwarp();
                    const int rows = span - 32 * k - warp * 8;
                    const int n = (rows > 8 ? 8 : rows) * B;
#pragma unroll
                    for (int q = 0; q < (8 * B + 31) / 32; ++q)
                        if (lane + 32 * q < n)
                            DQ_STORE(reinterpret_cast<uint32_t*>(to) + 32 * q, reinterpret_cast<const uint32_t*>(staged)[lane + 32 * q],
                                     a.packed, extent, a.status);
                }
            };
            // N tiles side by side: two workers', or both tiles of a worker's bucket
            auto encode = [&](const int j, const int k0, const auto& note, auto count) {
                constexpr int N = decltype(count)::value;
                uint32_t draws[N][4];
                ulonglong2 lo[N], hi[N], sc[N];
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    const unsigned char* stage = smem + (set * kRoundWarps + j + n) * kTileBytes;
                    sc[n] = *reinterpret_cast<const ulonglong2*>(scales + (j + n) * 32 + orow);
                    lo[n] = *reinterpret_cast<const ulonglong2*>(stage + opiece);
                    hi[n] = *reinterpret_cast<const ulonglong2*>(stage + (opiece ^ 16u));
                    third_round(draws[n], oct[T == 1 ? 0 : k0 + n], note[n]);
                }
                philox_rounds<2>(draws, a.keys);
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    uint32_t ft[8], fu[8], w[OctetWords<B>::n];
                    const int k = T == 1 ? 0 : k0 + n;
                    octet_codes<B, true>(lo[n], hi[n], sc[n].x, sc[n].y, sums[k], draws[n], ft, fu);
                    pack_octet<B>(w, ft, fu);
                    emit(j + n, k, w, words + (T == 1 ? n * (a.packed_stride * 4) : k * (128 * B)));
                }
            };
            if constexpr (B == 1) {
                const uint32_t w[1] = {0u};
                for (int j = 0; j < slots_used; j += T, words += a.packed_stride * 4)
                    for (int k = 0; k < T; ++k)
                        if (32 * k < span) emit(j + k, k, w, words + k * (128 * B));
            } else {
                int j = 0;
#pragma unroll 1
                while (j < slots_used) {
                    const uint4 note[2] = {notes[j], notes[j + 1 < kRoundWarps ? j + 1 : j]};
                    if (j + 1 < slots_used && (T == 1 || span > 32) && (note[0].w & note[1].w) != 0u) {
                        encode(j, 0, note, std::integral_constant<int, 2>{});
                        j += 2;
                        words += (2 / T) * (a.packed_stride * 4);
                        continue;
                    }
#pragma unroll
                    for (int k = 0; k < T; ++k) {
                        if (T > 1 && 32 * k >= span) break;
                        const ulonglong2 sc = *reinterpret_cast<const ulonglong2*>(scales + (j + k) * 32 + orow);
                        if (note[k].w == 0u && __all_sync(0xffffffffu, adds_zero(sc) || 32 * k + orow >= span)) {
                            // zero buckets (sparse gradients are full of them): every code is s, whatever the draw, and adds 0
                            uint32_t w[OctetWords<B>::n];
                            zero_octet_words<B>(w);
                            emit(j + k, k, w, words + k * (128 * B));
                        } else {
                            const uint4 one[1] = {note[k]};
                            encode(j + k, k, one, std::integral_constant<int, 1>{});
                        }
                    }
                    j += T;
                    words += a.packed_stride * 4;
                }
            }
            if (m0 + kWorkers >= M && !(B == 1 && a.update)) {
                // ---- the position's sums
#pragma unroll
                for (int k = 0; k < T; ++k) {
                    const int at = 32 * k + orow;
                    if (at < span) {
                        float r[8];
#pragma unroll
                        for (int q = 0; q < 4; ++q) unpack_pair(sums[k][q], r[2 * q], r[2 * q + 1]);
                        const int valid = (TEAM ? t.len - at * 32 : (t.regular ? 32 : (int)valids[orow])) - 8 * oq;
                        if (valid < 8) {
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                if (q >= valid) r[q] = 0.0f;
                        }
                        store_sums(a.out + ((int64_t)row0 + at) * 32 + 8 * oq, r, a.update != 0, a.neg_lr, a.wide_out != 0, a.out,
                                   (int64_t)a.v.total_groups * 128, a.status);
                    }
                }
            }
            __syncthreads();
            copies.next(set);
        }
    }
    copies.drain();
    if (bad) atomicOr(a.status, DQ_STAT_NONFINITE);
}

template <int MODE, bool LINF, int T>
__global__ void __launch_bounds__(kRoundThreads, kTileCtasPerSm)
tile_round_kernel(const __grid_constant__ RoundArgs a)
{
    grid_dependency_wait();
    const int b = *reinterpret_cast<const volatile int32_t*>(a.dev_b);
    const bool tbl_in_smem = copy_table(a, TileSmem::table);
    double* part = reinterpret_cast<double*>(smem + TileSmem::sums);
    // The first copies are on their way before b is here and its code is fetched; a call that cannot run waits for them.
    // Every CTA takes every hop-th position, `each` of them, the first `extra` CTAs one more.
    const int n_pos = (int)(a.each + (blockIdx.x < a.extra ? 1u : 0u));
    TileMap<MODE> tiles(a, tbl_in_smem, TileSmem::table, (int)(threadIdx.x >> 5) & (T - 1));
    TileFetch<MODE, T> copies(tiles, n_pos);
    copies.next(0);
    copies.next(1);
    uint32_t trouble = 0;
    if (b < 1 || b > DQ_MAX_BITS) trouble = DQ_STAT_BAD_BITS;
    else if ((int64_t)b * a.v.total_groups > a.packed_stride) trouble = DQ_STAT_CAPACITY;
    if (trouble) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.status, (int)trouble);
        copies.drain();
        // nothing is written but the next b, which follows from the norms that are there
        if (a.with_rule) rule_at_end<kRoundThreads>(a.rule, 0.0, a.norms, (int64_t)a.M * a.v.nb, part, a.dev_b, b, a.status);
        return;
    }
    double square_sum = 0.0;
    switch (b) {
#define DQ_CASE(BB) case BB: tile_rounds<BB, MODE, LINF, T>(a, tiles, copies, n_pos, square_sum); break;
        DQ_CASE(1) DQ_CASE(2) DQ_CASE(3) DQ_CASE(4) DQ_CASE(5) DQ_CASE(6) DQ_CASE(7) DQ_CASE(8)
        DQ_CASE(9) DQ_CASE(10) DQ_CASE(11) DQ_CASE(12) DQ_CASE(13) DQ_CASE(14) DQ_CASE(15) DQ_CASE(16)
#undef DQ_CASE
        default: break;
    }
    if (a.with_rule) rule_at_end<kRoundThreads>(a.rule, square_sum, nullptr, 0, part, a.dev_b, b, a.status);
}

// units: of work per CTA: warps, teams, or the CTA itself
template <class Map, class... Maps>
int launch_persistent(void (*kernel)(RoundArgs, Maps...), int ctas_per_sm, int units, RoundArgs a, int n_seg, int64_t entries,
                      cudaStream_t st, const Maps&... maps)
{
    size_t smem_need = (size_t)Map::table;
    if (n_seg > 1 && n_seg <= kMaxSmemSegs) smem_need += (size_t)3 * (n_seg + 1) * 4;
    // (the limit of the largest table, whatever this one's size: with each call's own, another thread's call for a
    // smaller layout can narrow it again before this launch, which then fails)
    constexpr int kLargest = Map::table + 3 * (kMaxSmemSegs + 1) * 4;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLargest) != cudaSuccess) {
        (void)cudaGetLastError();
        return DQ_ERR_CUDA;
    }
    int64_t blocks = (int64_t)dq_sm_count() * ctas_per_sm;
    if (blocks * units > entries) blocks = (entries + units - 1) / units;
    a.each = (uint32_t)(entries / (blocks * units));
    a.extra = (uint32_t)(entries - (int64_t)a.each * blocks * units);
    dq_launch(kernel, dim3((unsigned)blocks), dim3(kRoundThreads), smem_need, st, a, maps...);
    return cudaGetLastError() == cudaSuccess ? DQ_OK : DQ_ERR_CUDA;
}

template <int MODE>
int units_per_cta(const RoundArgs& a)
{
    return MODE == kTeamBuckets ? kRoundWarps >> (a.gpb_shift - 5) : kRoundWarps;
}

}  // namespace

template <int MODE, bool LINF>
int dq_launch_norms(const RoundArgs& a, const CUtensorMap& map, int n_seg, int64_t entries, cudaStream_t st)
{
    return launch_persistent<SmemMap>(norms_kernel<MODE, LINF>, kNormCtasPerSm, units_per_cta<MODE>(a), a, n_seg, entries, st, map);
}
template <int MODE, bool AVG, bool LINF>
int dq_launch_round(const RoundArgs& a, const CUtensorMap& map, int n_seg, int64_t entries, cudaStream_t st)
{
    return launch_persistent<SmemMap>(round_kernel<MODE, AVG, LINF>, RoundShape<AVG>::ctas_per_sm, units_per_cta<MODE>(a), a,
                                      n_seg, entries, st, map);
}
template <int MODE, bool LINF>
int dq_launch_tile_round(const RoundArgs& a, int n_seg, int64_t entries, cudaStream_t st)
{
    constexpr int T = MODE == kTeamBuckets ? 2 : 1;
    if (MODE == kTeamBuckets && a.gpb_shift != 6) return DQ_ERR_RANGE;          // (the kernel's teams are pairs; see dq_cta_form)
    return launch_persistent<TileSmem>(tile_round_kernel<MODE, LINF, T>, kTileCtasPerSm, 1, a, n_seg, entries, st);
}

#endif  // DQ_ROUND_KERNELS
