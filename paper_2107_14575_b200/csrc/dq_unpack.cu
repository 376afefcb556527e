// dq_unpack_dequant_average: the server's "Average" step of Algorithm 1 on
// packed codes: out_j = (1/M) sum_m (code_m - s) * norm_m / s  (Eq. 5 inverted;
// a code holds s + sgn * level).
//
// Every WARP is a pipeline of its own.  It takes tiles of 32 groups (one group = 32 padded elements =
// one lane, which keeps its 32 fp32 sums in registers) through the M workers, up to eight workers
// at a time: their words of the tile are as many linear bulk copies, one per lane, into one of two
// 4 KB stages, so that the copies of the next workers travel while these are decoded.  The norms of the
// next workers are requested before the wait.  A code is decoded where it stands in its word (mask under
// the exponent of 2^23, subtract 2^23 + s: see accumulate_pair) and accumulated with one FMA; the power of two
// its position carries is removed once per element after the last worker.  The 32 rows of sums go through a
// swizzled 4 KB tile of the warp and leave with one bulk tensor store (straight from registers, 32 bytes a
// lane, every store touched 32 lines: one worker, 2^25 elements, b = 4 37 us against 30).
// HBM traffic per output element: M*b/8 bytes read, 4 written.  Bound by the logic pipe for small b
// (one half-rate operation per code) and the issue of about 100 instructions per lane, worker and group,
// by HBM from b = 8 on.  Measured, d = 8.4M, M = 16: b = 4 21.0 us (4.8 TB/s), b = 8 29.6 us (5.7), b = 16 51.7 us (5.8);
// one worker, 2^25 elements, b = 4 28.2 us (5.3).  (Codes taken two at a time as fp16 pairs,
// for half the logic operations, and widened by mixed-precision adds: 9 % slower at b = 4.)
//
// dq_unpack_average_update ends with the parameter update of Algorithm 1 instead, x <- x - eta * average;
// the averaged gradient itself never reaches memory (M*b/8 + 4 bytes read and 4 written per element).
#include "dq_common.cuh"
#include "dq_device.cuh"
#include "dq_tma.cuh"

namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr int kCtasPerSm = 4;
constexpr int kStages = 2;
constexpr int kStageBytes = 4096;
constexpr int kMaxChunk = 8;                  // workers per stage at most
constexpr int kMaxSmemSegs = 1023;

// Dynamic shared memory, addressed only through this symbol so that every access compiles to a
// shared-memory instruction: the warps' output tiles (1024-byte aligned for the swizzle), their stages,
// the barriers of stages and of the tiles of x, the tensor table.
extern __shared__ __align__(1024) unsigned char smem[];
constexpr int kOutBytes = 32 * 128;
constexpr int kStageOffset = kWarps * kOutBytes;
constexpr int kBarOffset = kStageOffset + kWarps * kStages * kStageBytes;
constexpr int kTblOffset = kBarOffset + kWarps * (kStages + 1) * 8;

__device__ __forceinline__ uint64_t* stage_bar(int warp, int st)
{
    return reinterpret_cast<uint64_t*>(smem + kBarOffset) + warp * kStages + st;
}
__device__ __forceinline__ uint32_t* stage_words(int warp, int st)
{
    return reinterpret_cast<uint32_t*>(smem + kStageOffset + (warp * kStages + st) * kStageBytes);
}
__device__ __forceinline__ uint64_t* x_bar(int warp) { return stage_bar(kWarps, 0) + warp; }

struct AverageArgs {
    LayoutView v;
    const uint32_t* packed;
    int64_t packed_stride;
    const float* norms;
    const int32_t* dev_b;
    float* out;
    int32_t* status;
    int32_t M;
    uint32_t div_magic;
    int32_t div_shift;
    uint32_t magic;               // 0x4B000000, kept out of the compiler's sight (see and_or)
    int32_t update;               // out <- out + neg_lr * average instead of out <- average
    uint32_t each, extra;         // tiles per warp: `each`, one more for the first `extra` of them
    float neg_lr;                 // -eta of the parameter update
    WaitLimits wait;
};

__device__ __forceinline__ uint32_t div_gpb(const AverageArgs& a, uint32_t n)
{
    if (a.div_shift >= 0) return n >> a.div_shift;
    return (uint32_t)(((uint64_t)n * a.div_magic) >> 33);     // exact for n < 2^26, divisor <= 128
}

// A norm load that stays where it is written: the compiler may not sink it past the barrier wait and
// the decode that follow (a volatile statement keeps its place among the other volatile statements),
// so the value is on its way while the unit is decoded.
__device__ __forceinline__ float load_norm_early(const float* p)
{
    float x;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(x) : "l"(p));
    return x;
}

// workers per stage: as many as fit with 32 groups of B words each, at most kMaxChunk
template <int B>
struct ChunkOf {
    static constexpr int fit = kStageBytes / (128 * B);
    static constexpr int value = fit < 1 ? 1 : (fit > kMaxChunk ? kMaxChunk : fit);
};

template <int B>
__device__ __forceinline__ void load_words(const uint32_t* __restrict__ src, uint32_t (&wd)[B])
{
    if constexpr (B % 4 == 0) {
#pragma unroll
        for (int i = 0; i < B / 4; ++i) {
            const uint4 t = reinterpret_cast<const uint4*>(src)[i];
            wd[4 * i] = t.x; wd[4 * i + 1] = t.y; wd[4 * i + 2] = t.z; wd[4 * i + 3] = t.w;
        }
    } else if constexpr (B % 2 == 0) {
#pragma unroll
        for (int i = 0; i < B / 2; ++i) {
            const uint2 t = reinterpret_cast<const uint2*>(src)[i];
            wd[2 * i] = t.x; wd[2 * i + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < B; ++i) wd[i] = src[i];
    }
}

// The 32 sums of a group live in 16 register pairs (elements 2q and 2q + 1), see accumulate_pair.
template <int B, int Q>
struct AccumulateAll {
    static __device__ __forceinline__ void run(uint64_t (&acc2)[16], const uint32_t (&wd)[B], const uint32_t (&hi)[B],
                                               const uint64_t scale2, const uint32_t magic)
    {
        acc2[Q] = accumulate_pair<B, Q>(acc2[Q], wd, hi, scale2, magic);
        AccumulateAll<B, Q + 1>::run(acc2, wd, hi, scale2, magic);
    }
};
template <int B>
struct AccumulateAll<B, 16> {
    static __device__ __forceinline__ void run(uint64_t (&)[16], const uint32_t (&)[B], const uint32_t (&)[B], const uint64_t,
                                               const uint32_t) {}
};

// The upper halves of the words whose codes need them (see CodePos) come straight from shared
// memory as 16-bit loads, two bytes into the word: the load pipe has room, the logic pipe, which a
// shift would use, is the busiest one of this kernel.
template <int B, int W>
struct UpperHalves {
    static __device__ __forceinline__ void run(const uint32_t* __restrict__ src, uint32_t (&hi)[B])
    {
        if constexpr (NeedsUpper<B, W>::value) hi[W] = reinterpret_cast<const uint16_t*>(src)[2 * W + 1];
        else hi[W] = 0u;
        UpperHalves<B, W + 1>::run(src, hi);
    }
};
template <int B>
struct UpperHalves<B, B> {
    static __device__ __forceinline__ void run(const uint32_t* __restrict__, uint32_t (&)[B]) {}
};

// removes the power of two each element's decoded value carried
template <int B, int E>
struct Normalise {
    static __device__ __forceinline__ void run(float (&acc)[32])
    {
        constexpr int k = CodePos<B, E>::k;
        if constexpr (k != 0) acc[E] *= __uint_as_float((uint32_t)(127 - k) << 23);
        Normalise<B, E + 1>::run(acc);
    }
};
template <int B>
struct Normalise<B, 32> {
    static __device__ __forceinline__ void run(float (&)[32]) {}
};

// The end of a tile: the powers of two removed, padding zeroed, the rows through the warp's output tile.
// kOutOfRange (nothing stored): some lane says so of its sums.  kLost: the tile of x did not arrive.
enum TileEnd { kDone, kOutOfRange, kLost };
template <int B>
__device__ __forceinline__ TileEnd finish_tile(const AverageArgs& a, const CUtensorMap* out_map, unsigned char* out_tile,
                                            const uint64_t (&acc2)[16], const int tile, const int valid, const bool out_of_range,
                                            uint64_t* xbar, const uint32_t x_parity)
{
    const int lane = threadIdx.x & 31;
    // (B = 1: s = 0, every value is 0, and an update by 0 leaves x as it is)
    if (!(B == 1 && a.update)) {
        if (B > 1 && __any_sync(0xffffffffu, out_of_range)) return kOutOfRange;
        float acc[32];
#pragma unroll
        for (int q = 0; q < 16; ++q) unpack_pair(acc2[q], acc[2 * q], acc[2 * q + 1]);
        Normalise<B, 0>::run(acc);
        if (valid < 32) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
                if (e >= valid) acc[e] = 0.0f;
        }
        if (a.update) {
            // nothing is stored from a tile whose parameters did not arrive
            if (!__all_sync(0xffffffffu, tma::mbar_wait(xbar, x_parity, a.wait))) return kLost;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float4* p = reinterpret_cast<float4*>(out_tile + tma::swizzle128(lane, c));
                const float4 x = *p;
                *p = make_float4(fmaf(a.neg_lr, acc[4 * c], x.x), fmaf(a.neg_lr, acc[4 * c + 1], x.y),
                                 fmaf(a.neg_lr, acc[4 * c + 2], x.z), fmaf(a.neg_lr, acc[4 * c + 3], x.w));
            }
        } else {
            if (lane == 0) tma::store_wait_read();
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 8; ++c)
                *reinterpret_cast<float4*>(out_tile + tma::swizzle128(lane, c)) =
                    make_float4(acc[4 * c], acc[4 * c + 1], acc[4 * c + 2], acc[4 * c + 3]);
        }
        tma::fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
            tma::store_tile_2d(out_map, out_tile, 0, tile * 32);          // (rows outside the layout are clipped)
            tma::store_commit();
        }
    }
    return kDone;
}
// The start of a tile of the update: the tile before must have left the warp's output tile; the tile of x
// travels while the codes are decoded.
__device__ __forceinline__ void request_x(const CUtensorMap* out_map, unsigned char* out_tile, const int tile, uint64_t* xbar)
{
    tma::store_wait_read();
    tma::mbar_expect_tx(xbar, kOutBytes);
    tma::load_tile_2d(out_tile, out_map, xbar, 0, tile * 32);
}
// Bucket and valid elements of this lane's group in a tile (valid 0: the group lies beyond the layout).
__device__ __forceinline__ void locate_group(const AverageArgs& a, const bool tbl_in_smem, const int tile, int& bucket, int& valid)
{
    const int32_t* tbl_s = reinterpret_cast<const int32_t*>(smem + kTblOffset);
    auto tbl = [&](int i) -> int { return tbl_in_smem ? tbl_s[i] : __ldg(a.v.seg_group0 + i); };
    const int n1 = a.v.n_seg + 1;
    const int g = tile * 32 + (threadIdx.x & 31);
    int seg = 0;
    if (a.v.n_seg > 1) seg = last_not_above_by_warp(tile * 32, a.v.n_seg, tbl);
    bucket = 0;
    valid = 0;
    if (g >= a.v.total_groups) return;
    int local = g, n = a.v.seg0_elems, b0 = 0;
    if (a.v.n_seg > 1) {
        while (g >= tbl(seg + 1)) ++seg;
        local = g - tbl(seg);
        b0 = tbl(n1 + seg);
        n = tbl(2 * n1 + seg);
    }
    bucket = b0 + (int)div_gpb(a, (uint32_t)local);
    const int left = n - local * 32;
    valid = left < 32 ? left : 32;
}

// Tiles `tile`, `tile` + `hop`, ... (n of them) with every code shifted down and without the power of two of its
// position, which takes sums of 2^106 and more out of the fp32 range: the same values, order and roundings as in
// the one-pass kernels.  The warp ends here with the first tile that has such norms (an infinity or a NaN among them); what
// it has in flight has landed by then.  Out of line, with plain loads and stores.
__device__ __noinline__ void average_tiles_plain(const AverageArgs& a, const bool tbl_in_smem, const int B, int tile, const int hop, int n)
{
    const int lane = threadIdx.x & 31;
    const int s = (1 << (B - 1)) - 1;
    const float unit = __fdiv_rn(1.0f, (float)s * (float)a.M);
    for (; n > 0; --n, tile += hop) {
        int bucket, valid;
        locate_group(a, tbl_in_smem, tile, bucket, valid);
        if (valid == 0) continue;
        const int group = tile * 32 + lane;
        const uint32_t* words = a.packed + (int64_t)group * B;
        const float* norm = a.norms + bucket;
        float sums[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) sums[e] = 0.0f;
#pragma unroll 1
        for (int m = 0; m < a.M; ++m, words += a.packed_stride, norm += a.v.nb) {
            const float scale = __ldg(norm) * unit;
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const int i = e * B >> 5, sh = e * B & 31;
                const uint32_t lo = __ldg(words + i), hi = sh + B > 32 ? __ldg(words + i + 1) : 0u;
                const int code = (int)(__funnelshift_r(lo, hi, sh) & ((1u << B) - 1u));
                sums[e] = fmaf((float)(code - s), scale, sums[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < 32; ++e)
            if (e >= valid) sums[e] = 0.0f;
        store_row(a.out + (int64_t)group * 32, sums, a.update != 0, a.neg_lr, false, a.out, (int64_t)a.v.total_groups * 128, a.status);
    }
}

// ---- b = 2, 3 and workers in whole eights: words straight into registers --------------------------
// A lane's words of a worker are one to three loads that neighbouring lanes coalesce.  Eight workers' words and
// norms wait in registers; as soon as one has been decoded, its registers are the target of the load for the worker
// eight further on (of the next tile, when this one's are through), so nothing is moved, staged or waited for.
// Measured, by asynchronous copies / direct (us): 2^25 elements M = 8 b = 2 45.0 / 41.2, b = 3 49.2 / 46.6, M = 16 72.2 /
// 69.5 and 77.2 / 74.1; 2^24 elements M = 24 52.3 / 51.8 and 55.9 / 54.1, M = 64 123.4 / 124.9 and 131.7 / 129.9; d = 4.2M M = 8
// 7.8 / 8.2 and 8.3 / 8.8.  A last group of fewer than eight costs more than it saves: 2^24 elements M = 20 47.4 / 51.4 and
// 50.7 / 55.2; and at b = 4 so do the wider loads: M = 32 68.9 / 73.7.
template <int B>
struct DirectWords {
    static constexpr bool value = B == 2 || B == 3;
    static constexpr int workers = 8;
};
template <int B>
__device__ __forceinline__ void request_words(const uint32_t* p, uint32_t (&w)[B])
{
    if constexpr (B == 2) {
        asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p));
    } else {
#pragma unroll
        for (int i = 0; i < B; ++i) asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(w[i]) : "l"(p + i));
    }
}
// Whether a lane's 32 sums are finite: 0 times each of them adds up to 0.
__device__ __forceinline__ bool sums_finite(const uint64_t (&acc2)[16])
{
    uint64_t t = 0ull;
#pragma unroll
    for (int q = 0; q < 16; ++q) t = fma_pair(acc2[q], 0ull, t);
    float lo, hi;
    unpack_pair(t, lo, hi);
    return lo + hi == 0.0f;
}
template <int B>
__device__ __forceinline__ void average_tiles_direct(const AverageArgs& a, const CUtensorMap* out_map, const bool tbl_in_smem)
{
    constexpr int s = (1 << (B - 1)) - 1;
    constexpr int MC = DirectWords<B>::workers;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int G = a.v.total_groups, M = a.M, nb = a.v.nb;
    const float unit = __fdiv_rn(1.0f, (float)s * (float)M);      // 1 / (s * M)
    const uint32_t magic = a.magic;
    const uint32_t id = blockIdx.x * kWarps + warp;
    const int hop = (int)(gridDim.x * kWarps);
    const int n_tiles = (int)(a.each + (id < a.extra ? 1u : 0u));
    if (n_tiles == 0) return;
    if (a.wait.lose_first != 0u) {               // (test hook; there is no copy in flight yet)
        if (lane == 0) atomicOr(a.status, DQ_STAT_WAIT);
        return;
    }
    unsigned char* out_tile = smem + warp * kOutBytes;

    int tile = (int)id, bucket, valid;
    locate_group(a, tbl_in_smem, tile, bucket, valid);
    // words and norm of worker m for this lane's group of a tile (a group beyond the layout reads the last one)
    auto words_of = [&](int tl, int m) -> const uint32_t* {
        const int g = tl * 32 + lane;
        return a.packed + (int64_t)m * a.packed_stride + (int64_t)(g < G ? g : G - 1) * B;
    };
    uint32_t wd[MC][B];
    float nrm[MC];
    {
        const uint32_t* p = words_of(tile, 0);
        const float* q = a.norms + bucket;
#pragma unroll
        for (int j = 0; j < MC; ++j, p += a.packed_stride, q += nb) {
            request_words<B>(p, wd[j]);
            nrm[j] = load_norm_early(q);
        }
    }
    auto decode = [&](uint64_t (&acc2)[16], const uint32_t (&w)[B], const float norm) {
        uint32_t hi[B];
#pragma unroll
        for (int i = 0; i < B; ++i) hi[i] = w[i] >> 16;
        const uint32_t sc = __float_as_uint(norm * unit);
        AccumulateAll<B, 0>::run(acc2, w, hi, pack_pair(sc, sc), magic);
    };
    for (int k = 0; k < n_tiles; ++k) {
        uint64_t acc2[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) acc2[q] = 0ull;
        int nbucket = bucket, nvalid = valid;
        if (a.update && lane == 0) request_x(out_map, out_tile, tile, x_bar(warp));
#pragma unroll 1
        for (int m0 = 0; m0 < M; m0 += MC) {
            // the workers eight further on: of this tile, or the first ones of the next, if there is one.  (The second
            // loop keeps its bounds, although groups are whole here: without them the compiler orders the first
            // one's loads worse, 2^26 elements M = 32 b = 3 262.5 -> 268.8 us.)
            const bool same = m0 + MC < M;
            if (!same && k + 1 < n_tiles) locate_group(a, tbl_in_smem, tile + hop, nbucket, nvalid);
            const int first = same ? m0 + MC : 0;
            const uint32_t* p = words_of(same ? tile : tile + hop, first);
            const float* q = a.norms + (int64_t)first * nb + (same ? bucket : nbucket);
            const int more = same ? M - first : (k + 1 < n_tiles ? M : 0);
            if (m0 + MC <= M && more >= MC) {
#pragma unroll
                for (int j = 0; j < MC; ++j, p += a.packed_stride, q += nb) {
                    decode(acc2, wd[j], nrm[j]);
                    request_words<B>(p, wd[j]);
                    nrm[j] = load_norm_early(q);
                }
            } else {
#pragma unroll
                for (int j = 0; j < MC; ++j) {
                    if (m0 + j < M) decode(acc2, wd[j], nrm[j]);
                    if (j < more) {
                        request_words<B>(p, wd[j]);
                        nrm[j] = load_norm_early(q);
                    }
                    p += a.packed_stride; q += nb;
                }
            }
        }
        const TileEnd end = finish_tile<B>(a, out_map, out_tile, acc2, tile, valid, valid > 0 && !sums_finite(acc2), x_bar(warp),
                                           (uint32_t)k & 1u);
        if (end != kDone) {
            if (lane == 0) {
                if (end == kLost) atomicOr(a.status, DQ_STAT_WAIT);
                tma::store_wait_read();
            }
            // (the copy must not outlive the shared memory)
            if (a.update && !__all_sync(0xffffffffu, tma::mbar_wait(x_bar(warp), (uint32_t)k & 1u, a.wait)) && lane == 0)
                atomicOr(a.status, DQ_STAT_WAIT);
            if (end == kOutOfRange) average_tiles_plain(a, tbl_in_smem, B, tile, hop, n_tiles - k);
            return;
        }
        tile += hop;
        bucket = nbucket;
        valid = nvalid;
    }
    if (lane == 0) tma::store_wait_read();         // shared memory must outlive the last store's reads
}

// ---- how the words come into a stage --------------------------------------------------------------
// ASYNC = false: one bulk copy of 128 * b bytes per worker.  ASYNC = true: 16 bytes per lane and instruction, straight
// to shared memory.  The bulk copies are so small that their rate is the limit where there are many workers (2^25
// elements, M = 12, b = 2: one copy of 256 bytes every 15 cycles of an SM); with few, a stage is a few copies, which cost
// the warp less than its own.  Measured, bulk / async (us): 2^25 elements M = 12 b = 2 66.7 / 62.5, b = 4 68.4 / 65.7,
// b = 5 71.7 / 74.2; M = 8 b = 2 46.9 / 45.6, b = 4 49.3 / 49.7, b = 5 57.7 / 59.9, b = 7 60.1 / 62.5; M = 4 b = 2 34.5 / 35.8,
// b = 5 38.3 / 43.2; d = 8.4M M = 16 b = 4 22.9 / 21.0, b = 6 29.1 / 29.1, b = 7 30.4 / 30.1; 2^24 elements M = 32 b = 5
// 89.2 / 88.2, b = 6 91.5 / 87.9, b = 7 99.4 / 95.0, b = 8 94.3 / 93.2 (M = 16 29.6 / 29.8).
template <int B>
struct AsyncCopies {
    static constexpr bool value = B >= 2 && B <= 7;
    static constexpr int min_workers = B <= 4 ? 8 : 16;
};
// The codes of N workers of a stage, added to the sums; moves on to the workers behind them.
template <int B, int N, int MC>
__device__ __forceinline__ void add_workers(uint64_t (&acc2)[16], const uint32_t*& base, float (&scale)[MC], const uint32_t magic)
{
#pragma unroll
    for (int j = 0; j < N; ++j) {
        uint32_t wd[B], hi[B];
        load_words<B>(base + j * (32 * B), wd);
        UpperHalves<B, 0>::run(base + j * (32 * B), hi);
        const uint32_t sc = __float_as_uint(scale[j]);
        AccumulateAll<B, 0>::run(acc2, wd, hi, pack_pair(sc, sc), magic);
    }
    base += N * (32 * B);
#pragma unroll
    for (int j = 0; j + N < MC; ++j) scale[j] = scale[j + N];
}

template <int B, bool ASYNC>
__device__ __forceinline__ void average_tiles(const AverageArgs& a, const CUtensorMap* out_map, const bool tbl_in_smem)
{
    constexpr int s = (1 << (B - 1)) - 1;
    constexpr int MC = ChunkOf<B>::value;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int G = a.v.total_groups, M = a.M, nb = a.v.nb;
    const int nchunk = (M + MC - 1) / MC;
    const float unit = (B == 1) ? 0.0f : __fdiv_rn(1.0f, (float)s * (float)M);      // 1 / (s * M)
    const uint32_t magic = a.magic;

    // every warp takes every hop-th tile, `each` of them, the first `extra` warps one more
    const uint32_t id = blockIdx.x * kWarps + warp;
    const int hop = (int)(gridDim.x * kWarps);
    const int n_tiles = (int)(a.each + (id < a.extra ? 1u : 0u));
    const int items = (B == 1) ? 0 : n_tiles * nchunk;

    auto locate = [&](int tl, int& bk, int& vl) { locate_group(a, tbl_in_smem, tl, bk, vl); };

    // ---- producer side: item = (tile, chunk of workers), fetched two ahead of the consumer
    int p_tile = (int)id, p_m0 = 0, p_left = items;
    auto fetch = [&](int st) {
        if (p_left > 0) {
            --p_left;
            const int rows = (G - p_tile * 32) < 32 ? (G - p_tile * 32) : 32;
            const uint32_t bytes = ((uint32_t)(rows * B * 4) + 15u) & ~15u;      // the stream's stride is a multiple of 16 bytes
            if constexpr (ASYNC) {
                const uint32_t dst = tma::smem_addr(stage_words(warp, st)) + lane * 16;
                const uint32_t* src = a.packed + (int64_t)p_m0 * a.packed_stride + (int64_t)p_tile * (32 * B) + lane * 4;
#pragma unroll
                for (int j = 0; j < MC; ++j, src += a.packed_stride) {
                    if (p_m0 + j < M) {
#pragma unroll
                        for (int u = 0; u < 128 * B; u += 512)
                            if ((uint32_t)(lane * 16 + u) < bytes)
                                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + j * (128 * B) + u), "l"(src + u / 4)
                                             : "memory");
                    }
                }
            } else {
                const int mc = (M - p_m0) < MC ? (M - p_m0) : MC;
                if (lane == 0) tma::mbar_expect_tx(stage_bar(warp, st), bytes * (uint32_t)mc);
                if (lane < mc)
                    tma::load_bulk(stage_words(warp, st) + lane * (32 * B),
                                   a.packed + (int64_t)(p_m0 + lane) * a.packed_stride + (int64_t)p_tile * (32 * B), bytes,
                                   stage_bar(warp, st));
            }
            p_m0 += MC;
            if (p_m0 >= M) { p_m0 = 0; p_tile += hop; }
        }
        // (an empty group where nothing is left to copy: the wait counts groups)
        if constexpr (ASYNC) asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int st = 0; st < kStages; ++st) fetch(st);

    int tile = (int)id, bucket, valid;
    locate(tile < (G + 31) / 32 ? tile : 0, bucket, valid);
    float scale[MC], nxt[MC];
    auto request_norms = [&](int m0, int bk) {
        const float* p = a.norms + (int64_t)m0 * nb + bk;
        if (m0 + MC <= M) {
#pragma unroll
            for (int j = 0; j < MC; ++j) nxt[j] = load_norm_early(p + (int64_t)j * nb);
        } else {
#pragma unroll
            for (int j = 0; j < MC; ++j) nxt[j] = m0 + j < M ? load_norm_early(p + (int64_t)j * nb) : 0.0f;
        }
    };
    if (items > 0) request_norms(0, bucket);

    unsigned char* out_tile = smem + warp * kOutBytes;
    uint32_t it = 0;
    bool timed_out = false;
    int plain_left = 0;                           // tiles left to average_tiles_plain
    uint32_t x_parity = 0;                        // of the tile of x at hand
    // (test hook: the warp's first wait counts as lost, and the warp goes straight to what follows a time-out)
    const bool skip_all = a.wait.lose_first != 0u && items > 0;
    for (int k = 0; k < n_tiles && !skip_all; ++k) {
        uint64_t acc2[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) acc2[q] = 0ull;
        float largest = 0.0f;
        int nbucket = bucket, nvalid = valid;
        x_parity = (uint32_t)k & 1u;
        if (B > 1 && a.update && lane == 0) request_x(out_map, out_tile, tile, x_bar(warp));
        if constexpr (B > 1) {
#pragma unroll 1
            for (int m0 = 0; m0 < M; m0 += MC, ++it) {
                const int st = (int)(it & 1u);
                // the norms of the chunk after this one travel during the wait and the decoding
#pragma unroll
                for (int j = 0; j < MC; ++j) {
                    scale[j] = nxt[j] * unit;
                    if (j & 1 || j + 1 == MC) largest = max_magnitude(largest, nxt[j], nxt[j > 0 ? j - 1 : 0]);
                }
                if (m0 + MC < M) {
                    request_norms(m0 + MC, bucket);
                } else if (k + 1 < n_tiles) {
                    locate(tile + hop, nbucket, nvalid);
                    request_norms(0, nbucket);
                }
                if constexpr (ASYNC) {
                    asm volatile("cp.async.wait_group 1;" ::: "memory");           // all but the stage after this one
                    __syncwarp();
                } else if (!__all_sync(0xffffffffu, tma::mbar_wait(stage_bar(warp, st), (it >> 1) & 1u, a.wait))) {
                    // (every lane polls the barrier itself; the verdict is made warp-uniform)
                    timed_out = true;
                    break;
                }
                const uint32_t* base = stage_words(warp, st) + lane * B;
                if (m0 + MC <= M) {              // a full stage, or what is left in blocks of 4, 2 and 1: no loop
                    add_workers<B, MC>(acc2, base, scale, magic);
                } else {
                    const int left = M - m0;
                    if constexpr (MC > 4) {
                        if (left & 4) add_workers<B, 4>(acc2, base, scale, magic);
                    }
                    if constexpr (MC > 2) {
                        if (left & 2) add_workers<B, 2>(acc2, base, scale, magic);
                    }
                    if (left & 1) add_workers<B, 1>(acc2, base, scale, magic);
                }
                // the warp's reads of the stage come before the copies that refill it (another proxy, if they are bulk copies)
                if constexpr (!ASYNC) tma::fence_proxy_async();
                __syncwarp();
                fetch(st);
                __syncwarp();
            }
            if (timed_out) break;
        }
        // (decoded values carry up to 2^21: sums of norms below 2^104 stay in the fp32 range)
        const TileEnd end = finish_tile<B>(a, out_map, out_tile, acc2, tile, valid, !(largest < 0x1p104f), x_bar(warp), x_parity);
        if (end == kOutOfRange) { plain_left = n_tiles - k; break; }
        if (end == kLost) { timed_out = true; break; }
        tile += hop;
        if (B == 1 && k + 1 < n_tiles) locate(tile, nbucket, nvalid);
        bucket = nbucket;
        valid = nvalid;
    }
    if (lane == 0) tma::store_wait_read();         // shared memory must outlive the last store's reads
    if constexpr (ASYNC) asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (timed_out || skip_all || plain_left > 0) {
        // every copy the warp has issued and not seen land, the one whose wait ran out included, gets the
        // full limit before the CTA's shared memory is released
        bool landed = plain_left > 0;
        for (uint32_t i = it; !ASYNC && i < (uint32_t)(items - p_left); ++i)
            landed &= tma::mbar_wait(stage_bar(warp, (int)(i & 1u)), (i >> 1) & 1u, a.wait);
        if (B > 1 && a.update && !skip_all) landed &= tma::mbar_wait(x_bar(warp), x_parity, a.wait);
        landed = __all_sync(0xffffffffu, landed);
        if (lane == 0 && !landed) atomicOr(a.status, DQ_STAT_WAIT);
        if (plain_left > 0) average_tiles_plain(a, tbl_in_smem, B, tile, hop, plain_left);
    }
}

__global__ void __launch_bounds__(kThreads, kCtasPerSm)
unpack_average_kernel(const __grid_constant__ AverageArgs a, const __grid_constant__ CUtensorMap out_map)
{
    // (nothing up to the wait touches memory that an earlier kernel may still be writing)
    if (threadIdx.x == 0) {
        tma::prefetch_tensor_map(&out_map);
        for (int i = 0; i < kWarps * (kStages + 1); ++i) tma::mbar_init(stage_bar(0, i), 1);
        tma::fence_barrier_init();
    }
    grid_dependency_wait();
    const int b = __ldg(a.dev_b);       // issued first, looked at after the set-up below so that the loads overlap
    const bool tbl_in_smem = a.v.n_seg > 1 && a.v.n_seg <= kMaxSmemSegs;
    if (tbl_in_smem) {
        int32_t* tbl_s = reinterpret_cast<int32_t*>(smem + kTblOffset);
        for (int i = threadIdx.x; i < 3 * (a.v.n_seg + 1); i += kThreads) tbl_s[i] = __ldg(a.v.seg_group0 + i);
    }
    __syncthreads();
    if (tma::smem_addr(smem) & 1023u) {           // the swizzled tiles need a 1024-byte aligned base
        if (threadIdx.x == 0) atomicOr(a.status, DQ_STAT_INTERNAL);
        return;
    }
    if (b < 1 || b > DQ_MAX_BITS) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.status, DQ_STAT_BAD_BITS);
        return;
    }
    if ((int64_t)b * a.v.total_groups > a.packed_stride) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.status, DQ_STAT_CAPACITY);
        return;
    }

    switch (b) {
#define DQ_CASE(BB) case BB:                                                                             \
            if constexpr (DirectWords<BB>::value) {                                                       \
                if (a.M % DirectWords<BB>::workers == 0) {                                                \
                    average_tiles_direct<BB>(a, &out_map, tbl_in_smem);                                   \
                    break;                                                                                \
                }                                                                                         \
            }                                                                                             \
            if constexpr (AsyncCopies<BB>::value) {                                                       \
                if (a.M >= AsyncCopies<BB>::min_workers) {                                                \
                    average_tiles<BB, true>(a, &out_map, tbl_in_smem);                                    \
                    break;                                                                                \
                }                                                                                         \
            }                                                                                             \
            average_tiles<BB, false>(a, &out_map, tbl_in_smem);                                           \
            break;
        DQ_CASE(1) DQ_CASE(2) DQ_CASE(3) DQ_CASE(4) DQ_CASE(5) DQ_CASE(6) DQ_CASE(7) DQ_CASE(8)
        DQ_CASE(9) DQ_CASE(10) DQ_CASE(11) DQ_CASE(12) DQ_CASE(13) DQ_CASE(14) DQ_CASE(15) DQ_CASE(16)
#undef DQ_CASE
        default: break;
    }
}

// Checks and launch shared by the two entry points; `dev_out` is the averaged gradient, or the
// parameters, read and written (update).
int launch_average(const dq_layout_t* L, const uint32_t* dev_packed, int64_t packed_stride_words, const float* dev_norms,
                   int32_t M, const int32_t* dev_b, bool update, float lr, float* dev_out, int32_t* dev_status, void* stream)
{
    const int rc = dq_check_common(L, M);
    if (rc != DQ_OK) return rc;
    if (!dev_packed || !dev_norms || !dev_b || !dev_out || !dev_status) return DQ_ERR_ARG;
    if (!aligned16(dev_packed) || !aligned16(dev_out) || (packed_stride_words % 4) != 0 ||
        (reinterpret_cast<uintptr_t>(dev_norms) & 3u) || (reinterpret_cast<uintptr_t>(dev_b) & 3u) ||
        (reinterpret_cast<uintptr_t>(dev_status) & 3u))
        return DQ_ERR_ALIGN;
    if (packed_stride_words < L->padded / 32) return DQ_ERR_RANGE;
    if (update && !(lr == lr && lr - lr == 0.0f)) return DQ_ERR_RANGE;      // eta must be finite

    AverageArgs a = {};
    a.v = make_view(L);
    a.packed = dev_packed;
    a.packed_stride = packed_stride_words;
    a.norms = dev_norms;
    a.dev_b = dev_b;
    a.out = dev_out;
    a.status = dev_status;
    a.M = M;
    a.magic = 0x4B000000u;
    a.update = update ? 1 : 0;
    a.neg_lr = -lr;
    a.wait = dq_wait_limits();
    const uint32_t gpb = (uint32_t)a.v.groups_per_bucket;
    if ((gpb & (gpb - 1)) == 0) {
        a.div_shift = 0;
        while ((1u << a.div_shift) < gpb) ++a.div_shift;
        a.div_magic = 0;
    } else {
        a.div_shift = -1;
        a.div_magic = (uint32_t)(((uint64_t(1) << 33) + gpb - 1) / gpb);
    }

    // tensor map over the output: [group][32 floats], box = one warp tile of 32 groups, 128-byte swizzle
    CUtensorMap out_map;
    const uint64_t dims[2] = {32, (uint64_t)a.v.total_groups};
    const uint64_t strides[1] = {128};
    const uint32_t box[2] = {32, 32};
    if (!dq_encode_tensor_map(&out_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, dev_out, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
        return DQ_ERR_CUDA;

    size_t smem_need = (size_t)kTblOffset;
    if (L->n_seg > 1 && L->n_seg <= kMaxSmemSegs) smem_need += (size_t)3 * (L->n_seg + 1) * 4;
    // (the limit of the largest table, whatever this one's size: with each call's own, another thread's call for a
    // smaller layout can narrow it again before this launch, which then fails)
    constexpr int kLargest = kTblOffset + 3 * (kMaxSmemSegs + 1) * 4;
    if (cudaFuncSetAttribute(unpack_average_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLargest) != cudaSuccess) {
        (void)cudaGetLastError();
        return DQ_ERR_CUDA;
    }
    const int64_t tiles = ((int64_t)a.v.total_groups + 31) / 32;
    int64_t blocks = (int64_t)dq_sm_count() * kCtasPerSm;
    if (blocks * kWarps > tiles) blocks = (tiles + kWarps - 1) / kWarps;
    a.each = (uint32_t)(tiles / (blocks * kWarps));
    a.extra = (uint32_t)(tiles - (int64_t)a.each * blocks * kWarps);
    dq_launch(unpack_average_kernel, dim3((unsigned)blocks), dim3(kThreads), smem_need, static_cast<cudaStream_t>(stream), a, out_map);
    return cudaGetLastError() == cudaSuccess ? DQ_OK : DQ_ERR_CUDA;
}

}  // namespace

extern "C" int dq_unpack_dequant_average(const dq_layout_t* L, const uint32_t* dev_packed,
                                         int64_t packed_stride_words, const float* dev_norms, int32_t M,
                                         const int32_t* dev_b, float* dev_out, int32_t* dev_status, void* stream)
{
    return launch_average(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, false, 0.0f, dev_out, dev_status, stream);
}

extern "C" int dq_unpack_average_update(const dq_layout_t* L, const uint32_t* dev_packed,
                                        int64_t packed_stride_words, const float* dev_norms, int32_t M,
                                        const int32_t* dev_b, float lr, float* dev_params, int32_t* dev_status,
                                        void* stream)
{
    return launch_average(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, true, lr, dev_params, dev_status, stream);
}
