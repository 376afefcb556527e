// dq_bucket_norms: per-bucket norm of every worker's gradient (the scale factor
// ||g||_p of Eq. 5 applied per bucket; p = 2, or p = infinity for layouts created
// with DQ_NORM_LINF), and dq_tensor_norms: one norm per tensor.
//
// Bucket lengths of up to 1024 elements, 2048 and 4096 are taken by the norm kernels of dq_round.cuh (the
// pipelines of the quantizer without the codes), the others by the kernel below: 128-bit coalesced
// loads, four independent fp32 accumulators per lane, a warp per run of consecutive buckets of one
// worker (blockIdx.y), so that the tensor a bucket belongs to is searched once per run and then followed.
// HBM-bound: 4 bytes read per element, 4/bucket bytes written.
#include "dq_common.cuh"
#include "dq_device.cuh"
#include "dq_round.cuh"

bool dq_norms_inside(const dq_layout_t* L)
{
    const uint32_t gpb = (uint32_t)(L->bucket / 32);
    return !L->whole_tensor && ((gpb & (gpb - 1)) == 0 || gpb < 32);
}

int64_t dq_tile_positions(const RoundArgs& a, bool given)
{
    if (given) return (a.v.total_groups + 31) / 32;
    if (a.div_shift >= 0 && a.gpb_shift > 5) return a.v.nb;
    const int64_t R = 32 / a.v.groups_per_bucket;
    return (a.v.nb + R - 1) / R;
}

int dq_norms_of_buckets(const RoundArgs& a, const CUtensorMap& map, int n_seg, cudaStream_t st)
{
    const int64_t entries = dq_tile_positions(a, false) * a.M;
    if (a.div_shift < 0)
        return a.linf ? dq_launch_norms<kOddBuckets, true>(a, map, n_seg, entries, st)
                      : dq_launch_norms<kOddBuckets, false>(a, map, n_seg, entries, st);
    if (a.gpb_shift <= 5)
        return a.linf ? dq_launch_norms<kWarpBuckets, true>(a, map, n_seg, entries, st)
                      : dq_launch_norms<kWarpBuckets, false>(a, map, n_seg, entries, st);
    return a.linf ? dq_launch_norms<kTeamBuckets, true>(a, map, n_seg, entries, st)
                  : dq_launch_norms<kTeamBuckets, false>(a, map, n_seg, entries, st);
}

bool dq_fill_round(RoundArgs& a, CUtensorMap& map, const dq_layout_t* L, const LayoutView& v, const float* dev_grads,
                   int64_t worker_stride_elems, int32_t M, int32_t* dev_status)
{
    a = RoundArgs{};
    a.v = v;
    a.grads = dev_grads;
    a.grad_stride = M > 1 ? worker_stride_elems : 0;
    a.status = dev_status;
    a.M = M;
    a.linf = L->norm == DQ_NORM_LINF ? 1 : 0;
    a.wait = dq_wait_limits();
    a.stream_reads = ((int64_t)M * L->padded * 4 > (int64_t(64) << 20)) ? 1 : 0;
    const bool worker_dim = (M > 1 && worker_stride_elems != 0);
    a.map_has_worker_dim = worker_dim ? 1 : 0;
    const uint32_t gpb = (uint32_t)v.groups_per_bucket;
    a.div_shift = -1;
    a.div_magic = (uint32_t)(((uint64_t(1) << 33) + gpb - 1) / gpb);
    if ((gpb & (gpb - 1)) == 0) {
        a.div_shift = 0;
        while ((1u << a.div_shift) < gpb) ++a.div_shift;
        a.gpb_shift = a.div_shift;
    }
    // tensor map over the gradients, [worker][group][32 floats], box = one warp tile of 32 groups
    const uint64_t dims[3] = {32, (uint64_t)v.total_groups, worker_dim ? (uint64_t)M : 1};
    const uint64_t strides[2] = {128, worker_dim ? (uint64_t)worker_stride_elems * 4 : (uint64_t)L->padded * 4};
    const uint32_t box[3] = {32, 32, 1};
    return dq_encode_tensor_map(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, dev_grads, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

namespace {

constexpr int kThreads = 256;
constexpr int kRun = 8;            // bucket rows a warp handles per run

// l2 norm of a bucket whose fp32 sum of squares is out of range (see l2_sum_in_range), read
// again with plain loads by the warp: largest magnitude first, then the squares of
// the scaled entries.  Called by all lanes of the warp; out of line, it is rarely needed.
__device__ __noinline__ float rescaled_norm_global(const float* __restrict__ g, const int len, const int lane)
{
    const MaxMagnitude mag;
    float mx = 0.f;
    for (int i = lane; i < len; i += 32) mx = mag.take(mx, __ldg(g + i));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = mag.join(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const int e = scale_exponent(mx);
    const ScaledSquares sq{e};
    float ss = 0.f;
    for (int i = lane; i < len; i += 32) ss = sq.take(ss, __ldg(g + i));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss = sq.join(ss, __shfl_xor_sync(0xffffffffu, ss, o));
    return rescaled_l2(mx, ss, e);
}

// A warp takes a run of
// eight consecutive buckets: it first works out where each of them lies (so
// that table lookups never sit between a load and its use), then streams the
// eight buckets with independent accumulators, and finally reduces the eight
// per-lane sums together with a butterfly that halves the number of live
// values at each of its first three steps (9 shuffles instead of 40).
template <int P>
__global__ void __launch_bounds__(kThreads)
bucket_norms_warp_kernel(const LayoutView v, const float* __restrict__ grads, const int64_t worker_stride,
                         float* __restrict__ norms, int32_t* __restrict__ status)
{
    extern __shared__ int32_t tbl_s[];
    grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const int m = blockIdx.y;
    const float4* gw4 = reinterpret_cast<const float4*>(grads + (int64_t)m * worker_stride);
    const float* gw = grads + (int64_t)m * worker_stride;
    float* nw = norms + (int64_t)m * v.nb;
    const int warps_total = gridDim.x * (kThreads / 32);
    const int nchunks = (v.nb + kRun - 1) / kRun;
    const int bsz = v.groups_per_bucket * 32;
    const int n1 = v.n_seg + 1;
    bool bad = false;

    const int32_t* tbl = v.seg_group0;                 // [group0 | bucket0 | elems], n_seg + 1 entries each
    if (v.n_seg > 1 && 3 * n1 * 4 <= 12 * 1024) {
        for (int i = threadIdx.x; i < 3 * n1; i += kThreads) tbl_s[i] = __ldg(v.seg_group0 + i);
        __syncthreads();
        tbl = tbl_s;
    }

    for (int chunk = blockIdx.x * (kThreads / 32) + threadIdx.x / 32; chunk < nchunks; chunk += warps_total) {
        const int k0 = chunk * kRun;
        int first[kRun], len[kRun];                    // first float4 and valid elements of each bucket
        {
            int seg = 0;
            if (v.n_seg > 1) {                         // binary search for the run's first bucket
                int lo = 0, hi = v.n_seg;
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (tbl[n1 + mid] <= k0) lo = mid; else hi = mid;
                }
                seg = lo;
            }
#pragma unroll
            for (int r = 0; r < kRun; ++r) {
                const int k = k0 + r;
                first[r] = 0;
                len[r] = 0;
                if (k < v.nb) {
                    int local, n, g0;
                    if (v.n_seg == 1) {
                        local = k; n = v.seg0_elems; g0 = 0;
                    } else {
                        while (k >= tbl[n1 + seg + 1]) ++seg;
                        local = k - tbl[n1 + seg];
                        n = tbl[2 * n1 + seg];
                        g0 = tbl[seg];
                    }
                    first[r] = (g0 + local * v.groups_per_bucket) * 8;
                    const int left = n - local * bsz;
                    len[r] = left < bsz ? left : bsz;
                }
            }
        }
        float part[kRun];
#pragma unroll
        for (int r = 0; r < kRun; ++r) {
            const float4* g4 = gw4 + first[r];
            const int n4 = len[r] >> 2;
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
            for (int i = lane; i < n4; i += 128) {
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 x0 = __ldg(g4 + i);
                const float4 x1 = (i + 32 < n4) ? __ldg(g4 + i + 32) : z;
                const float4 x2 = (i + 64 < n4) ? __ldg(g4 + i + 64) : z;
                const float4 x3 = (i + 96 < n4) ? __ldg(g4 + i + 96) : z;
                a0 = take<P>(a0, x0.x); a1 = take<P>(a1, x0.y); a2 = take<P>(a2, x0.z); a3 = take<P>(a3, x0.w);
                a0 = take<P>(a0, x1.x); a1 = take<P>(a1, x1.y); a2 = take<P>(a2, x1.z); a3 = take<P>(a3, x1.w);
                a0 = take<P>(a0, x2.x); a1 = take<P>(a1, x2.y); a2 = take<P>(a2, x2.z); a3 = take<P>(a3, x2.w);
                a0 = take<P>(a0, x3.x); a1 = take<P>(a1, x3.y); a2 = take<P>(a2, x3.z); a3 = take<P>(a3, x3.w);
            }
            if (lane < (len[r] & 3)) {                 // ragged tail of a tensor's last bucket
                const float x = __ldg(gw + (int64_t)first[r] * 4 + n4 * 4 + lane);
                a0 = take<P>(a0, x);
            }
            part[r] = join<P>(join<P>(a0, a1), join<P>(a2, a3));
        }
        // butterfly: after the three halving steps lane l holds bucket (l & 7) summed over its octet
        float q[4], h[2], t;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float keep = (lane & 1) ? part[2 * i + 1] : part[2 * i];
            const float give = (lane & 1) ? part[2 * i] : part[2 * i + 1];
            q[i] = join<P>(keep, __shfl_xor_sync(0xffffffffu, give, 1));
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float keep = (lane & 2) ? q[2 * i + 1] : q[2 * i];
            const float give = (lane & 2) ? q[2 * i] : q[2 * i + 1];
            h[i] = join<P>(keep, __shfl_xor_sync(0xffffffffu, give, 2));
        }
        {
            const float keep = (lane & 4) ? h[1] : h[0];
            const float give = (lane & 4) ? h[0] : h[1];
            t = join<P>(keep, __shfl_xor_sync(0xffffffffu, give, 4));
        }
        t = join<P>(t, __shfl_xor_sync(0xffffffffu, t, 8));
        t = join<P>(t, __shfl_xor_sync(0xffffffffu, t, 16));
        float nrm = finish<P>(t);
        if constexpr (P == DQ_NORM_L2) {
            // lane r holds bucket r of the run: the buckets out of range are taken again one by one
            const unsigned need = __ballot_sync(0xffffffffu, lane < kRun && k0 + lane < v.nb && !l2_sum_in_range(t));
            if (need) {
#pragma unroll
                for (int r = 0; r < kRun; ++r) {
                    if ((need >> r) & 1u) {
                        const float again = rescaled_norm_global(gw + (int64_t)first[r] * 4, len[r], lane);
                        if (lane == r) nrm = again;
                    }
                }
            }
        }
        if (lane < kRun && k0 + lane < v.nb) {
            DQ_STORE(nw + (k0 + lane), nrm, norms, (int64_t)gridDim.y * v.nb * 4, status);
            bad |= !isfinite(nrm);
        }
    }
    if (bad) atomicOr(status, DQ_STAT_NONFINITE);
}

// Second step of dq_tensor_norms: block (tensor, worker) joins the norms of the tensor's pieces in
// a fixed order -- thread t takes pieces t, t + 256, ..., then a tree over the block -- and writes
// the tensor's norm.  l2: the squares of the piece norms are exact in fp64 and cannot leave its
// range; their sum is at least p^2 for every piece norm p, the fp64 square root is monotone and
// gives back p for p^2, and so is the rounding to fp32, which has p among its values: the tensor's
// norm is at least every piece norm, which in turn is at least every entry of the piece.
constexpr int kJoinThreads = 256;

template <int P>
__global__ void __launch_bounds__(kJoinThreads)
tensor_norms_join_kernel(const int32_t n_seg, const int32_t* __restrict__ piece0, const int32_t* __restrict__ bucket0,
                         const int32_t n_pieces, const int32_t nb, const float* __restrict__ partial,
                         float* __restrict__ norms, int32_t* __restrict__ status)
{
    __shared__ double part_d[kJoinThreads / 32];
    __shared__ float part_f[kJoinThreads / 32];
    grid_dependency_wait();
    const int seg = blockIdx.x, m = blockIdx.y;
    int c0 = 0, c1 = n_pieces, k = 0;
    if (n_seg > 1) {
        c0 = __ldg(piece0 + seg);
        c1 = __ldg(piece0 + seg + 1);
        k = __ldg(bucket0 + seg);
    }
    if (c0 >= c1) return;                                    // an empty tensor has no norm
    const float* src = partial + (int64_t)m * n_pieces;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float nrm;
    if constexpr (P == DQ_NORM_L2) {
        double acc = 0.0;
        for (int i = c0 + tid; i < c1; i += kJoinThreads) {
            const double p = (double)__ldg(src + i);
            acc = fma(p, p, acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) part_d[warp] = acc;
        __syncthreads();
        if (tid != 0) return;
        double total = 0.0;
        for (int w = 0; w < kJoinThreads / 32; ++w) total += part_d[w];
        nrm = (float)sqrt(total);
    } else {
        float acc = 0.0f;
        for (int i = c0 + tid; i < c1; i += kJoinThreads) acc = max_nan(acc, __ldg(src + i));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc = max_nan(acc, __shfl_xor_sync(0xffffffffu, acc, o));
        if (lane == 0) part_f[warp] = acc;
        __syncthreads();
        if (tid != 0) return;
        float total = 0.0f;
        for (int w = 0; w < kJoinThreads / 32; ++w) total = max_nan(total, part_f[w]);
        nrm = total;
    }
    DQ_STORE(norms + ((int64_t)m * nb + k), nrm, norms, (int64_t)gridDim.y * nb * 4, status);
    if (!isfinite(nrm)) atomicOr(status, DQ_STAT_NONFINITE);
}

// Norms of the buckets of view `v` (see dq_norms_inside).
int launch_norms(const dq_layout_t* L, const LayoutView& v, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
                 float* dev_out, int32_t* dev_status, cudaStream_t st)
{
    RoundArgs a;
    CUtensorMap map;
    if (!dq_fill_round(a, map, L, v, dev_grads, worker_stride_elems, M, dev_status)) return DQ_ERR_CUDA;
    a.norms = dev_out;
    return dq_norms_of_buckets(a, map, L->n_seg, st);
}

// other bucket sizes: the plain-load kernel
template <int P>
int launch_plain(const dq_layout_t* L, const LayoutView& v, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
                 float* dev_norms, int32_t* dev_status, cudaStream_t st)
{
    const int64_t chunk = kRun;
    const int64_t nchunks = (L->nb + chunk - 1) / chunk;
    int64_t bx = (nchunks + kThreads / 32 - 1) / (kThreads / 32);
    // about 8 resident CTAs of 256 threads per SM over all workers
    int64_t cap = ((int64_t)dq_sm_count() * 8 + M - 1) / M;
    if (cap < 1) cap = 1;
    if (bx > cap) bx = cap;
    if (bx < 1) bx = 1;
    const dim3 grid((unsigned)bx, (unsigned)M);
    const size_t smem = (L->n_seg > 1 && (size_t)3 * (L->n_seg + 1) * 4 <= 12 * 1024) ? (size_t)3 * (L->n_seg + 1) * 4 : 0;
    dq_launch(bucket_norms_warp_kernel<P>, grid, dim3(kThreads), smem, st, v, dev_grads, worker_stride_elems, dev_norms, dev_status);
    if (cudaGetLastError() != cudaSuccess) return DQ_ERR_CUDA;
    return DQ_OK;
}

int check_norm_args(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
                    const float* dev_norms, const int32_t* dev_status)
{
    const int rc = dq_check_common(L, M);
    if (rc != DQ_OK) return rc;
    if (!dev_grads || !dev_norms || !dev_status) return DQ_ERR_ARG;
    if (!aligned16(dev_grads) || (worker_stride_elems % 32) != 0 || (reinterpret_cast<uintptr_t>(dev_norms) & 3u) ||
        (reinterpret_cast<uintptr_t>(dev_status) & 3u))
        return DQ_ERR_ALIGN;
    if (M > 1 && worker_stride_elems < L->padded && worker_stride_elems != 0) return DQ_ERR_RANGE;
    return DQ_OK;
}

}  // namespace

extern "C" int dq_bucket_norms(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems,
                               int32_t M, float* dev_norms, int32_t* dev_status, void* stream)
{
    const int rc = check_norm_args(L, dev_grads, worker_stride_elems, M, dev_norms, dev_status);
    if (rc != DQ_OK) return rc;
    if (L->whole_tensor) return DQ_ERR_RANGE;           // one norm per tensor comes from dq_tensor_norms

    const LayoutView v = make_view(L);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool linf = (L->norm == DQ_NORM_LINF);
    if (dq_norms_inside(L)) return launch_norms(L, v, dev_grads, worker_stride_elems, M, dev_norms, dev_status, st);
    return linf ? launch_plain<DQ_NORM_LINF>(L, v, dev_grads, worker_stride_elems, M, dev_norms, dev_status, st)
                : launch_plain<DQ_NORM_L2>(L, v, dev_grads, worker_stride_elems, M, dev_norms, dev_status, st);
}

extern "C" size_t dq_tensor_norms_scratch_bytes(const dq_layout_t* L, int32_t M)
{
    if (!L || !L->whole_tensor || M < 1) return 0;
    return (size_t)M * (size_t)L->n_pieces * sizeof(float);
}

extern "C" int dq_tensor_norms(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
                               float* dev_norms, void* dev_scratch, size_t scratch_bytes, int32_t* dev_status,
                               void* stream)
{
    const int rc = check_norm_args(L, dev_grads, worker_stride_elems, M, dev_norms, dev_status);
    if (rc != DQ_OK) return rc;
    if (!L->whole_tensor) return DQ_ERR_RANGE;          // bucketed layouts: dq_bucket_norms
    if (!dev_scratch) return DQ_ERR_ARG;
    if (!aligned16(dev_scratch)) return DQ_ERR_ALIGN;
    if (scratch_bytes < dq_tensor_norms_scratch_bytes(L, M)) return DQ_ERR_RANGE;

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float* partial = static_cast<float*>(dev_scratch);
    const LayoutView pv = make_piece_view(L);
    const bool linf = (L->norm == DQ_NORM_LINF);
    const int r1 = launch_norms(L, pv, dev_grads, worker_stride_elems, M, partial, dev_status, st);
    if (r1 != DQ_OK) return r1;
    const int32_t n1 = L->n_seg + 1;
    const int32_t* piece0 = L->n_seg > 1 ? L->dev_table + 4 * n1 : nullptr;
    const int32_t* bucket0 = L->n_seg > 1 ? L->dev_table + n1 : nullptr;
    const dim3 grid((unsigned)L->n_seg, (unsigned)M);
    if (linf)
        dq_launch(tensor_norms_join_kernel<DQ_NORM_LINF>, grid, dim3(kJoinThreads), 0, st, L->n_seg, piece0, bucket0,
                  (int32_t)L->n_pieces, (int32_t)L->nb, partial, dev_norms, dev_status);
    else
        dq_launch(tensor_norms_join_kernel<DQ_NORM_L2>, grid, dim3(kJoinThreads), 0, st, L->n_seg, piece0, bucket0,
                  (int32_t)L->n_pieces, (int32_t)L->nb, partial, dev_norms, dev_status);
    if (cudaGetLastError() != cudaSuccess) return DQ_ERR_CUDA;
    return DQ_OK;
}
