// Host side of the quantizer calls (kernels: dq_round.cuh).
//
//   dq_quantize_pack          codes for norms that are given
//   dq_norms_quantize_pack    norms and codes in one pass over the gradients
//   dq_quantize_average       codes for given norms and the average of all workers in one pass
//   dq_norms_quantize_average norms, codes, average (or parameter update) and the next b in one pass
//
// Algorithm 1 takes b_{t+1} from the gradients of iteration t, so the bit width of a step is known
// before its gradients are: a bucket that sits in registers can be measured, coded and added to the
// average at once, and every gradient byte is read from HBM a single time.
#include "dq_round.cuh"

namespace {

bool power_of_two(uint32_t x) { return (x & (x - 1)) == 0; }

constexpr int kMaxTableSegs = 1023;      // tensors the computed-norm kernels keep in shared memory

// Arguments every call shares; dev_norms is written or read as the call has it.
int check_args(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M, const float* dev_norms,
               const int32_t* dev_b, const uint32_t* dev_packed, int64_t packed_stride_words, const int32_t* dev_status)
{
    const int rc = dq_check_common(L, M);
    if (rc != DQ_OK) return rc;
    if (!dev_grads || !dev_norms || !dev_b || !dev_packed || !dev_status) return DQ_ERR_ARG;
    if (!aligned16(dev_grads) || !aligned16(dev_packed) || (worker_stride_elems % 32) != 0 ||
        (packed_stride_words % 4) != 0 || (reinterpret_cast<uintptr_t>(dev_norms) & 3u) ||
        (reinterpret_cast<uintptr_t>(dev_b) & 3u) || (reinterpret_cast<uintptr_t>(dev_status) & 3u))
        return DQ_ERR_ALIGN;
    if (M > 1 && worker_stride_elems < L->padded && worker_stride_elems != 0) return DQ_ERR_RANGE;
    if (packed_stride_words < L->padded / 32) return DQ_ERR_RANGE;   // not even b = 1 fits
    return DQ_OK;
}

// Everything but the parts of AVG: kernel arguments and the tensor map over the gradients,
// [worker][group][32 floats], box = one warp tile of 32 groups.
bool fill_args(RoundArgs& a, CUtensorMap& map, const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
               const float* dev_norms, const int32_t* dev_b, uint64_t seed, uint32_t step, uint32_t first_worker,
               uint32_t* dev_packed, int64_t packed_stride_words, int32_t* dev_status)
{
    a = RoundArgs{};
    a.v = make_view(L);
    a.norms = const_cast<float*>(dev_norms);
    a.dev_b = const_cast<int32_t*>(dev_b);
    a.packed = dev_packed;
    a.packed_stride = packed_stride_words;
    a.status = dev_status;
    a.keys = make_philox_keys(seed);
    a.step = step;
    a.worker0 = first_worker;
    a.M = M;
    a.linf = L->norm == DQ_NORM_LINF ? 1 : 0;
    a.wide_words = (reinterpret_cast<uintptr_t>(dev_packed) % 32 == 0 && packed_stride_words % 8 == 0) ? 1 : 0;
    a.wait = dq_wait_limits();
    a.stream_reads = ((int64_t)M * L->padded * 4 > (int64_t(64) << 20)) ? 1 : 0;
    const bool worker_dim = (M > 1 && worker_stride_elems != 0);
    a.map_has_worker_dim = worker_dim ? 1 : 0;
    const uint32_t gpb = (uint32_t)a.v.groups_per_bucket;
    a.div_shift = -1;
    a.div_magic = (uint32_t)(((uint64_t(1) << 33) + gpb - 1) / gpb);
    if (power_of_two(gpb)) {
        a.div_shift = 0;
        while ((1u << a.div_shift) < gpb) ++a.div_shift;
        a.gpb_shift = a.div_shift;
    }
    const uint64_t dims[3] = {32, (uint64_t)a.v.total_groups, worker_dim ? (uint64_t)M : 1};
    const uint64_t strides[2] = {128, worker_dim ? (uint64_t)worker_stride_elems * 4 : (uint64_t)L->padded * 4};
    const uint32_t box[3] = {32, 32, 1};
    return dq_encode_tensor_map(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, dev_grads, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

// Norms inside the pass: bucket lengths of 32 * 2^k (one warp or one team per bucket) and a tensor
// table that fits; other layouts take their norms in a pass of their own.
bool norms_inside(const dq_layout_t* L)
{
    return !L->whole_tensor && power_of_two((uint32_t)(L->bucket / 32)) && L->n_seg <= kMaxTableSegs;
}

// Tile positions of a worker, and how many warps (or teams) go through them at a time.
int64_t positions(const RoundArgs& a, const dq_layout_t* L, bool given)
{
    if (given) return (a.v.total_groups + 31) / 32;
    if (a.gpb_shift > 5) return L->nb;
    const int64_t R = 32 >> a.gpb_shift;
    return (L->nb + R - 1) / R;
}

template <bool AVG>
int launch(const RoundArgs& a, const CUtensorMap& map, const dq_layout_t* L, bool given, cudaStream_t st)
{
    const int64_t entries = positions(a, L, given) * (AVG ? 1 : a.M);
    if (given) return dq_launch_round<kGivenNorms, AVG>(a, map, L->n_seg, entries, st);
    if (a.gpb_shift <= 5) return dq_launch_round<kWarpBuckets, AVG>(a, map, L->n_seg, entries, st);
    return dq_launch_round<kTeamBuckets, AVG>(a, map, L->n_seg, entries, st);
}

// One pass for codes and average, or codes (all workers' tiles side by side) and then the average from
// the words?  In one pass a warp takes a position through all M workers, one after the other: P positions
// on U warps are `full` turns of M tiles and a last turn in which only a fraction f of the warps has work.
// Two kernels spread the M * P tiles evenly, but cost a launch and read the words back.  Per worker, a
// turn's tile takes 1.8 us when the SMs are nearly empty (1.2 with given norms) and 0.9 more when they are
// full; two kernels take 2.6 us times the turns' share, and 7.5 us for the second launch; a full turn is
// 0.4 us cheaper in one pass (0.7 with given norms).  So the last turn decides.  Measured on one B200, b = 5, bucket 512, one
// pass / two kernels (us): 70k elements M = 4 14.5 / 13.2, M = 32 80 / 20; 600k M = 4 12.6 / 14.2, M = 8
// 20.4 / 19.2, M = 32 66 / 35; 1.5M M = 8 24.9 / 26.0, M = 32 82 / 64; 3M M = 8 36.5 / 39.3, M = 32
// 123 / 114; 6M M = 32 210 / 217; bucket 480: 600k M = 8 21.6 / 22.9, M = 32 66 / 55.
bool one_pass(const RoundArgs& a, const dq_layout_t* L, bool given)
{
    int64_t units = (int64_t)dq_sm_count() * RoundShape<true>::ctas_per_sm * kRoundWarps;
    if (!given && a.gpb_shift > 5) units >>= a.gpb_shift - 5;
    const int64_t p = positions(a, L, given);
    const int64_t full = p / units;
    const double f = (double)(p - full * units) / (double)units;
    if (a.M == 1 || f == 0.0) return true;                       // no worker to wait for, or no idle warp
    return a.M * ((given ? 1.2 : 1.8) - 1.7 * f - (given ? 0.7 : 0.4) * (double)full) <= 7.5;
}

}  // namespace

extern "C" int dq_quantize_pack_worker(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems,
                                       int32_t M, const float* dev_norms, const int32_t* dev_b,
                                       uint64_t seed, uint32_t step, uint32_t first_worker,
                                       uint32_t* dev_packed, int64_t packed_stride_words,
                                       int32_t* dev_status, void* stream)
{
    const int rc = check_args(L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, dev_packed, packed_stride_words, dev_status);
    if (rc != DQ_OK) return rc;
    RoundArgs a;
    CUtensorMap map;
    if (!fill_args(a, map, L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, seed, step, first_worker, dev_packed,
                   packed_stride_words, dev_status))
        return DQ_ERR_CUDA;
    return launch<false>(a, map, L, true, static_cast<cudaStream_t>(stream));
}

extern "C" int dq_quantize_pack(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems,
                                int32_t M, const float* dev_norms, const int32_t* dev_b,
                                uint64_t seed, uint32_t step,
                                uint32_t* dev_packed, int64_t packed_stride_words,
                                int32_t* dev_status, void* stream)
{
    return dq_quantize_pack_worker(L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, seed, step, 0u, dev_packed,
                                   packed_stride_words, dev_status, stream);
}

extern "C" int dq_norms_quantize_pack_worker(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems,
                                             int32_t M, const int32_t* dev_b, uint64_t seed, uint32_t step,
                                             uint32_t first_worker, float* dev_norms, uint32_t* dev_packed,
                                             int64_t packed_stride_words, int32_t* dev_status, void* stream)
{
    const int rc = check_args(L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, dev_packed, packed_stride_words, dev_status);
    if (rc != DQ_OK) return rc;
    if (L->whole_tensor) return DQ_ERR_RANGE;           // one norm per tensor: the codes need a second pass
    if (!norms_inside(L)) {
        const int r1 = dq_bucket_norms(L, dev_grads, worker_stride_elems, M, dev_norms, dev_status, stream);
        if (r1 != DQ_OK) return r1;
        return dq_quantize_pack_worker(L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, seed, step, first_worker,
                                       dev_packed, packed_stride_words, dev_status, stream);
    }
    RoundArgs a;
    CUtensorMap map;
    if (!fill_args(a, map, L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, seed, step, first_worker, dev_packed,
                   packed_stride_words, dev_status))
        return DQ_ERR_CUDA;
    return launch<false>(a, map, L, false, static_cast<cudaStream_t>(stream));
}

extern "C" int dq_norms_quantize_pack(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems,
                                      int32_t M, const int32_t* dev_b, uint64_t seed, uint32_t step,
                                      float* dev_norms, uint32_t* dev_packed, int64_t packed_stride_words,
                                      int32_t* dev_status, void* stream)
{
    return dq_norms_quantize_pack_worker(L, dev_grads, worker_stride_elems, M, dev_b, seed, step, 0u, dev_norms,
                                         dev_packed, packed_stride_words, dev_status, stream);
}

namespace {

// The arguments of AVG on top of fill_args'.
int check_average(const float* dev_out, int32_t update, float lr)
{
    if (!dev_out) return DQ_ERR_ARG;
    if (!aligned16(dev_out)) return DQ_ERR_ALIGN;
    if (update && !(lr == lr && lr - lr == 0.0f)) return DQ_ERR_RANGE;      // eta must be finite
    return DQ_OK;
}
void fill_average(RoundArgs& a, float* dev_out, int32_t update, float lr)
{
    a.out = dev_out;
    a.update = update ? 1 : 0;
    a.neg_lr = -lr;
    a.wide_out = reinterpret_cast<uintptr_t>(dev_out) % 32 == 0 ? 1 : 0;
}

// Workspace of the attached rule: the arrival counter (0 between calls) and this call's b, then a sum per CTA.
constexpr size_t kCounterBytes = 256;
constexpr size_t kThisBOffset = 128;
size_t rule_workspace_bytes()
{
    constexpr int ctas = RoundShape<true>::ctas_per_sm > RoundShape<false>::ctas_per_sm ? RoundShape<true>::ctas_per_sm
                                                                                       : RoundShape<false>::ctas_per_sm;
    return kCounterBytes + (size_t)dq_sm_count() * ctas * sizeof(double);
}

int average(const dq_layout_t* L, const uint32_t* dev_packed, int64_t packed_stride_words, const float* dev_norms, int32_t M,
            const int32_t* dev_b, float* dev_out, int32_t update, float lr, int32_t* dev_status, void* stream)
{
    return update ? dq_unpack_average_update(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, lr, dev_out, dev_status, stream)
                  : dq_unpack_dequant_average(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, dev_out, dev_status, stream);
}

}  // namespace

extern "C" int dq_quantize_average(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
                                   const float* dev_norms, const int32_t* dev_b, uint64_t seed, uint32_t step,
                                   uint32_t* dev_packed, int64_t packed_stride_words, float* dev_out, int32_t update, float lr,
                                   int32_t* dev_status, void* stream)
{
    int rc = check_args(L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, dev_packed, packed_stride_words, dev_status);
    if (rc == DQ_OK) rc = check_average(dev_out, update, lr);
    if (rc != DQ_OK) return rc;
    RoundArgs a;
    CUtensorMap map;
    if (!fill_args(a, map, L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, seed, step, 0u, dev_packed,
                   packed_stride_words, dev_status))
        return DQ_ERR_CUDA;
    if (!one_pass(a, L, true)) {
        rc = launch<false>(a, map, L, true, static_cast<cudaStream_t>(stream));
        if (rc != DQ_OK) return rc;
        return average(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, dev_out, update, lr, dev_status, stream);
    }
    fill_average(a, dev_out, update, lr);
    return launch<true>(a, map, L, true, static_cast<cudaStream_t>(stream));
}

extern "C" size_t dq_round_workspace_bytes(const dq_layout_t* L, int32_t M)
{
    if (!L || M < 1) return 0;
    const size_t rule = (rule_workspace_bytes() + 255) / 256 * 256;
    return rule + dq_tensor_norms_scratch_bytes(L, M);
}

extern "C" int dq_norms_quantize_average(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
                                         int32_t* dev_b, uint64_t seed, uint32_t step, float* dev_norms, uint32_t* dev_packed,
                                         int64_t packed_stride_words, float* dev_out, int32_t update, float lr,
                                         const dq_rule_t* next_rule, void* dev_workspace, size_t workspace_bytes,
                                         int32_t* dev_status, void* stream)
{
    int rc = check_args(L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, dev_packed, packed_stride_words, dev_status);
    if (rc == DQ_OK) rc = check_average(dev_out, update, lr);
    if (rc != DQ_OK) return rc;
    if (!next_rule || !dev_workspace) return DQ_ERR_ARG;
    rc = dq_check_rule(next_rule);
    if (rc != DQ_OK) return rc;
    if (!aligned16(dev_workspace)) return DQ_ERR_ALIGN;
    if (workspace_bytes < dq_round_workspace_bytes(L, M)) return DQ_ERR_RANGE;

    char* ws = static_cast<char*>(dev_workspace);
    const bool given = !norms_inside(L);
    if (given) {
        if (L->whole_tensor) {
            const size_t rule_bytes = (rule_workspace_bytes() + 255) / 256 * 256;
            rc = dq_tensor_norms(L, dev_grads, worker_stride_elems, M, dev_norms, ws + rule_bytes, workspace_bytes - rule_bytes,
                                 dev_status, stream);
        } else {
            rc = dq_bucket_norms(L, dev_grads, worker_stride_elems, M, dev_norms, dev_status, stream);
        }
        if (rc != DQ_OK) return rc;
    }
    RoundArgs a;
    CUtensorMap map;
    if (!fill_args(a, map, L, dev_grads, worker_stride_elems, M, dev_norms, dev_b, seed, step, 0u, dev_packed,
                   packed_stride_words, dev_status))
        return DQ_ERR_CUDA;
    a.with_rule = 1;
    a.rule = dq_rule_args(next_rule, M);
    a.rule.arrivals = reinterpret_cast<uint32_t*>(ws);
    a.rule.partial = reinterpret_cast<double*>(ws + kCounterBytes);
    if (!one_pass(a, L, given)) {
        // the next b is chosen at the end of the first kernel, which leaves its own for the second
        a.rule.this_b = reinterpret_cast<int32_t*>(ws + kThisBOffset);
        rc = launch<false>(a, map, L, given, static_cast<cudaStream_t>(stream));
        if (rc != DQ_OK) return rc;
        return average(L, dev_packed, packed_stride_words, dev_norms, M, a.rule.this_b, dev_out, update, lr, dev_status, stream);
    }
    fill_average(a, dev_out, update, lr);
    return launch<true>(a, map, L, given, static_cast<cudaStream_t>(stream));
}
