// Host side of the quantizer calls (kernels: dq_round.cuh).
//
//   dq_quantize_pack          codes for norms that are given
//   dq_norms_quantize_pack    norms and codes in one pass over the gradients
//   dq_quantize_average       codes for given norms and the average of all workers in one pass
//   dq_norms_quantize_average norms, codes, average (or parameter update) and the next b in one pass
//   dq_norms_choose_bits      norms and this round's b in one pass
//
// Algorithm 1 takes b_{t+1} from the gradients of iteration t, so the bit width of a step is known
// before its gradients are: a bucket that sits in registers can be measured, coded and added to the
// average at once, and every gradient byte is read from HBM a single time.
#include "dq_round.cuh"
#include "dq_route.h"

namespace {

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

// Everything but the parts of AVG.
bool fill_args(RoundArgs& a, CUtensorMap& map, const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
               const float* dev_norms, const int32_t* dev_b, uint64_t seed, uint32_t step, uint32_t first_worker,
               uint32_t* dev_packed, int64_t packed_stride_words, int32_t* dev_status)
{
    if (!dq_fill_round(a, map, L, make_view(L), dev_grads, worker_stride_elems, M, dev_status)) return false;
    a.norms = const_cast<float*>(dev_norms);
    a.dev_b = const_cast<int32_t*>(dev_b);
    a.packed = dev_packed;
    a.packed_stride = packed_stride_words;
    a.keys = make_philox_keys(seed);
    a.step = step;
    a.worker0 = first_worker;
    a.wide_words = (reinterpret_cast<uintptr_t>(dev_packed) % 32 == 0 && packed_stride_words % 8 == 0) ? 1 : 0;
    return true;
}

template <bool AVG>
int launch(const RoundArgs& a, const CUtensorMap& map, const dq_layout_t* L, bool given, cudaStream_t st)
{
    const int64_t entries = dq_tile_positions(a, given) * (AVG ? 1 : a.M);
    if (given) return dq_launch_round<kGivenNorms, AVG, false>(a, map, L->n_seg, entries, st);
    if (a.div_shift < 0)
        return a.linf ? dq_launch_round<kOddBuckets, AVG, true>(a, map, L->n_seg, entries, st)
                      : dq_launch_round<kOddBuckets, AVG, false>(a, map, L->n_seg, entries, st);
    if (a.gpb_shift <= 5)
        return a.linf ? dq_launch_round<kWarpBuckets, AVG, true>(a, map, L->n_seg, entries, st)
                      : dq_launch_round<kWarpBuckets, AVG, false>(a, map, L->n_seg, entries, st);
    return a.linf ? dq_launch_round<kTeamBuckets, AVG, true>(a, map, L->n_seg, entries, st)
                  : dq_launch_round<kTeamBuckets, AVG, false>(a, map, L->n_seg, entries, st);
}

// The round by CTAs.
int launch_tiles(const RoundArgs& a, const dq_layout_t* L, bool given, cudaStream_t st)
{
    const int64_t entries = dq_tile_positions(a, given);
    if (given) return dq_launch_tile_round<kGivenNorms, false>(a, L->n_seg, entries, st);
    if (a.div_shift < 0)
        return a.linf ? dq_launch_tile_round<kOddBuckets, true>(a, L->n_seg, entries, st)
                      : dq_launch_tile_round<kOddBuckets, false>(a, L->n_seg, entries, st);
    if (a.gpb_shift <= 5)
        return a.linf ? dq_launch_tile_round<kWarpBuckets, true>(a, L->n_seg, entries, st)
                      : dq_launch_tile_round<kWarpBuckets, false>(a, L->n_seg, entries, st);
    return a.linf ? dq_launch_tile_round<kTeamBuckets, true>(a, L->n_seg, entries, st)
                  : dq_launch_tile_round<kTeamBuckets, false>(a, L->n_seg, entries, st);
}

RoundRoute route_of(const RoundArgs& a, bool given)
{
    return dq_route_of(dq_tile_positions(a, given), (int64_t)dq_sm_count() * RoundShape<true>::ctas_per_sm * kRoundWarps,
                       a.v.groups_per_bucket, a.M, given, a.linf != 0, a.wait.lose_first != 0u);
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
    if (!dq_norms_inside(L)) {
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
    return (kCounterBytes + (size_t)dq_sm_count() * kRoundMaxCtasPerSm * sizeof(double) + 255) / 256 * 256;
}

int average(const dq_layout_t* L, const uint32_t* dev_packed, int64_t packed_stride_words, const float* dev_norms, int32_t M,
            const int32_t* dev_b, float* dev_out, int32_t update, float lr, int32_t* dev_status, void* stream)
{
    return update ? dq_unpack_average_update(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, lr, dev_out, dev_status, stream)
                  : dq_unpack_dequant_average(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, dev_out, dev_status, stream);
}

void attach_rule(RoundArgs& a, const dq_rule_t* rule, int32_t M, char* ws)
{
    a.with_rule = 1;
    a.rule = dq_rule_args(rule, M);
    a.rule.arrivals = reinterpret_cast<uint32_t*>(ws);
    a.rule.partial = reinterpret_cast<double*>(ws + kCounterBytes);
}

}  // namespace

extern "C" int dq_norms_choose_bits(const dq_layout_t* L, const float* dev_grads, int64_t worker_stride_elems, int32_t M,
                                    float* dev_norms, const dq_rule_t* rule, int32_t* dev_b, void* dev_workspace,
                                    size_t workspace_bytes, int32_t* dev_status, void* stream)
{
    int rc = dq_check_common(L, M);
    if (rc != DQ_OK) return rc;
    if (!dev_grads || !dev_norms || !rule || !dev_b || !dev_workspace || !dev_status) return DQ_ERR_ARG;
    rc = dq_check_rule(rule);
    if (rc != DQ_OK) return rc;
    if (!aligned16(dev_grads) || !aligned16(dev_workspace) || (worker_stride_elems % 32) != 0 ||
        (reinterpret_cast<uintptr_t>(dev_norms) & 3u) || (reinterpret_cast<uintptr_t>(dev_b) & 3u) ||
        (reinterpret_cast<uintptr_t>(dev_status) & 3u))
        return DQ_ERR_ALIGN;
    if (M > 1 && worker_stride_elems < L->padded && worker_stride_elems != 0) return DQ_ERR_RANGE;
    if (workspace_bytes < dq_round_workspace_bytes(L, M)) return DQ_ERR_RANGE;

    char* ws = static_cast<char*>(dev_workspace);
    if (dq_norms_inside(L)) {
        RoundArgs a;
        CUtensorMap map;
        if (!dq_fill_round(a, map, L, make_view(L), dev_grads, worker_stride_elems, M, dev_status)) return DQ_ERR_CUDA;
        a.norms = dev_norms;
        a.dev_b = dev_b;
        attach_rule(a, rule, M, ws);
        return dq_norms_of_buckets(a, map, L->n_seg, static_cast<cudaStream_t>(stream));
    }
    char* scratch = ws + rule_workspace_bytes();
    const size_t choose = dq_choose_bits_scratch_bytes(L, M);
    rc = L->whole_tensor ? dq_tensor_norms(L, dev_grads, worker_stride_elems, M, dev_norms, scratch + choose,
                                           dq_tensor_norms_scratch_bytes(L, M), dev_status, stream)
                         : dq_bucket_norms(L, dev_grads, worker_stride_elems, M, dev_norms, dev_status, stream);
    if (rc != DQ_OK) return rc;
    return dq_choose_bits(L, dev_norms, M, rule, dev_b, scratch, choose, dev_status, stream);
}

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
    const RoundRoute route = route_of(a, true);
    if (route == kTwoKernels) {
        rc = launch<false>(a, map, L, true, static_cast<cudaStream_t>(stream));
        if (rc != DQ_OK) return rc;
        return average(L, dev_packed, packed_stride_words, dev_norms, M, dev_b, dev_out, update, lr, dev_status, stream);
    }
    fill_average(a, dev_out, update, lr);
    if (route == kCtaTiles) return launch_tiles(a, L, true, static_cast<cudaStream_t>(stream));
    return launch<true>(a, map, L, true, static_cast<cudaStream_t>(stream));
}

extern "C" size_t dq_round_workspace_bytes(const dq_layout_t* L, int32_t M)
{
    if (!L || M < 1) return 0;
    // (behind it, scratch of the calls a layout may need besides)
    const size_t scratch = dq_tensor_norms_scratch_bytes(L, M) + dq_choose_bits_scratch_bytes(L, M);
    return rule_workspace_bytes() + scratch;
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
    const bool given = !dq_norms_inside(L);
    if (given) {
        if (L->whole_tensor) {
            const size_t rule_bytes = rule_workspace_bytes();
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
    attach_rule(a, next_rule, M, ws);
    const RoundRoute route = route_of(a, given);
    if (route == kTwoKernels) {
        // the next b is chosen at the end of the first kernel, which leaves its own for the second
        a.rule.this_b = reinterpret_cast<int32_t*>(ws + kThisBOffset);
        rc = launch<false>(a, map, L, given, static_cast<cudaStream_t>(stream));
        if (rc != DQ_OK) return rc;
        return average(L, dev_packed, packed_stride_words, dev_norms, M, a.rule.this_b, dev_out, update, lr, dev_status, stream);
    }
    fill_average(a, dev_out, update, lr);
    if (route == kCtaTiles) return launch_tiles(a, L, given, static_cast<cudaStream_t>(stream));
    return launch<true>(a, map, L, given, static_cast<cudaStream_t>(stream));
}
