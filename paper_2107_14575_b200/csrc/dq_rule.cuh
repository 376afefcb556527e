// The bit rule of Eq. 17 on the device, for the kernels of dq_choose_bits and for kernels that end
// with the choice of the next b.
//
//   G-bar^2 = (1/M) sum over workers and buckets of norm^2        (Lemma 1)
//   x       = sqrt(T/eps_hat) * alpha^((T-1-t)/2) * G-bar
//   b       = smallest b in [b_min, b_max] with 2^(b-1) - 1 >= x   (else b_max)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dq.h"

struct RuleArgs {
    double coef;                  // sqrt(T/eps_hat) * alpha^((T-1-t)/2), a host scalar
    int32_t b_min, b_max, fixed_b;
    int32_t M;
    double* partial;              // one sum per CTA
    uint32_t* arrivals;           // CTAs that have written theirs; 0 between launches
    int32_t* this_b;              // where the call's own b is kept for the kernel that follows, or null
};

// Host: the rule's argument check and its coefficient (dq_bits.cu).
int dq_check_rule(const dq_rule_t* rule);
RuleArgs dq_rule_args(const dq_rule_t* rule, int32_t M);

#ifdef __CUDACC__

// Sum over the CTA in a fixed order: shuffle tree inside each warp, then the warp sums
// added in warp order by thread 0.  Returns the total in thread 0.
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double total = 0.0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) total += sh[w];
    }
    return total;
}

// One thread: b from the sum of squared norms, into dev_b[0] and its s into dev_b[1].
__device__ __forceinline__ void write_next_bits(const RuleArgs& r, const double sum, int32_t* dev_b, int32_t* status)
{
    int b;
    if (r.fixed_b != 0) {
        b = r.fixed_b;
    } else {
        const double x = r.coef * sqrt(sum / (double)r.M);
        b = r.b_max;
        if (isfinite(x)) {
            for (int c = r.b_min; c <= r.b_max; ++c) {
                if ((double)((1 << (c - 1)) - 1) >= x) { b = c; break; }
            }
        } else {
            atomicOr(status, DQ_STAT_NONFINITE);
        }
    }
    dev_b[0] = b;
    dev_b[1] = (1 << (b - 1)) - 1;
}

// End of a kernel whose CTAs all come here: `v` is a thread's share of the sum of squared norms.
// Every CTA leaves its sum in `partial`, the last one to arrive adds them up in CTA order and writes
// the next b -- in place, since by then every CTA has read this one's.  The counter wraps to 0 by
// itself, so it is ready for the next launch.  With `norms` (a call that could not run: all CTAs
// agree on that) the sum is taken from the n norms in memory instead.  b: this call's.  sh: NT / 32
// doubles and one word.
template <int NT>
__device__ __forceinline__ void rule_at_end(const RuleArgs& r, const double v, const float* norms, const int64_t n, double* sh,
                                            int32_t* dev_b, const int b, int32_t* status)
{
    uint32_t* last = reinterpret_cast<uint32_t*>(sh + NT / 32);
    const bool sums = r.fixed_b == 0 && norms == nullptr;
    if (sums) {
        const double mine = block_sum<NT>(v, sh);
        if (threadIdx.x == 0) r.partial[blockIdx.x] = mine;       // one entry per CTA: in bounds by construction
    } else {
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        __threadfence();
        *last = atomicInc(r.arrivals, gridDim.x - 1) == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (!*last) return;
    double acc = 0.0;
    if (sums) {
        __threadfence();
        for (uint32_t i = threadIdx.x; i < gridDim.x; i += NT) acc += __ldcg(r.partial + i);
    } else if (r.fixed_b == 0) {
        for (int64_t i = threadIdx.x; i < n; i += NT) {
            const double x = (double)norms[i];
            acc = fma(x, x, acc);
        }
    }
    const double sum = block_sum<NT>(acc, sh);
    if (threadIdx.x == 0) {
        if (r.this_b) *r.this_b = b;
        write_next_bits(r, sum, dev_b, status);
    }
}

#endif  // __CUDACC__
