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

// One warp, all of it (lane 0 has the sum of squared norms): b into dev_b[0] and its s into dev_b[1].  The sixteen
// thresholds are looked at by a lane each: one after the other, with a conversion to fp64 in every step, they took up to
// 400 cycles of the tail of a round.
__device__ __forceinline__ void write_next_bits(const RuleArgs& r, double sum, int32_t* dev_b, int32_t* status)
{
    const int lane = threadIdx.x & 31;
    int b;
    if (r.fixed_b != 0) {
        b = r.fixed_b;
    } else {
        sum = __shfl_sync(0xffffffffu, sum, 0);
        const double x = r.coef * sqrt(sum / (double)r.M);
        const int c = lane + 1;
        const uint32_t enough = __ballot_sync(0xffffffffu, c >= r.b_min && c <= r.b_max && (double)((1 << lane) - 1) >= x);
        b = r.b_max;
        if (isfinite(x)) {
            if (enough) b = __ffs(enough);
        } else if (lane == 0) {
            atomicOr(status, DQ_STAT_NONFINITE);
        }
    }
    if (lane == 0) {
        dev_b[0] = b;
        dev_b[1] = (1 << (b - 1)) - 1;
    }
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
        // (eight at a time: a load behind the other's addition costs the round its latency each time)
        for (uint32_t first = threadIdx.x; first < gridDim.x; first += 8 * NT) {
            double x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = first + k * NT < gridDim.x ? __ldcg(r.partial + first + k * NT) : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) acc += x[k];
        }
    } else if (r.fixed_b == 0) {
        for (int64_t i = threadIdx.x; i < n; i += NT) {
            const double x = (double)norms[i];
            acc = fma(x, x, acc);
        }
    }
    const double sum = block_sum<NT>(acc, sh);
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0 && r.this_b) *r.this_b = b;
        write_next_bits(r, sum, dev_b, status);
    }
}

#endif  // __CUDACC__
