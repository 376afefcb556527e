// The kernel of dq_round.cuh in which a CTA takes its tiles through the workers: given norms.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_tile_round<kGivenNorms, false>(const RoundArgs&, int, int64_t, cudaStream_t);
