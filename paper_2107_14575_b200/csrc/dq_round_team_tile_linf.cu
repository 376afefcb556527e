// The kernel of dq_round.cuh in which a CTA takes its tiles through the workers: buckets of 2048 elements, l-infinity norms.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_tile_round<kTeamBuckets, true>(const RoundArgs&, int, int64_t, cudaStream_t);
