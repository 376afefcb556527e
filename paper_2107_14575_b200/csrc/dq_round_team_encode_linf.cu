// The quantizer kernel of dq_round.cuh for buckets of 2048 and 4096 elements, l-inf norms.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_round<kTeamBuckets, false, true>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
