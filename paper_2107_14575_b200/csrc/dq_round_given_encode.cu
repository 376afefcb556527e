// The quantizer kernel of dq_round.cuh for norms that are given.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_round<kGivenNorms, false, false>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
