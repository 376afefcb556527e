// The quantize-and-average kernel of dq_round.cuh for norms that are given.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_round<kGivenNorms, true, false>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
