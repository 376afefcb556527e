// The quantizer kernel of dq_round.cuh for other buckets of up to 992 elements, l-inf norms.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_round<kOddBuckets, false, true>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
