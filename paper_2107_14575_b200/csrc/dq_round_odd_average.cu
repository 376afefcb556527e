// The quantize-and-average kernel of dq_round.cuh for other buckets of up to 992 elements, l2 norms.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_round<kOddBuckets, true, false>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
