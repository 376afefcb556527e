// The quantize-and-average kernel of dq_round.cuh for buckets of up to 1024 elements, l2 norms.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_round<kWarpBuckets, true, false>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
