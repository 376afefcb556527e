// The norm kernels of dq_round.cuh.
#define DQ_ROUND_KERNELS
#include "dq_round.cuh"

template int dq_launch_norms<kWarpBuckets, false>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
template int dq_launch_norms<kWarpBuckets, true>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
template int dq_launch_norms<kTeamBuckets, false>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
template int dq_launch_norms<kTeamBuckets, true>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
template int dq_launch_norms<kOddBuckets, false>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
template int dq_launch_norms<kOddBuckets, true>(const RoundArgs&, const CUtensorMap&, int, int64_t, cudaStream_t);
