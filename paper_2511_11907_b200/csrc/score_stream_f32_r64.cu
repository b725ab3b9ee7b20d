// The scorers for fp32 metadata of rank 64.
#include "score_select_cluster.cuh"
#include "score_stream.cuh"

namespace kvswap {
KVSWAP_SCORE_STREAM_ROWS(KVSWAP_F32, 64)
KVSWAP_SCORE_SELECT_ROWS(KVSWAP_F32, 64)
}  // namespace kvswap
