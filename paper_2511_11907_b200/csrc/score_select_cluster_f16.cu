// The one-cluster predictor for fp16 metadata of rank 32.
#include "score_select_cluster.cuh"

namespace kvswap {
KVSWAP_SCORE_SELECT_ROWS(KVSWAP_F16, 32)
}  // namespace kvswap
