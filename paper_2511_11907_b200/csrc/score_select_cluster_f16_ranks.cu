// The one-cluster predictor for fp16 metadata of ranks 16 and 64.
#include "score_select_cluster.cuh"

namespace kvswap {
KVSWAP_SCORE_SELECT_ROWS(KVSWAP_F16, 16)
KVSWAP_SCORE_SELECT_ROWS(KVSWAP_F16, 64)
}  // namespace kvswap
