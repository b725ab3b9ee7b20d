// The one-cluster predictor for 8-bit and fp32 metadata.
#include "score_select_cluster.cuh"

namespace kvswap {
KVSWAP_SCORE_SELECT_ROWS(KVSWAP_E4M3, 32)
KVSWAP_SCORE_SELECT_ROWS(KVSWAP_F32, 16)
KVSWAP_SCORE_SELECT_ROWS(KVSWAP_F32, 32)
}  // namespace kvswap
