// The streaming scorer for fp32 metadata.
#include "score_stream.cuh"

namespace kvswap {
KVSWAP_SCORE_STREAM_ROWS(KVSWAP_F32, 16)
KVSWAP_SCORE_STREAM_ROWS(KVSWAP_F32, 32)
}  // namespace kvswap
