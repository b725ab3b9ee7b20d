// The streaming scorer for fp16 metadata of ranks 16 and 64.
#include "score_stream.cuh"

namespace kvswap {
KVSWAP_SCORE_STREAM_ROWS(KVSWAP_F16, 16)
KVSWAP_SCORE_STREAM_ROWS(KVSWAP_F16, 64)
}  // namespace kvswap
