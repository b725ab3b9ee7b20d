// The streaming scorer for fp16 metadata of rank 32.
#include "score_stream.cuh"

namespace kvswap {
KVSWAP_SCORE_STREAM_ROWS(KVSWAP_F16, 32)
}  // namespace kvswap
