// The streaming scorer for 8-bit metadata.
#include "score_stream.cuh"

namespace kvswap {
KVSWAP_SCORE_STREAM_ROWS(KVSWAP_E4M3, 32)
}  // namespace kvswap
