// The projection of short prompts (project_keys_short.cu): plan and launch.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace kvswap {

struct ShortPlan {
  int tiles;                 // token tiles per row
  int cluster, hpc;          // CTAs per tile, heads (or pairs of 64-channel heads) per CTA
  int64_t items;             // (sequence, metadata head, tile)
  bool pair;
};
bool plan_project_keys_short(const Problem& p, int n_begin, int n_end, ShortPlan* pl);
cudaError_t launch_project_keys_short(const Problem& p, const ShortPlan& pl, const CUtensorMap& map_k, const float* proj,
                                      void* meta, int n_begin, int n_end, uint32_t* err, cudaStream_t st);

}  // namespace kvswap
