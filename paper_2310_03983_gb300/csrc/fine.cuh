// fine.cuh -- blocked Floyd-Warshall over 64 x 64 tiles for matrices too small to fill the GPU with
// 128 x 128 tiles (fine.cu).
#pragma once

#include "tgemm.cuh"

namespace apsp {

// fw_loop closes matrices of kFineMinN < n <= kFineMaxN with 64-vertex blocks.  Up to 128 vertices the
// 128-vertex loop is one launch over one tile; above kFineMaxN its larger tiles do more per load
// (n = 3200: 2311 us against 2461 with 128-vertex blocks for int32, 2513 against 2544 with weights up
// to 10^6, 2312 against 2648 for float32; n = 3300: 2623 against 2588, 2819 against 2662, 2626 against 2783).
constexpr int64_t kFineMinN = 128, kFineMaxN = 3200;

// Device words of the counters block (Bound::counters): all zero between launches.
constexpr int kFineMaxStages = 8;  // of one launch
constexpr int kFineWords = 2 + 2 * kFineMaxStages;

// Closes the n x n block at d (16-byte aligned, ld % 4 == 0, normalised, n > kFineMinN) in place in two
// launches and one per 128 vertices, as the 128-vertex loop does.  wmax / wmult: the bound of the exact
// fp32 sequence for int32 storage (null: float32).
int fine_closure(void *d, int64_t n, int64_t ld, int dtype, int inf_i, const int *wmax, int64_t wmult,
                 int *counters, int trace_class, cudaStream_t s);

// The same for many graphs in lockstep, staged one below the other in d (rows x ld, each graph padded to
// whole 128-vertex blocks with isolated vertices, groups by decreasing nb; gsize: device, vertices of
// each graph, 0 for one to leave alone).  wmax[0]: the largest (n - 1) * weight of any graph.
int fine_batch(void *d, int64_t rows, int64_t ld, const GraphGroup *groups, int ngroups, const int *gsize, int dtype,
               int inf_i, const int *wmax, int *counters, cudaStream_t s);
int64_t fine_batch_tiles(const GraphGroup *groups, int ngroups);  // 64 x 64 tiles of one stage

}  // namespace apsp
