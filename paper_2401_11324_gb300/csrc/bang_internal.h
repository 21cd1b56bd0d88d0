// Internal helpers shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cstdint>
#include <string>

struct bang_index;
struct bang_search_params;

namespace bang {
// Record the message returned by bang_last_error() for the calling thread.
void set_error(const std::string &msg);
// CUDA device and placement flags of an index.
int index_device(const bang_index *ix);
uint32_t index_placement(const bang_index *ix);
// Where a caller's pointer lives: 0 host memory (pageable or page-locked),
// 1 device memory of `device` or managed memory, 2 device memory of another
// GPU (which kernels on `device` must not be given).
int pointer_kind(const void *p, int device);
// bang_search_batched for a caller whose launches overlap on the GPU (the
// server): with `overlapped` the form of the search is chosen for a full GPU,
// whatever this launch's own number of queries.
int search_batched(bang_index *ix, const void *queries, uint32_t nq, const uint32_t *k_per_q,
                   const uint32_t *L_per_q, uint32_t k_max, uint32_t L_max, const bang_search_params *params,
                   uint32_t *out_ids, float *out_dist, void *stream, bool overlapped);
}  // namespace bang
