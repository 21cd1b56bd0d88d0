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
// How a search runs, beside its parameters; each field as in SearchArgs
// (search_kernel.cuh).  overlapped: the caller's launches overlap on the GPU
// (the server's), so the form of the search is chosen for a full GPU, whatever
// this launch's own number of queries.
struct SearchForm {
    bool overlapped = false;
    uint32_t form = 0;
    uint32_t *form_out = nullptr;
    long long wait_cycles = 0;
    uint32_t *gave_up = nullptr;
    uint32_t mute = 0;
};
int search_batched(bang_index *ix, const void *queries, uint32_t nq, const uint32_t *k_per_q,
                   const uint32_t *L_per_q, uint32_t k_max, uint32_t L_max, const bang_search_params *params,
                   uint32_t *out_ids, float *out_dist, void *stream, const SearchForm &form);
}  // namespace bang

// For tests and measurements, exported but not part of the ABI (bang.h): the
// calls of the same names with the form of the search, the limit of its waits
// and a query whose first expander stays silent chosen by the caller.
extern "C" {
// bang_search (k_per_q and L_per_q null) or bang_search_batched; *form_out (host,
// may be null) receives the form that ran.
int bang_internal_search(bang_index *ix, const void *queries, uint32_t nq, const uint32_t *k_per_q,
                         const uint32_t *L_per_q, uint32_t k, uint32_t L, const bang_search_params *params,
                         uint32_t *out_ids, float *out_dist, void *stream, uint32_t form, long long wait_cycles,
                         uint32_t mute, uint32_t *form_out);
// The form (counted as SearchArgs::form) that a search of such an index with
// aligned rows takes on a GPU of `sms` SMs, and its shared memory per query.
// link: vectors read over the host link.  Needs no GPU.
int bang_internal_form(int dtype, uint64_t n, uint32_t d, uint32_t M, uint32_t R, uint32_t mode, uint32_t log2z,
                       uint32_t L, uint32_t k, uint32_t nq, uint32_t link, uint32_t batched, uint32_t overlapped,
                       uint32_t sms, uint32_t *bytes);
// The launches of a server after this call; no request may be pending or running.
int bang_internal_server_form(struct bang_server *s, uint32_t form, long long wait_cycles, uint32_t mute);
int bang_internal_build_shard_graph(int device, const void *base, int dtype, uint64_t n, uint32_t d,
                                    const float *centres, uint32_t S, uint32_t ell, uint32_t R, uint32_t Lb,
                                    float alpha, float batch_frac, uint32_t log2z, uint32_t iter_cap, uint32_t *adj,
                                    uint32_t *shard_of, void *stream, uint32_t form, long long wait_cycles,
                                    uint32_t mute);
}
