// sbh_sort.cuh -- the Morton-code and radix-sort step of the tree build (defined in sbh_build.cu),
// declared for the other translation unit that runs it.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sbh_internal.cuh"

namespace sbh {

constexpr int kSortThreads = 512;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kPasses = 8;  // of 8 bits: an even number, so that the sort ends in the buffers it began in
constexpr int kQueryPasses = 3;

// Zeroed before each sort
struct SortHead {
    uint32_t bounds[8];          // ordered-integer maxima of -x, -y, -z, x, y, z; bad coordinates, bad weights
    unsigned done[3];            // blocks of k_bounds, k_morton, the last pass that are through
    uint32_t next_tile[kPasses]; // tiles drawn in each pass
    int32_t error;               // nonzero: a bounded wait gave up
    int32_t hist[kPasses][256];  // counts of each digit, then where its run starts
};

// bytes of one of the two status arrays that a sort of n keys needs
size_t sort_status_bytes(int64_t n);

// Enqueue the root cube (c4, c2), the codes and their stable sort: k[0], v[0] get the sorted codes and
// the input index of each; k[1], v[1] are scratch of the same size, status 2 x sort_status_bytes(n).
// Where a bounded wait gave up, H->error is set when the sort has run, k[0] and v[0] are damaged, and
// *report (unless it is null) is -1.
cudaError_t sort_codes(const float* pts, const float* w, int64_t n, uint64_t* const k[2], int32_t* const v[2],
                       SortHead* H, uint32_t* status, TreeCtrl* c4, TreeCtrl* c2, int32_t* report, cudaStream_t s);

// Order of n queries by their Morton codes in twice the tree's root cube (24 bits, three passes): order[i]
// is the query to take at place i, unless *error is set when the sort has run. Both are in *scratch,
// for the caller to dfree when the work that reads them is enqueued. Where there is no memory for it,
// where the stream is being captured (the scratch would be the graph's) or n is beyond the sort's
// counters, nothing is done and order stays null.
cudaError_t sort_queries(const float* q, int64_t n, const TreeCtrl* ctrl, void** scratch, const int32_t** order,
                         const int32_t** error, cudaStream_t s);

}  // namespace sbh
