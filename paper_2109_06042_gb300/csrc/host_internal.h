// host_internal.h -- host helpers shared by the C ABI (mhs_api.cpp) and the
// serving loop (server.cpp).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <functional>
#include <vector>

#include "mhs.h"
#include "mhs_internal.h"

namespace mhs {

// Record a thread-local message for mhs_last_error() and return st.
mhs_status set_error(mhs_status st, const char *fmt, ...);

// The library's stream-ordered memory pool of a device (freed blocks are
// kept for reuse, so load/free loops do not reach the driver).
cudaError_t pool_for(int dev, cudaMemPool_t *out);

// Tile shape of the tcgen05 contraction for a load: explicit options, else
// the autotuner's table (tiles.cpp), else the defaults.
struct TileChoice {
    int32_t tile_n;       // 128 or 256 columns per tile
    int32_t group_rows;   // row blocks per L2 group of the tile order
    int32_t half_stages;  // 1: a K block shared in one half is loaded as that half
    int32_t from_table;   // 1: the table gave the shape
};
// typical_rows: the larger of n and m (a batch: its mean over the instances).
TileChoice choose_tiles(int32_t count, int64_t typical_rows, const mhs_options &opt);
const char *tile_table_path();

// InstState::layout_sorted for an mhs_layout option.  The bit-packed passes gain
// from the degree layout only where many rows end early on a rare vertex;
// measured, load and kernelization (us) by degree / in input order:
//   uniform 4,000 x 8,000     314 / 287     8,000 x 16,000     406 / 394
//   power law 5,000 x 10,000  584 / 586     10,000 x 20,000    980 / 1046
constexpr int64_t kBitsInputOrder = 10000;  // hyperedges (of the largest instance)
inline int32_t layout_code(int32_t layout, int32_t contraction, int64_t m) {
    if (layout == MHS_LAYOUT_AUTO && contraction == kPopcount && m <= kBitsInputOrder) return 0;
    return layout == MHS_LAYOUT_INPUT ? 0 : layout == MHS_LAYOUT_SORTED ? 1 : 2;
}

// Are the len >= 1 ids strictly ascending and within [0, n)?  Then they are
// distinct.  (No early exit: the loop is short and vectorises.)
inline bool ascending_row(const int32_t *ids, int64_t len, int32_t n) {
    int32_t bad = (ids[0] < 0) | (ids[len - 1] >= n);
    for (int64_t k = 1; k < len; ++k) bad |= ids[k - 1] >= ids[k];
    return !bad;
}

// One request of a group that solve_sparse_group reduces together.
struct GroupItem {
    int32_t n, m;
    int64_t k;                       // in: the budget; out: what rule FE left of it
    const int32_t *ptr, *vtx, *dem;  // host CSR and demands, already checked
    std::vector<int32_t> *vout, *eout, *dout, *forced;  // the result lists
    int32_t rounds;
    mhs_status status;               // of this request
};
// Reduces the group on the sparse path, all requests in the same launches, on
// `stream` (synchronises it).  reserve is asked before anything is allocated:
// may the group hold so many bytes on the device?  *again: it may not, the path
// does not pay for this group, or it failed in a way that need not be every
// request's; nothing has been written.  opt: contraction auto.
mhs_status solve_sparse_group(const mhs_options &opt, cudaStream_t stream,
                              std::vector<GroupItem> &group,
                              const std::function<bool(int64_t)> &reserve, bool *again);
// Would MHS_CONTRACT_AUTO try the sparse path with these options?
bool auto_takes_sparse(const mhs_options &opt);

// Blocks of kPinnedBlock bytes of page-locked host memory from a
// process-wide slab.  cudaMallocHost / cudaFreeHost cost tens of
// microseconds and cudaFreeHost synchronises the device, which every
// load / free would otherwise pay.  Blocks are 256-byte aligned.
constexpr size_t kPinnedBlock = 1024;
void *pinned_block();  // nullptr if page-locked memory is unavailable
void pinned_release(void *p);

// Larger page-locked staging buffers (a batch's instance states and tensor
// maps), from a process-wide pool in size classes of powers of two from
// 64 KB; a buffer goes back to the pool, never to the system.  *cls receives
// the class to give back; nullptr if page-locked memory is unavailable.
void *pinned_take(size_t bytes, size_t *cls);
void pinned_give(void *p, size_t cls);

}  // namespace mhs
