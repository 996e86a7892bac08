// kernels.cu -- encode, compaction, planning and the bit-packed DP / MD passes.
//
// Round structure (Algorithm 3, Section 4.1), all on the device:
//   plan(phase 0) -> encode A -> contract(DP or SE) -> compact_edges
//   plan(phase 1) -> clear A + encode A^T -> contract(MD) -> clear A^T -> compact_vertices
//   [rule FE at a fixpoint, fe.cu]
// (bit-packed: both operands are set before DP and cleared after MD.)  The
// contraction (contract_tc.cu: tcgen05 FP8) computes the pair counts of Eq. (1)
// / Eq. (2) tile by tile, the bit-packed passes (this file) 32 pairs to a
// word; neither writes them out: they turn them into the deletion flags of
// Algorithm 1 or the dominator counts of Algorithm 2.
#include <algorithm>

#include <cuda_runtime.h>

#include "bounded_wait.cuh"
#include "kernels.h"
#include "mhs_internal.h"

namespace mhs {

namespace {

constexpr uint8_t kFp8One = 0x38;  // 1.0 in E4M3


// Exclusive block scan of one value per thread (blockDim.x a multiple of
// 32, at most 1024).  *total receives the block total.
template <typename T>
__device__ T block_exclusive_scan(T x, T *total, T *sh /*[33]*/) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    T inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nwarps ? sh[lane] : T(0);
        T winc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, winc, o);
            if (lane >= o) winc += y;
        }
        if (lane < nwarps) sh[lane] = winc - w;
        if (lane == 31) sh[32] = winc;
    }
    __syncthreads();
    T r = inc - x + sh[warp];
    *total = sh[32];
    __syncthreads();
    return r;
}

// Locate the instance owning global item `g` in a prefix array off[0..count].
template <typename T>
__device__ __forceinline__ int find_owner(const T *off, int count, T g) {
    int lo = 0, hi = count;  // off[lo] <= g < off[hi]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (off[mid] <= g) lo = mid; else hi = mid;
    }
    return lo;
}

// ---------------------------------------------------------------- setup --

// Structural checks of device-resident inputs (blockIdx.y = instance):
// edge_ptr starts at 0, is non-decreasing and ends at nnz; vertex ids lie in
// [0, n); demands are >= 1.
__global__ void k_validate(InstState *st, int count) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (tid == 0) {
        if (s.eptr[0] != 0 || (int64_t)s.eptr[s.m0] != s.nnz0) atomicOr(&s.status, kErrBadPtr);
    }
    for (int64_t e = tid; e < s.m0; e += stride) {
        if (s.eptr[e + 1] < s.eptr[e]) atomicOr(&s.status, kErrBadPtr);
        if (s.f[e] < 1) atomicOr(&s.status, kErrBadDemand);
        if (s.f[e] >= kBigDemand) s.big_demand = 1;
    }
    for (int64_t p = tid; p < s.nnz0; p += stride) {
        int32_t v = s.evtx[p];
        if (v < 0 || v >= s.n0) atomicOr(&s.status, kErrBadVertex);
    }
}

// OR of the instances' status words (and kSawBigDemand), so that a batch load
// reads back one word instead of every instance's state.
__global__ void k_status_or(const InstState *st, int count, int32_t *out) {
    int32_t x = 0;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < count; b += gridDim.x * blockDim.x)
        x |= st[b].status | (st[b].big_demand ? kSawBigDemand : 0);
    x = __reduce_or_sync(0xffffffffu, x);
    if ((threadIdx.x & 31) == 0 && x) atomicOr(out, x);
}

// Batch inputs from device arrays: convert the global int64 CSR offsets of
// instance b (hyperedges [e0[b], e0[b] + m0)) to its local int32 offsets.
__global__ void k_localize_ptr(InstState *st, int count, const int64_t *gptr, const int64_t *e0) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    int32_t *eptr = const_cast<int32_t *>(s.eptr);
    const int64_t base = gptr[e0[b]];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= s.m0;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = gptr[e0[b] + i] - base;
        eptr[i] = (x >= 0 && x <= s.nnz0) ? (int32_t)x : -1;
    }
}

// Gather gptr[e0[b]] for b in [0, count] (instance boundaries of a batch).
__global__ void k_gather_bounds(const int64_t *gptr, const int64_t *e0, int64_t *out, int count) {
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b <= count; b += gridDim.x * blockDim.x)
        out[b] = gptr[e0[b]];
}

// Chained-scan compaction of a single instance (see k_compact_edges): status
// word epochs (30 bits) and the time limit of a wait on a predecessor chunk.
constexpr uint32_t kEpochMask = (1u << 30) - 1;
constexpr uint64_t kChainWaitNs = 2000000000ull;  // 2 s

// Zero the occupancy bits of phase p's operand for its first R rows (all
// row blocks a tile over R rows can touch).  Block-cooperative.
__device__ __forceinline__ void zero_occupancy(InstState &s, int p, int32_t R, int64_t first,
                                               int64_t stride) {
    if (!s.occ[p]) return;
    const int64_t words = (int64_t)((R + 255) / 256) * 2 * s.occ_words[p];
    for (int64_t w = first; w < words; w += stride) s.occ[p][w] = 0;
}

// Round state and vertex id maps (one block per instance).  In input
// layout the hyperedge maps are the identity too; in sorted layout they are
// filled by the k_layout_* kernels below, whose buckets (v_cnt) and cursors
// (v_deg) are zeroed here.
// (blockIdx.y = instance; the blocks of an instance split its ranges)
__global__ void k_init(InstState *st, int count, int32_t max_rounds) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    const int32_t t0 = blockIdx.x * blockDim.x + threadIdx.x, ts = gridDim.x * blockDim.x;
    for (int32_t v = t0; v < s.n0; v += ts) { s.v_o2c[v] = v; s.v_c2o[v] = v; }
    if (s.layout_sorted == 2)  // degrees for the vertex layout (v_maxf is free until MD)
        for (int32_t v = t0; v < s.n0; v += ts) s.v_maxf[v] = 0;
    if (s.layout_sorted) {
        for (int32_t v = t0; v <= s.n0; v += ts) { s.v_cnt[v] = 0; s.v_deg[v] = 0; }
    } else {
        for (int32_t e = t0; e < s.m0; e += ts) { s.e_o2c[e] = e; s.e_c2o[e] = e; }
    }
    if (s.forced)
        for (int32_t v = t0; v < s.n0; v += ts) s.forced[v] = 0;
    if (s.v_dirty)
        for (int32_t v = t0; v < s.n0; v += ts) s.v_dirty[v] = 0;
    if (s.v_dirty_rb)
        for (int32_t w = t0; w < s.At_rows / 128; w += ts) s.v_dirty_rb[w] = 0;
    if (s.e_dirty_rb)
        for (int32_t w = t0; w < s.A_rows / 128; w += ts) s.e_dirty_rb[w] = 0;
    zero_occupancy(s, 0, s.m0, t0, ts);
    if (s.scan_status)
        for (int32_t c = t0; c < s.scan_chunks; c += ts) s.scan_status[c] = 0;
    if (t0 == 0) {
        s.n = s.n0; s.m = s.m0; s.m_dp = s.m0; s.n_next = s.n0;
        s.rounds = 0; s.active = s.status == 0; s.max_rounds = max_rounds; s.changed = 0;
        s.dp_deleted = 0; s.md_deleted = 0; s.has_loose = 0; s.bounds_deleted = 0;
        s.fe_stage = 0; s.fe_passes = 0; s.md_full = 1; s.skip_a = 0; s.skip_at = 0;
    }
}

// Degree layout, step 1 (blockIdx.y = instance): vertex degrees into v_maxf.
__global__ void k_vertex_degrees(InstState *st, int count) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    if (s.layout_sorted != 2 || s.status) return;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < s.nnz0;
         p += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&s.v_maxf[s.evtx[p]], 1);
}

// Degree layout, step 2 (one block of 1024 threads per instance): vertices
// grouped by degree class floor(log4(deg)) in ascending order, input order
// inside a class (a stable counting sort).  With skewed degrees, sorting
// hyperedges by their smallest position then places each hyperedge by its
// rarest vertex: the rows of a row block share rare vertices, and their
// popular vertices fall in the few K blocks at the end, so far fewer
// (row block, K block) pairs are occupied.  Near-uniform degrees keep the
// input order (one or two classes), and with it any locality.
constexpr int kDegClasses = 16;
__device__ __forceinline__ int deg_class(int32_t d) {
    return d <= 1 ? 0 : min((31 - __clz(d)) / 2, kDegClasses - 1);
}
__global__ void __launch_bounds__(1024) k_vertex_layout(InstState *st, int count) {
    __shared__ int32_t start[kDegClasses];
    __shared__ int32_t wcnt[32][kDegClasses];  // this chunk: per warp, per class
    const int b = blockIdx.x;
    if (b >= count) return;
    InstState &s = st[b];
    if (s.layout_sorted != 2 || s.status) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < kDegClasses) start[threadIdx.x] = 0;
    __syncthreads();
    for (int32_t v = threadIdx.x; v < s.n0; v += blockDim.x) atomicAdd(&start[deg_class(s.v_maxf[v])], 1);
    __syncthreads();
    if (threadIdx.x == 0) {  // exclusive prefix over the classes
        int32_t acc = 0;
        for (int c = 0; c < kDegClasses; ++c) { const int32_t x = start[c]; start[c] = acc; acc += x; }
    }
    __syncthreads();
    for (int32_t base = 0; base < s.n0; base += blockDim.x) {
        const int32_t v = base + threadIdx.x;
        const int c = v < s.n0 ? deg_class(s.v_maxf[v]) : -1;
        const uint32_t peers = __match_any_sync(0xffffffffu, c);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (lane < kDegClasses) wcnt[warp][lane] = 0;
        __syncwarp();
        if (c >= 0 && rank == 0) wcnt[warp][c] = __popc(peers);
        __syncthreads();
        if (threadIdx.x < kDegClasses) {  // per class: prefix over the warps, then advance
            int32_t acc = start[threadIdx.x];
            for (int w = 0; w < 32; ++w) { const int32_t x = wcnt[w][threadIdx.x]; wcnt[w][threadIdx.x] = acc; acc += x; }
            start[threadIdx.x] = acc;
        }
        __syncthreads();
        if (c >= 0) {
            const int32_t pos = wcnt[warp][c] + rank;
            s.v_c2o[pos] = v;
            s.v_o2c[v] = pos;
        }
        __syncthreads();
    }
}

// Sorted layouts, step 1 (blockIdx.y = instance): key of each hyperedge =
// its smallest vertex id (layout 1) or position (layout 2), n0 if empty,
// kept in e_s; bucket counts in v_cnt.
__global__ void k_layout_keys(InstState *st, int count) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    if (!s.layout_sorted || s.status) return;
    const bool by_pos = s.layout_sorted == 2;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < s.m0;
         e += (int64_t)gridDim.x * blockDim.x) {
        int32_t key = s.n0;
        for (int32_t p = s.eptr[e]; p < s.eptr[e + 1]; ++p)
            key = min(key, by_pos ? s.v_o2c[s.evtx[p]] : s.evtx[p]);
        s.e_s[e] = key;
        atomicAdd(&s.v_cnt[key], 1);
    }
}

// Sorted layout, step 2 (one block per instance): bucket starts in v_deg,
// an exclusive scan of the n0 + 1 bucket counts, 8 consecutive buckets per
// thread.
__global__ void k_layout_scan(InstState *st, int count) {
    __shared__ int32_t sh[33];
    constexpr int kPer = 8;
    const int b = blockIdx.x;
    if (b >= count) return;
    InstState &s = st[b];
    if (!s.layout_sorted || s.status) return;
    const int32_t nb = s.n0 + 1;
    int32_t carry = 0;
    for (int32_t base = 0; base < nb; base += blockDim.x * kPer) {
        const int32_t i0 = base + threadIdx.x * kPer;
        int32_t x[kPer], sum = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            x[k] = i0 + k < nb ? s.v_cnt[i0 + k] : 0;
            sum += x[k];
        }
        int32_t tot;
        int32_t ex = carry + block_exclusive_scan<int32_t>(sum, &tot, sh);
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (i0 + k < nb) s.v_deg[i0 + k] = ex;
            ex += x[k];
        }
        carry += tot;
    }
}

// Sorted layout, step 3: place every hyperedge at the next slot of its
// bucket, in arbitrary order (steps 4 and 5 sort each bucket by input id,
// so that every load of an instance gets the same layout: sharded passes
// split the tile rows of replicas that must agree on it).
__global__ void k_layout_place(InstState *st, int count) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    if (!s.layout_sorted || s.status) return;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < s.m0;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t pos = atomicAdd(&s.v_deg[s.e_s[e]], 1);
        s.e_c2o[pos] = (int32_t)e;
        s.e_o2c[e] = pos;
    }
}

// Sorted layout, step 4: each hyperedge's final position is its bucket's
// start plus the number of hyperedges of the bucket with a smaller input id
// (after step 3, v_deg[key] is the bucket's end and v_cnt[key] its size).
// The cost is the sum of the squared bucket sizes; buckets hold the
// hyperedges sharing their smallest vertex (id or position).  Eight lanes per
// hyperedge: a lane per hyperedge took 32 us on the power-law instance (the
// largest bucket, entry by entry), eight take 20.
constexpr int kRankLanes = 8;
__global__ void k_layout_rank(InstState *st, int count) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    if (!s.layout_sorted || s.status) return;
    const int sub = threadIdx.x % kRankLanes;
    for (int64_t e0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x - threadIdx.x % 32) / kRankLanes;
         e0 < s.m0; e0 += (int64_t)gridDim.x * blockDim.x / kRankLanes) {
        const int64_t e = e0 + threadIdx.x % 32 / kRankLanes;
        int32_t lo = 0, hi = 0, rank = 0;
        if (e < s.m0) {
            const int32_t key = s.e_s[e];
            hi = s.v_deg[key];
            lo = hi - s.v_cnt[key];
        }
        for (int32_t p = lo + sub; p < hi; p += kRankLanes) rank += s.e_c2o[p] < (int32_t)e;
        __syncwarp();
#pragma unroll
        for (int o = kRankLanes / 2; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        if (sub == 0 && e < s.m0) s.e_o2c[e] = lo + rank;
    }
}

// Sorted layout, step 5: the position -> id map from the final positions.
__global__ void k_layout_commit(InstState *st, int count) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    if (!s.layout_sorted || s.status) return;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < s.m0;
         e += (int64_t)gridDim.x * blockDim.x)
        s.e_c2o[s.e_o2c[e]] = (int32_t)e;
}

// Hyperedge rows of round 1, by position; no bounds, no degrees (bit-packed) yet.
__global__ void k_edge_rows(InstState *st, int count) {
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    if (s.status) return;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < s.m0;
         r += (int64_t)gridDim.x * blockDim.x) {
        s.e_f[r] = s.f[s.e_c2o[r]];
        s.e_s[r] = -1;  // never tested: every hyperedge is a DP candidate
        s.e_del[r] = 0;
    }
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < s.n0;
         r += (int64_t)gridDim.x * blockDim.x) {
        if (s.Ab) s.v_deg[r] = 0;
        s.v_maxf[r] = 0;
    }
}

// ------------------------------------------------------------- planning --

// phase 0: rows = current hyperedges (DP); phase 1: rows = current vertices (MD).
// tc: 0 units of the bit-packed passes, 1 tcgen05 tiles (128 x plan->tile_n).
__global__ void k_plan(InstState *st, Plan *plan, int phase, int tc, BatchCounters *ctr) {
    __shared__ int32_t sh[33];
    __shared__ int64_t sh64[33];
    const int count = plan->count;
    int32_t rcarry = 0;
    int64_t tcarry = 0;
    int32_t act_any = 0;
    for (int base = 0; base < count; base += blockDim.x) {
        int b = base + threadIdx.x;
        int32_t rows = 0;
        int64_t tiles = 0;
        if (b < count) {
            const InstState &s = st[b];
            if (s.scan_status) {  // this phase's compaction: tickets from 0, a new epoch
                st[b].scan_ticket = 0;
                st[b].scan_epoch = (s.scan_epoch + 1) & kEpochMask;
            }
            if (s.active && s.status == 0) {
                // Incremental rounds (tcgen05 path): a pass without candidates
                // deletes nothing, so its operand is not needed.  DP: no
                // hyperedge lost a vertex since the previous DP pass, i.e. the
                // previous MD pass deleted none (FE sets md_full).  MD: this
                // round's DP pass deleted no hyperedge.
                int32_t skip = 0;
                if (tc && !s.no_skip && !s.md_full) {
                    if (phase == 0) skip = s.e_dirty_rb && s.md_deleted == 0;
                    else skip = s.v_dirty && s.dp_deleted == 0;
                }
                if (phase == 0) st[b].skip_a = skip;
                else st[b].skip_at = skip;
                // hyperedges to scatter: phase 0 the current ones; phase 1 the
                // rows DP saw (the fused pass clears A at those rows and sets
                // A^T for the ones DP kept)
                // (tcgen05 path: rounded up to a multiple of 32, so a warp's
                // group of 32 rows lies in one instance and starts at a
                // 32-aligned position: k_set_a_tc, k_set_md_tc, k_clear_at_tc)
                const bool none = phase == 0 ? skip : skip && s.skip_a;
                rows = !tc ? s.m : none ? 0 : (s.m + 31) & ~31;
                const int32_t R = phase == 0 ? s.m : s.n;
                tiles = tc ? tc_tiles(R, plan->tile_n) : pop_units(phase, R);
                act_any = 1;
            }
        }
        int32_t rtot;
        int32_t rex = block_exclusive_scan<int32_t>(rows, &rtot, sh);
        if (b < count) plan->row_off[b] = rcarry + rex;
        rcarry += rtot;
        int64_t ttot;
        int64_t tex = block_exclusive_scan<int64_t>(tiles, &ttot, sh64);
        if (b < count) plan->tile_off[b] = tcarry + tex;
        tcarry += ttot;
    }
    act_any = __syncthreads_or(act_any);
    if (threadIdx.x == 0) {
        plan->row_off[count] = rcarry;
        plan->tile_off[count] = tcarry;
        plan->total_rows = rcarry;
        plan->list_count = 0;
        plan->list_next = 0;
        plan->list_light = 0;
        plan->list_next_light = 0;
        plan->total_tiles = tcarry;
        plan->any_active = act_any;
        if (phase == 0 && ctr) {
            ctr->active = 0; ctr->n_alive = 0; ctr->m_alive = 0; ctr->dp_deleted = 0;
            ctr->md_deleted = 0; ctr->max_rounds_seen = 0; ctr->changed_any = 0;
            ctr->status_any = 0; ctr->n_done = 0;
        }
    }
}

// --------------------------------------------------------------- encode --

// Bit-packed operands (popcount path), from the original vertex lists.  Phase
// 0 (rows = current hyperedges) sets A[e'][v'] (K = current vertices) and
// At[v'][e'] (K = current hyperedges) and counts |e| (= I^E_ii) and deg(v).
// Phase 1 walks the rows the DP pass saw (e_prev), at their positions of
// then: its set pass takes the hyperedges that DP deleted out of At and
// deg(v) (= I^V_jj) and marks their vertices as MD candidates, and collects
// the maximum demand over the kept ones; its clear pass clears both after the
// MD pass, so the operands are all-zero between rounds.  Only incidences whose
// bit changed are counted, so a repeated id inside one hyperedge counts once.
template <int kPhase, bool kSet>
__global__ void __launch_bounds__(256) k_scatter(InstState *st, const Plan *plan) {
    // Eight lanes per row: what bounds this is the chain of a row's dependent
    // loads and atomics, not their number (a row per lane, walked by the warp
    // together, left 250 warps for 8,000 rows of 9: 25 us instead of 12).
    constexpr int kLanes = 8;
    const int lane = threadIdx.x & 31, sub = lane % kLanes;
    const int32_t total = plan->total_rows;
    const int32_t step = gridDim.x * (blockDim.x / kLanes);
    for (int32_t g0 = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x - lane) / kLanes); g0 < total;
         g0 += step) {
        const int32_t g = g0 + lane / kLanes;
        int32_t fresh = 0, ce = 0, e = 0;  // incidences that changed a bit
        InstState *sp = nullptr;
        if (g < total) {
            const int b = find_owner(plan->row_off, plan->count, g);
            sp = st + b;
            InstState &s = *sp;
            ce = g - plan->row_off[b];
            e = kPhase == 0 ? s.e_c2o[ce] : s.e_prev[ce];
            const bool gone = kPhase == 1 && s.e_o2c[e] < 0;  // DP deleted it
            const int32_t end = s.eptr[e + 1];
            const int32_t f = kPhase == 1 && kSet ? s.f[e] : 0;
            for (int32_t p = s.eptr[e] + sub; p < end; p += kLanes) {
                const int32_t cv = s.v_o2c[s.evtx[p]];
                if (cv < 0) continue;
                if (ce >= s.m || cv >= s.n) { atomicOr(&s.status, kErrCapacity); continue; }
                uint32_t *a = &s.Ab[(int64_t)ce * s.Ab_pitch + (cv >> 5)];
                uint32_t *at = &s.Atb[(int64_t)cv * s.Atb_pitch + (ce >> 5)];
                const uint32_t a_bit = 1u << (cv & 31), at_bit = 1u << (ce & 31);
                if (!kSet) {  // every set bit of these words is cleared by some thread
                    *a = 0;
                    *at = 0;
                } else if (kPhase == 0) {
                    if ((atomicOr(a, a_bit) & a_bit) == 0) {
                        atomicOr(at, at_bit);
                        atomicAdd(&s.v_deg[cv], 1);
                        ++fresh;
                    }
                } else if (gone) {
                    if (s.v_dirty) {
                        s.v_dirty[cv] = 1;
                        s.v_dirty_rb[cv >> 7] = 1;
                    }
                    if (atomicAnd(at, ~at_bit) & at_bit) atomicSub(&s.v_deg[cv], 1);
                } else {
                    atomicMax(&s.v_maxf[cv], f);
                }
            }
        }
        if (kSet && kPhase == 0) {
            __syncwarp();
#pragma unroll
            for (int o = kLanes / 2; o > 0; o >>= 1) fresh += __shfl_xor_sync(0xffffffffu, fresh, o);
            if (sp && sub == 0) {
                InstState &s = *sp;
                // a hyperedge whose size changed since the previous DP pass (or
                // never tested) makes its row block a DP candidate
                if (s.e_dirty_rb && s.e_s[ce] != fresh) s.e_dirty_rb[ce >> 7] = 1;
                s.e_s[ce] = fresh;
            }
        }
    }
}

// ------------------------------------------ dense operands (tcgen05) --
//
// The FP8 operands hold one byte per incidence, and DRAM and L2 move them in
// 32-byte sectors.  A byte store or a byte atomic into a sector L2 does not
// hold makes L2 read the sector from DRAM first; a store that covers the
// whole sector does not.  So the set and clear passes of the dense operands
// write whole sectors, and each sector has one writer:
//  * A (rows = hyperedges): a sector lies in one row; the warp that owns the
//    row builds the sector's byte mask in a shared-memory table from the
//    row's incidences and writes the sector once.
//  * A^T (rows = vertices, K = hyperedge positions after DP): the warp that
//    owns positions [32w, 32w + 32) owns sector w of every vertex row, so it
//    builds those sectors from its hyperedges' incidences.
//  * A clear writes the zero sector: every nonzero byte in it belongs to the
//    row being cleared (A) or to the same all-clearing pass (A^T).
// Warps take groups of 32 rows (A, few rows: 8); the plan rounds every
// instance's rows up to a multiple of 32, so a group lies in one instance at a
// 32-aligned position.  A group whose incidences exceed its table sets its bytes with
// atomics instead, for all of its sectors, so no sector is written both
// ways.  The table also deduplicates: a vertex listed twice in a hyperedge
// sets one bit, so sizes and degrees count it once.

constexpr int kSecWarps = 4;          // warps per block
constexpr int kSecTab = 512;          // table entries per warp (a power of two)
constexpr int kSecTabLog = 9;
// Up to this, the A set pass gives a warp 8 rows and half of its table, and the
// MD set pass gives a group's vertices to four warps: 24,000 rows are 760 warps
// of 32 on 152 SMs (power law 20,000 x 40,000: 35 us for A, 22 with 8; MD 32 and
// 29, later rounds 25 and 20; uniform 2,000 x 4,000, all of FP8, 390 and 363).  A
// batch fills the chip either way, and walks and empties less with 32.
constexpr int32_t kFewRows = 65536;

// One entry per sector: key << 32 | byte mask (bit b: byte b is 1.0).
struct SecTable {
    unsigned long long e[kSecTab];
};
constexpr unsigned long long kSecFree = ~0ull;

// Sets `bit` in the entry of `key`, inserting the key if absent: one shared
// atomic in the common cases (the key present: an OR; its slot free: a
// compare-and-swap).  False if the table is full (callers insert at most
// `slots` keys, a power of two, so it never is).
__device__ __forceinline__ bool sec_set(SecTable &t, uint32_t key, uint32_t bit,
                                        int slots = kSecTab) {
    uint32_t h = (key * 2654435761u) >> (32 - kSecTabLog) & (uint32_t)(slots - 1);
    const unsigned long long mine = (unsigned long long)key << 32;
    for (int p = 0; p < slots; ++p) {
        const unsigned long long cur = *reinterpret_cast<volatile unsigned long long *>(&t.e[h]);
        if (cur != kSecFree && (cur >> 32) == key) {
            atomicOr(&t.e[h], (unsigned long long)bit);
            return true;
        }
        if (cur == kSecFree) {
            const unsigned long long old = atomicCAS(&t.e[h], kSecFree, mine | bit);
            if (old == kSecFree) return true;
            if ((old >> 32) == key) {
                atomicOr(&t.e[h], (unsigned long long)bit);
                return true;
            }
        }
        h = (h + 1) & (uint32_t)(slots - 1);
    }
    return false;
}

// Four mask bits -> four bytes of 0 or 1.0 (bit i -> byte i).
__device__ __forceinline__ uint32_t fp8_bytes(uint32_t nib) {
    return ((nib * 0x00204081u) & 0x01010101u) * kFp8One;
}

__device__ __forceinline__ void store_sector(uint8_t *p, uint32_t m) {
    uint4 *q = reinterpret_cast<uint4 *>(p);
    q[0] = make_uint4(fp8_bytes(m & 15u), fp8_bytes((m >> 4) & 15u), fp8_bytes((m >> 8) & 15u),
                      fp8_bytes((m >> 12) & 15u));
    q[1] = make_uint4(fp8_bytes((m >> 16) & 15u), fp8_bytes((m >> 20) & 15u),
                      fp8_bytes((m >> 24) & 15u), fp8_bytes(m >> 28));
}

__device__ __forceinline__ void zero_sector(uint8_t *p) {
    uint4 *q = reinterpret_cast<uint4 *>(p);
    q[0] = make_uint4(0u, 0u, 0u, 0u);
    q[1] = make_uint4(0u, 0u, 0u, 0u);
}

// Occupancy bit of (row block rr / 128, K block cc / kOccK) of phase p's operand.
__device__ __forceinline__ void set_occupancy(InstState &s, int p, int32_t rr, int32_t cc) {
    const int32_t kblk = cc / kOccK;
    uint32_t *ow = s.occ[p] + (int64_t)(rr >> 7) * s.occ_words[p] + (kblk >> 5);
    const uint32_t ob = 1u << (kblk & 31);
    if (!(*reinterpret_cast<volatile uint32_t *>(ow) & ob)) atomicOr(ow, ob);
}

// Byte atomic (groups whose incidences exceed the table); true if the byte was 0.
__device__ __forceinline__ bool set_byte(uint8_t *row, int32_t cc) {
    uint32_t *w = reinterpret_cast<uint32_t *>(row + (cc & ~3));
    const uint32_t sh = 8u * (cc & 3);
    const uint32_t old = atomicOr(w, (uint32_t)kFp8One << sh);
    return ((old >> sh) & 0xffu) == 0;
}

// The incidences of a warp's 32 rows (lane l: row l, its list at p0, len
// entries), flattened: *start = the lane's first flat index, returns the total.
__device__ __forceinline__ int32_t rows_prefix(int lane, int32_t len, int32_t *start) {
    int32_t incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    *start = incl - len;
    return __shfl_sync(0xffffffffu, incl, 31);
}

// Flat index f -> its row (the last lane whose run starts at or before f).
__device__ __forceinline__ int flat_owner(int32_t start, int32_t f) {
    int r = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
        const int c = r + step;
        const int32_t sc = __shfl_sync(0xffffffffu, start, c & 31);
        if (c < 32 && sc <= f) r = c;
    }
    return r;
}

// Walks the incidences of a warp's 32 rows whose vertices are alive (lane l:
// row l, its vertex list at p0, flattened from *start, tot in all), calling
// fn(r, cv, x_r) with the row r, the vertex's current position cv and row
// r's payload x.  The loads of kWalkU chunks of 32 incidences are issued
// before any is used, so a warp has that many dependent pairs in flight.
constexpr int kWalkU = 4;
template <typename F>
__device__ __forceinline__ void walk_live(const InstState &s, int lane, int32_t p0,
                                          int32_t start, int32_t tot, int32_t x, F &&fn) {
    const int32_t *evtx = s.evtx;
    const int32_t *o2c = s.v_o2c;
    for (int32_t f0 = 0; f0 < tot; f0 += 32 * kWalkU) {
        int r[kWalkU];
        int32_t v[kWalkU], xr[kWalkU];
#pragma unroll
        for (int u = 0; u < kWalkU; ++u) {
            const int32_t f = f0 + 32 * u + lane;
            r[u] = flat_owner(start, f);
            const int32_t rp = __shfl_sync(0xffffffffu, p0, r[u]) + f -
                               __shfl_sync(0xffffffffu, start, r[u]);
            xr[u] = __shfl_sync(0xffffffffu, x, r[u]);
            v[u] = f < tot ? __ldg(evtx + rp) : -1;
        }
#pragma unroll
        for (int u = 0; u < kWalkU; ++u) v[u] = v[u] >= 0 ? __ldg(o2c + v[u]) : -1;
#pragma unroll
        for (int u = 0; u < kWalkU; ++u)
            if (v[u] >= 0) fn(r[u], v[u], xr[u]);
    }
}

// Empties the table entries the warp has written: fn(key, mask) writes an
// entry's sector and returns, through *ow / *ob, the occupancy word and bit
// it sets.  The lanes of one pass over 32 slots set each distinct word with
// one atomic.
template <typename F>
__device__ __forceinline__ void drain_table(SecTable &t, int lane, int slots, F &&fn) {
    __syncwarp();
    for (int base = 0; base < slots; base += 32) {
        const int i = base + lane;
        const unsigned long long ent = t.e[i];
        uint32_t *ow = nullptr;
        uint32_t ob = 0;
        if (ent != kSecFree) {
            t.e[i] = kSecFree;
            fn((uint32_t)(ent >> 32), (uint32_t)ent, &ow, &ob);
        }
        const unsigned grp = __match_any_sync(0xffffffffu, (unsigned long long)(uintptr_t)ow);
        const uint32_t bits = __reduce_or_sync(grp, ob);
        if (ow && lane == __ffs(grp) - 1) atomicOr(ow, bits);
    }
    __syncwarp();
}

__device__ __forceinline__ void init_table(SecTable &t, int lane) {
    for (int i = lane; i < kSecTab; i += 32) t.e[i] = kSecFree;
    __syncwarp();
}

// Occupancy word and bit of (row block rr / 128, K block cc / kOccK) of
// phase p's operand.
__device__ __forceinline__ uint32_t *occ_word(InstState &s, int p, int32_t rr, int32_t cc,
                                              uint32_t *ob) {
    const int32_t kblk = cc / kOccK;
    *ob = 1u << (kblk & 31);
    return s.occ[p] + (int64_t)(rr >> 7) * s.occ_words[p] + (kblk >> 5);
}

// Phase 0 set: A[e'][v'] = 1.0 for the current hyperedges' live incidences,
// |e| (= I^E_ii), the epilogue's row records and the occupancy bits of A.
__global__ void __launch_bounds__(32 * kSecWarps) k_set_a_tc(InstState *st, const Plan *plan) {
    __shared__ SecTable tab[kSecWarps];
    __shared__ int32_t wfresh[kSecWarps][32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    SecTable &t = tab[wib];
    init_table(t, lane);
    const int32_t total = plan->total_rows;
    const int32_t nw = gridDim.x * kSecWarps;
    // few rows: 8 to a warp, and half of its table
    const int32_t rows = total <= kFewRows ? 8 : 32;
    const int slots = total <= kFewRows ? kSecTab / 2 : kSecTab;
    for (int32_t g0 = (blockIdx.x * kSecWarps + wib) * rows; g0 < total; g0 += nw * rows) {
        const int b = find_owner(plan->row_off, plan->count, g0);
        InstState &s = st[b];
        const int32_t ce0 = g0 - plan->row_off[b];
        const int32_t ce = ce0 + lane;
        const bool row = lane < rows && ce < s.m;
        int32_t e = 0, p0 = 0, len = 0;
        if (row) {
            e = __ldg(s.e_c2o + ce);
            p0 = __ldg(s.eptr + e);
            len = __ldg(s.eptr + e + 1) - p0;
        }
        int32_t start;
        const int32_t tot = rows_prefix(lane, len, &start);
        const bool table = tot <= slots;
        const int32_t K = s.n;
        uint8_t *const A = s.A;
        const int64_t pitch = s.A_pitch;
        wfresh[wib][lane] = 0;
        __syncwarp();
        walk_live(s, lane, p0, start, tot, 0, [&](int r, int32_t cv, int32_t) {
            if (cv >= K) { atomicOr(&s.status, kErrCapacity); return; }
            if (table) {
                if (!sec_set(t, ((uint32_t)r << 26) | (uint32_t)(cv >> 5), 1u << (cv & 31), slots))
                    atomicOr(&s.status, kErrCapacity);
            } else {
                const int32_t rr = ce0 + r;
                if (set_byte(A + (int64_t)rr * pitch, cv)) atomicAdd(&wfresh[wib][r], 1);
                set_occupancy(s, 0, rr, cv);
            }
        });
        if (table) {
            drain_table(t, lane, slots, [&](uint32_t key, uint32_t m, uint32_t **ow, uint32_t *ob) {
                const int r = (int)(key >> 26);
                const int32_t c0 = (int32_t)(key & 0x3ffffffu) * 32;
                const int32_t rr = ce0 + r;
                store_sector(A + (int64_t)rr * pitch + c0, m);
                atomicAdd(&wfresh[wib][r], __popc(m));
                *ow = occ_word(s, 0, rr, c0, ob);
            });
        } else {
            __syncwarp();
        }
        if (row) {
            const int32_t size = wfresh[wib][lane];
            // a hyperedge whose size changed since the previous DP pass (or
            // never tested) makes its row block a DP candidate
            if (s.e_dirty_rb && s.e_s[ce] != size) s.e_dirty_rb[ce >> 7] = 1;
            s.e_s[ce] = size;
            const int32_t fe = s.e_f[ce];
            if (s.e_rec) s.e_rec[ce] = make_int4(fe, s.edge_rule ? size : fe - size, e, 0);
            // a count of 0 decides a pair only from a hyperedge with f > |e|
            // (DP) or an empty one (SE)
            if (s.edge_rule ? size == 0 : fe > size) s.has_loose = 1;
        }
        __syncwarp();  // wfresh is reused by the next group
    }
}

// Phase 1 set, two walks over groups of positions:
//  (a) the rows the DP pass saw there (e_prev): zero their sectors of A (the
//      DP pass's clear), and mark the vertices of the hyperedges DP deleted
//      as MD candidates;
//  (b) the hyperedges DP kept in [c0, c0 + 32) (e_c2o after DP): sector c0 / 32 of
//      A^T's vertex rows, deg(v) (= I^V_jj), the maximum demand over E(v),
//      and the occupancy bits of A^T.
__global__ void __launch_bounds__(32 * kSecWarps) k_set_md_tc(InstState *st, const Plan *plan) {
    __shared__ SecTable tab[kSecWarps];
    __shared__ int32_t wdem[kSecWarps][32];  // demands of the group's hyperedges
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    SecTable &t = tab[wib];
    init_table(t, lane);
    const int32_t total = plan->total_rows;
    const int32_t nw = gridDim.x * kSecWarps;
    const bool few = total <= kFewRows;
    const int32_t rows = few ? 8 : 32;
    for (int32_t g0 = (blockIdx.x * kSecWarps + wib) * rows; g0 < total; g0 += nw * rows) {
        const int b = find_owner(plan->row_off, plan->count, g0);
        InstState &s = st[b];
        const int32_t c0 = g0 - plan->row_off[b];
        const int32_t n = s.n;
        if (!s.skip_a) {  // (a)
            const int32_t ce = c0 + lane;
            int32_t p0 = 0, len = 0, mark = 0;
            if (lane < rows && ce < s.m) {
                const int32_t e = __ldg(s.e_prev + ce);
                p0 = __ldg(s.eptr + e);
                len = __ldg(s.eptr + e + 1) - p0;
                mark = s.v_dirty && __ldg(s.e_o2c + e) < 0;
            }
            int32_t start;
            const int32_t tot = rows_prefix(lane, len, &start);
            uint8_t *const A = s.A;
            const int64_t pitch = s.A_pitch;
            uint8_t *const vd = s.v_dirty;
            uint8_t *const vdrb = s.v_dirty_rb;
            walk_live(s, lane, p0, start, tot, mark, [&](int r, int32_t cv, int32_t rmark) {
                if (rmark && cv < n) {
                    vd[cv] = 1;
                    vdrb[cv >> 7] = 1;
                }
                zero_sector(A + (int64_t)(c0 + r) * pitch + (cv & ~31));
            });
        }
    }
    const int32_t parts = few ? 4 : 1;  // of a group's vertices, by position
    for (int32_t u = blockIdx.x * kSecWarps + wib; u < total / 32 * parts; u += nw) {
        const int32_t g0 = u / parts * 32, part = u % parts;
        const int b = find_owner(plan->row_off, plan->count, g0);
        InstState &s = st[b];
        const int32_t c0 = g0 - plan->row_off[b];
        const int32_t n = s.n;
        if (!s.skip_at) {  // (b)
            const int32_t cn = c0 + lane;
            int32_t p0 = 0, len = 0, fe = 0;
            if (cn < s.m_dp) {
                const int32_t e = __ldg(s.e_c2o + cn);
                p0 = __ldg(s.eptr + e);
                len = __ldg(s.eptr + e + 1) - p0;
                fe = __ldg(s.f + e);
            }
            int32_t start;
            const int32_t tot = rows_prefix(lane, len, &start);
            const bool table = tot <= kSecTab;
            wdem[wib][lane] = fe;
            __syncwarp();
            uint8_t *const At = s.At;
            const int64_t pitch = s.At_pitch;
            int32_t *const deg = s.v_deg;
            int32_t *const maxf = s.v_maxf;
            walk_live(s, lane, p0, start, tot, fe, [&](int r, int32_t cv, int32_t rfe) {
                if (cv >= n) { atomicOr(&s.status, kErrCapacity); return; }
                if ((cv & (parts - 1)) != part) return;
                if (table) {
                    if (!sec_set(t, (uint32_t)cv, 1u << r)) atomicOr(&s.status, kErrCapacity);
                } else {
                    if (set_byte(At + (int64_t)cv * pitch, c0 + r)) {
                        atomicAdd(&deg[cv], 1);
                        atomicMax(&maxf[cv], rfe);
                    }
                    set_occupancy(s, 1, cv, c0);
                }
            });
            if (table) {
                drain_table(t, lane, kSecTab, [&](uint32_t cv, uint32_t m, uint32_t **ow, uint32_t *ob) {
                    int32_t mf = 0;  // the largest demand among the sector's hyperedges
                    for (uint32_t bits = m; bits; bits &= bits - 1)
                        mf = max(mf, wdem[wib][__ffs(bits) - 1]);
                    store_sector(At + (int64_t)cv * pitch + c0, m);
                    atomicAdd(&deg[cv], __popc(m));
                    atomicMax(&maxf[cv], mf);
                    *ow = occ_word(s, 1, (int32_t)cv, c0, ob);
                });
            } else {
                __syncwarp();
            }
        }
    }
}

// Phase 1 clear, after the MD contraction: zero the sectors of A^T that the
// set pass wrote (group [c0, c0 + 32): sector c0 / 32 of its vertices' rows).
__global__ void __launch_bounds__(32 * kSecWarps) k_clear_at_tc(InstState *st,
                                                              const Plan *plan) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int32_t total = plan->total_rows;
    const int32_t nw = gridDim.x * kSecWarps;
    for (int32_t g0 = (blockIdx.x * kSecWarps + wib) * 32; g0 < total; g0 += nw * 32) {
        const int b = find_owner(plan->row_off, plan->count, g0);
        InstState &s = st[b];
        const int32_t c0 = g0 - plan->row_off[b];
        if (s.skip_at) continue;
        const int32_t cn = c0 + lane;
        int32_t p0 = 0, len = 0;
        if (cn < s.m_dp) {
            const int32_t e = __ldg(s.e_c2o + cn);
            p0 = __ldg(s.eptr + e);
            len = __ldg(s.eptr + e + 1) - p0;
        }
        int32_t start;
        const int32_t tot = rows_prefix(lane, len, &start);
        uint8_t *const At = s.At;
        const int64_t pitch = s.At_pitch;
        const int32_t n = s.n;
        walk_live(s, lane, p0, start, tot, 0, [&](int, int32_t cv, int32_t) {
            if (cv < n) zero_sector(At + (int64_t)cv * pitch + c0);
        });
    }
}

// ----------------------------------------------------------- compaction --

// Chained scan across the blocks compacting one instance: the exclusive
// prefix, over chunks 0..c-1 of this launch, of the kept counts, given
// chunk c's own count `agg` (decoupled look-back, one thread per block).
// Chunk c first publishes its count, then walks back over its
// predecessors until one has published its inclusive prefix, and
// publishes its own.  Returns -1 if a predecessor published nothing within
// the time limit.  Every predecessor belongs to a block that took its
// ticket earlier, so it is running.
__device__ int32_t chain_exclusive(unsigned long long *status, uint32_t epoch, int32_t c,
                                   int32_t agg) {
    const unsigned long long tag = (unsigned long long)epoch << 34;
    if (c == 0) {
        atomicExch(&status[0], tag | (2ull << 32) | (uint32_t)agg);
        return 0;
    }
    atomicExch(&status[c], tag | (1ull << 32) | (uint32_t)agg);
    int32_t excl = 0;
    uint64_t t0 = 0;
    for (int32_t p = c - 1; p >= 0;) {
        const unsigned long long w = *reinterpret_cast<volatile unsigned long long *>(&status[p]);
        const uint32_t flag = (uint32_t)(w >> 32) & 3u;
        if ((uint32_t)(w >> 34) != epoch || flag == 0) {  // not published in this launch yet
            const uint64_t t = globaltimer();
            if (t0 == 0) t0 = t;
            else if (t - t0 > kChainWaitNs) return -1;
            continue;
        }
        excl += (int32_t)(uint32_t)w;
        if (flag == 2) break;
        --p;
    }
    atomicExch(&status[c], tag | (2ull << 32) | (uint32_t)(excl + agg));
    return excl;
}

// ---------------------------------------------------------- vertex bounds --
//
// tcgen05 path, first round (every hyperedge is a candidate): e_i supersedes
// every e_j that shares one vertex with it and has f_j <= f_i - |e_i| + 1, so
// the largest such bound of each vertex (in v_maxf, free until MD) deletes most
// of what the pass deletes, in two walks over the incidences, before the operand
// is built.  "Supersedes or wins the tie" is transitive, so the rest of the pass
// gives the same result without them.  (|e_j| = 1: f_j < the bound, its own included; equal ones are left to
// the contraction.  Rule SE: only hyperedges of one vertex bound.)  A vertex
// listed twice makes a size too large, which only weakens a bound; one vertex
// alone is told by its smallest and largest position.
// Bounded by the latency of the walks' loads (eight lanes per row).  Power law
// 20,000 x 40,000: 16 of the pass's 27 thousand deletions; the DP passes take
// 483 us with them, 880 without (uniform 16,000 x 32,000: 2.0 and 4.3 ms).
// The first round only: later ones, full again after an FE pass, find the
// largest demands of the last MD pass in v_maxf, not zeros.
__device__ __forceinline__ bool bounds_apply(const InstState &s) {
    return s.active && !s.status && s.rounds == 0 && !s.no_skip;
}

// kTest false: collect the bounds; true: flag the rows they delete.  Rows above
// kBoundRow are left to the contraction: a bound needs f >= |e|, and eight lanes
// walk such a row while the rest waits (one of 3,000 among 20,000 of 10: 1,206 us
// in all; 979 without the bounds).
constexpr int32_t kBoundRow = 64;
template <bool kTest>
__global__ void __launch_bounds__(256) k_bounds(InstState *st, int count) {
    constexpr int kLanes = 8;  // per row
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    if (!bounds_apply(s)) return;
    if (!kTest && blockIdx.x == 0 && threadIdx.x == 0 && s.scan_status) {
        s.scan_ticket = 0;  // for the compaction after the test
        s.scan_epoch = (s.scan_epoch + 1) & kEpochMask;
    }
    const int lane = threadIdx.x & 31, sub = lane % kLanes;
    const int32_t m = s.m, step = gridDim.x * (blockDim.x / kLanes);
    for (int32_t r0 = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x - lane) / kLanes); r0 < m;
         r0 += step) {
        const int32_t r = r0 + lane / kLanes;
        int32_t p0 = 0, p1 = 0, size = 0, lo = 0x7fffffff, hi = -1, bound = 0;
        if (r < m) {
            const int32_t e = s.e_c2o[r];
            p0 = s.eptr[e];
            p1 = s.eptr[e + 1];
            if (p1 - p0 > kBoundRow) p1 = p0;
        }
        for (int32_t p = p0 + sub; p < p1; p += kLanes) {
            const int32_t cv = s.v_o2c[s.evtx[p]];
            if (cv < 0) continue;
            ++size;
            lo = min(lo, cv);
            hi = max(hi, cv);
            if (kTest) bound = max(bound, s.v_maxf[cv]);
        }
        __syncwarp();
#pragma unroll
        for (int o = kLanes / 2; o > 0; o >>= 1) {
            size += __shfl_xor_sync(0xffffffffu, size, o);
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            if (kTest) bound = max(bound, __shfl_xor_sync(0xffffffffu, bound, o));
        }
        if (hi < 0) continue;
        const bool one = lo == hi;
        const int32_t f = s.e_f[r];
        if (kTest) {
            if (sub == 0 && (one ? f < bound : f <= bound)) s.e_del[r] = 1;
            continue;
        }
        bound = one ? f : s.edge_rule ? 0 : f - size + 1;
        if (bound < 1) continue;
        for (int32_t p = p0 + sub; p < p1; p += kLanes) {
            const int32_t cv = s.v_o2c[s.evtx[p]];
            if (cv >= 0 && *reinterpret_cast<volatile int32_t *>(&s.v_maxf[cv]) < bound)
                atomicMax(&s.v_maxf[cv], bound);
        }
    }
}

// Order-preserving compaction of the hyperedges that DP kept (Algorithm 1's
// returned rows), and the zeroed vertex rows of this round's MD pass.  With
// one block per instance (blockIdx.y), chunked so the in-place update of
// e_c2o never overwrites an entry not yet read.  With several blocks (a
// single instance), block t of the ticket order takes chunk t of 1024 rows:
// it writes only after every earlier chunk has published its count, which
// each does after reading its rows, and never beyond its own chunk.
// kPre: the hyperedges that the bounds flagged, before the DP pass proper.
template <bool kPre>
__global__ void k_compact_edges(InstState *st, int count) {
    __shared__ int32_t sh[33];
    __shared__ int32_t sh_x[2];
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    const bool chained = gridDim.x > 1;
    int32_t c = 0;  // this block's chunk (chained)
    if (chained) {
        if (threadIdx.x == 0) sh_x[0] = (int32_t)atomicAdd(&s.scan_ticket, 1u);
        __syncthreads();
        c = sh_x[0];
    }
    if (kPre ? !bounds_apply(s) : !s.active || s.status) return;
    const int32_t m = s.m;
    int32_t kept = 0;  // rows kept before this block's chunk (chained: of chunk c)
    bool last_chunk = false;
    for (int32_t base = chained ? c * 1024 : 0; base < m; base += blockDim.x) {
        int32_t r = base + threadIdx.x;
        int32_t keep = 0, orig = -1, size = 0, f = 0;
        if (r < m) {
            keep = s.e_del[r] == 0;
            orig = s.e_c2o[r];
            size = s.e_s[r];
            if (kPre) f = s.e_f[r];
            else s.e_prev[r] = orig;  // row r of A as this DP pass saw it
        }
        int32_t tot;
        int32_t ex = block_exclusive_scan<int32_t>(keep, &tot, sh);  // syncs after reads
        if (chained) {
            if (threadIdx.x == 0)
                sh_x[1] = chain_exclusive(s.scan_status, s.scan_epoch, c, tot);
            __syncthreads();
            kept = sh_x[1];
            if (kept < 0) {
                if (threadIdx.x == 0) atomicOr(&s.status, kErrTimeout);
                return;
            }
        }
        if (r < m) {
            s.e_o2c[orig] = keep ? kept + ex : -1;
            if (keep) {
                s.e_c2o[kept + ex] = orig;
                s.e_s[kept + ex] = size;  // the size this DP pass saw moves with the row
                if (kPre) {
                    s.e_f[kept + ex] = f;
                    s.e_del[kept + ex] = 0;
                }
            }
        }
        kept += tot;
        if (chained) {
            last_chunk = base + 1024 >= m;
            break;
        }
        __syncthreads();
    }
    if (m == 0 && c == 0) last_chunk = true;
    if (kPre) {
        if (threadIdx.x == 0 && (chained ? last_chunk : true)) {
            s.bounds_deleted = m - kept;
            s.m = kept;  // (a block without a chunk below m has none below `kept` either)
        }
        return;
    }
    if (threadIdx.x == 0 && (chained ? last_chunk : true)) {
        const int32_t before = m + s.bounds_deleted;
        s.bounds_deleted = 0;
        s.m_dp = kept;
        s.dp_deleted = before - kept;
        if (s.rounds < kTraceRounds) {
            s.trace[s.rounds][0] = before;
            s.trace[s.rounds][1] = s.n;
            s.trace[s.rounds][2] = kept;
        }
    }
    // vertex rows of this round's MD pass (s.n is not changed here)
    const int32_t first = chained ? c * 1024 + (int32_t)threadIdx.x : (int32_t)threadIdx.x;
    const int32_t stride = chained ? (int32_t)gridDim.x * 1024 : (int32_t)blockDim.x;
    const int32_t nv = s.n;
    zero_occupancy(s, 1, nv, first, stride);
    for (int32_t r = first; r < nv; r += stride) {
        if (!s.Ab) s.v_deg[r] = 0;  // (bit-packed: counted before the DP pass)
        s.v_maxf[r] = 0;
        s.v_cnt[r] = 0;
        s.v_del[r] = 0;
    }
}

// MD decision (Algorithm 2: delete v_j iff C_j >= max f over E(v_j)),
// order-preserving compaction of the vertices, and round bookkeeping.  One
// block per instance, or (a single instance) one block per chunk of 1024
// vertices as in k_compact_edges; then the block of the last chunk keeps
// the books, and each block clears the next round's rows in its own range.
__global__ void k_compact_vertices(InstState *st, int count, BatchCounters *ctr,
                                   int32_t *done_list) {
    __shared__ int32_t sh[33];
    __shared__ int32_t sh_x[2];
    const int b = blockIdx.y;
    if (b >= count) return;
    InstState &s = st[b];
    const bool chained = gridDim.x > 1;
    int32_t c = 0;
    if (chained) {
        if (threadIdx.x == 0) sh_x[0] = (int32_t)atomicAdd(&s.scan_ticket, 1u);
        __syncthreads();
        c = sh_x[0];
    }
    // The state is read before any block can finish the books: the block
    // of chunk 0 reads it before publishing, and the last chunk waits for
    // that.  A block without a chunk does only the clears of its range.
    const bool run = s.active && s.status == 0;
    const int32_t n = s.n, m_dp = s.m_dp;
    bool books = !chained;  // this block keeps the books
    if (run) {
        int32_t kept = 0;
        // (chained: chunk 0 runs even when n = 0, so that some block keeps the books)
        for (int32_t base = chained ? c * 1024 : 0; base < n || (chained && base == 0);
             base += blockDim.x) {
            int32_t r = base + threadIdx.x;
            int32_t keep = 0, orig = -1;
            if (r < n) {
                // a vertex that lost no hyperedge since it last survived MD
                // survives again: its dominator count can only have dropped
                const bool cand = s.md_full || !s.v_dirty || s.v_dirty[r];
                keep = !cand || s.v_cnt[r] < s.v_maxf[r];
                orig = s.v_c2o[r];
                s.v_del[r] = !keep;
            }
            int32_t tot;
            int32_t ex = block_exclusive_scan<int32_t>(keep, &tot, sh);
            if (chained) {
                if (threadIdx.x == 0)
                    sh_x[1] = chain_exclusive(s.scan_status, s.scan_epoch, c, tot);
                __syncthreads();
                kept = sh_x[1];
                if (kept < 0) {
                    if (threadIdx.x == 0) atomicOr(&s.status, kErrTimeout);
                    return;
                }
            }
            if (r < n) {
                s.v_o2c[orig] = keep ? kept + ex : -1;
                if (keep) s.v_c2o[kept + ex] = orig;
            }
            kept += tot;
            if (chained) {
                books = base + 1024 >= n;
                break;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0 && books) {
            s.n_next = kept;
            s.md_deleted = n - kept;
            s.changed = (s.dp_deleted + s.md_deleted) > 0;
            s.m = m_dp;
            s.n = kept;
            s.rounds += 1;
            s.md_full = 0;
            if (!s.changed && s.full_edges && s.max_rounds == 0) {
                // fixpoint: rule FE decides (fe.cu) whether it goes on; no
                // vertex was deleted, so v_del is already all zero
                s.fe_stage = 1;
            } else if (!s.changed || (s.max_rounds > 0 && s.rounds >= s.max_rounds)) {
                s.active = 0;
                if (done_list && ctr) done_list[atomicAdd(&ctr->n_done, 1)] = b;
            }
        }
        // the next round's rows: MD candidates start empty; hyperedge rows
        // of the DP pass (e_s keeps the sizes).  One block skips them once
        // the instance has finished; several blocks cannot know that and
        // clear them anyway, which is harmless.
        bool next_rows = true;
        int32_t nv = n;  // vertex rows to clear
        if (!chained) {
            __syncthreads();  // the books are kept
            next_rows = s.active != 0;
            nv = s.n;
        }
        if (next_rows) {  // (32 bits suffice: blocks x 1024 < max(n0, m0) + 1024)
            const int32_t first = chained ? c * 1024 + (int32_t)threadIdx.x : (int32_t)threadIdx.x;
            const int32_t stride = chained ? (int32_t)gridDim.x * 1024 : (int32_t)blockDim.x;
            if (s.v_dirty) {
                for (int32_t r = first; r < nv; r += stride) s.v_dirty[r] = 0;
                for (int32_t w = first; w < (nv + 127) / 128; w += stride) s.v_dirty_rb[w] = 0;
            }
            if (s.Ab)
                for (int32_t r = first; r < nv; r += stride) s.v_deg[r] = 0;
            for (int32_t r = first; r < m_dp; r += stride) {
                s.e_f[r] = s.f[s.e_c2o[r]];
                s.e_del[r] = 0;
            }
            if (s.e_dirty_rb)
                for (int32_t w = first; w < (m_dp + 127) / 128; w += stride) s.e_dirty_rb[w] = 0;
            zero_occupancy(s, 0, m_dp, first, stride);
            if (first == 0) s.has_loose = 0;
        }
    } else {
        books = !chained || c == 0;  // nothing changes: one block reports it
    }
    if (threadIdx.x == 0 && ctr && books) {  // read by a later kernel
        atomicAdd(&ctr->active, s.active);
        atomicAdd(&ctr->n_alive, s.n);
        atomicAdd(&ctr->m_alive, s.m);
        atomicAdd(&ctr->dp_deleted, s.dp_deleted);
        atomicAdd(&ctr->md_deleted, s.md_deleted);
        atomicMax(&ctr->max_rounds_seen, s.rounds);
        atomicOr(&ctr->changed_any, s.changed);
        atomicOr(&ctr->status_any, s.status);
    }
}

// ---------------------------------------------------- bit-packed passes --
//
// Both passes take the rows' intersections from bitmaps of the OTHER side,
// 32 pairs per instruction, instead of counting each pair's bits:
//  * DP, superseder e_i: for every v in e_i the bitmap of v's hyperedges says
//    which e_j do not miss it, so a few bitwise operations per word keep, for
//    32 columns j at once, whether more than t vertices of e_i are missed
//    (t = 0..3; demands above 4 count the misses in bit planes).
//  * MD, candidate v_j: the vertices in all of its hyperedges are the AND of
//    those hyperedges' bitmaps.
// A warp stops as soon as no column of its block is left, after some three
// vertices of a hyperedge or two hyperedges of a vertex.  "Supersedes or wins
// the tie" is transitive, so a hyperedge already flagged is no superseder, and
// columns that go are flagged by a lane per word or, where a word has many, a
// lane per column (a lane per word and no skipping took 1.46 ms where 4,096
// hyperedges are equal; 0.32 now, 0.36 with the tiles).  Bounded by the
// latency of chains of three loads (a row's bitmap, its members' bitmaps, what
// is known of the pairs found); the AND + POPC of all pairs, 64 x 64 to a
// tile, was bounded by POPC (16 a clock and SM).  On one GB300, uniform 4,000 x
// 8,000, |e| 2..16: both passes of two rounds 53 us, load to result 317 us,
// 1,704 with the tiles; power law 20,000 x 40,000: the rounds 2.5 ms, 138 with
// the tiles; 2,000 x 3,000, |e| 200..400, demands up to 200: 0.98 ms, 1.93 with
// the tiles.

constexpr int kPopWarps = 8;
// Blocks per SM.  (4 for DP spill 64 bytes a thread; 3 take 524 us instead of
// 447 for the DP passes of uniform 16,000 x 32,000.)
constexpr int kPopDpBlocks = 4, kPopMdBlocks = 4;
constexpr int kPopIds = 512;    // members of a row gathered at a time
constexpr int kPopT = 4;        // demands up to this: misses counted in unary
constexpr int kPopFew = 4;      // columns of a word flagged by one lane
constexpr int kPopPlanes = 24;  // above: in binary (sizes are < 2^24)

// Members of a row of W words, from word *k0 on, into ids: as many as fit.
// The whole warp.
__device__ __forceinline__ int32_t pop_ids(const uint32_t *row, int32_t W, int32_t *k0,
                                           int32_t *ids, int lane) {
    int32_t n = 0;
    __syncwarp();  // ids is free
    while (*k0 < W) {
        const int32_t k = *k0 + 4 * lane;  // (the pitch is a multiple of 4 words, zero behind W)
        uint4 x = make_uint4(0, 0, 0, 0);
        if (k < W) x = *reinterpret_cast<const uint4 *>(row + k);
        int32_t c = __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
        int32_t step = 128;
        if (n + __reduce_add_sync(0xffffffffu, c) > kPopIds) {
            if (n > 0) break;
            step = kPopIds / 32;  // a dense row: what always fits
            if (4 * lane >= step) {
                x = make_uint4(0, 0, 0, 0);
                c = 0;
            }
        }
        int32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        int32_t at = n + inc - c;
        n += __shfl_sync(0xffffffffu, inc, 31);
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
            for (uint32_t b = w[u]; b; b &= b - 1) ids[at++] = (k + u) * 32 + __ffs(b) - 1;
        *k0 += step;
    }
    __syncwarp();
    return n;
}

// Four words of a lane.
struct Quad {
    uint32_t w[4];
    __device__ __forceinline__ bool any() const { return (w[0] | w[1] | w[2] | w[3]) != 0; }
};
__device__ __forceinline__ Quad quad_fill(uint32_t x) { return {{x, x, x, x}}; }
__device__ __forceinline__ Quad quad_load(const uint32_t *p) {
    const uint4 x = *reinterpret_cast<const uint4 *>(p);
    return {{x.x, x.y, x.z, x.w}};
}
// Bits of rows < R other than `self`, from row r0 on.
__device__ __forceinline__ Quad quad_rows(int32_t r0, int32_t R, int32_t self) {
    Quad q;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int32_t left = R - (r0 + 32 * u), at = self - (r0 + 32 * u);
        q.w[u] = left >= 32 ? ~0u : left > 0 ? (1u << left) - 1u : 0u;
        if (at >= 0 && at < 32) q.w[u] &= ~(1u << at);
    }
    return q;
}

struct PopRow {  // a superseder
    int32_t i, f, size, id;
};

// Is hyperedge i flagged?  One answer for the warp, while others may flag it.
__device__ __forceinline__ bool pop_gone(const InstState &s, int32_t i) {
    return __any_sync(0xffffffffu, __ldcg(s.e_del + i) != 0);
}

// e_j goes unless the two are equal and e_j's index is the lower one.
__device__ __forceinline__ void pop_delete(const InstState &s, const PopRow &r, int32_t j,
                                           bool missed) {
    if (missed || s.e_f[j] != r.f || s.e_s[j] != r.size || r.id < s.e_c2o[j]) s.e_del[j] = 1;
}

// Demands above kPopT: the misses of 32 columns a lane, in binary, seven
// vertices to an addition (four full adders, then one ripple), until every
// column has missed too many (looked at after every 28 vertices).
__device__ __noinline__ void pop_dp_planes(const InstState &s, PopRow r, int32_t jb, int32_t *ids,
                                           int lane) {
    const int32_t W = (s.n + 31) / 32, K = (s.m + 31) / 32;
    const int np = max(3, 32 - __clz(r.size));
    const int32_t t = s.edge_rule ? 0 : min(r.f - 1, r.size);
    for (int32_t k0 = jb * 128; k0 < min(K, jb * 128 + 128); k0 += 32) {
        const int32_t k = k0 + lane, left = s.m - k * 32;
        uint32_t may = left >= 32 ? ~0u : left > 0 ? (1u << left) - 1u : 0u;
        if (r.i >> 5 == k) may &= ~(1u << (r.i & 31));
        uint32_t cnt[kPopPlanes];
#pragma unroll
        for (int p = 0; p < kPopPlanes; ++p) cnt[p] = 0;
        auto at_most_t = [&] {
            uint32_t less = 0, same = ~0u;  // misses below, equal to t
#pragma unroll
            for (int p = kPopPlanes - 1; p >= 0; --p) {
                if (p >= np) continue;
                if (t >> p & 1) {
                    less |= same & ~cnt[p];
                    same &= cnt[p];
                } else {
                    same &= ~cnt[p];
                }
            }
            return less | same;
        };
        bool any = true;
        for (int32_t at = 0, group = 0; at < W && any;) {
            const int32_t n = pop_ids(s.Ab + (int64_t)r.i * s.Ab_pitch, W, &at, ids, lane);
#pragma unroll 1
            for (int32_t q = 0; q < n && any; q += 7, ++group) {
                uint32_t x[7];
#pragma unroll
                for (int u = 0; u < 7; ++u)
                    x[u] = q + u < n && k < K ? ~s.Atb[(int64_t)ids[q + u] * s.Atb_pitch + k] : 0;
                auto add = [](uint32_t a, uint32_t b, uint32_t c, uint32_t *carry) {
                    *carry = (a & b) | (c & (a | b));
                    return a ^ b ^ c;
                };
                uint32_t c0, c1, c2, four, two, carry;
                const uint32_t s0 = add(x[0], x[1], x[2], &c0), s1 = add(x[3], x[4], x[5], &c1);
                const uint32_t one = add(s0, s1, x[6], &c2);
                two = add(c0, c1, c2, &four);
                cnt[0] = add(cnt[0], one, 0, &carry);
                cnt[1] = add(cnt[1], two, carry, &carry);
                cnt[2] = add(cnt[2], four, carry, &carry);
#pragma unroll
                for (int p = 3; p < kPopPlanes; ++p)
                    if (p < np) cnt[p] = add(cnt[p], 0, carry, &carry);
                if ((group & 3) == 3) {
                    may &= at_most_t();
                    any = __any_sync(0xffffffffu, may != 0);
                }
            }
        }
        may &= at_most_t();
        if (!__any_sync(0xffffffffu, may != 0)) continue;
        if (pop_gone(s, r.i)) return;
        for (; may; may &= may - 1) {
            const int b = __ffs(may) - 1;
            const int32_t j = k * 32 + b;
            int32_t miss = 0;
#pragma unroll
            for (int p = 0; p < kPopPlanes; ++p)
                if (p < np) miss |= (int32_t)(cnt[p] >> b & 1u) << p;
            if (s.e_f[j] <= r.f - miss) pop_delete(s, r, j, miss > 0);
        }
    }
}

// Algorithm 1, D_ij = [f_i - |e_i \ e_j| >= f_j]; delete j iff D_ij and (not
// D_ji or i < j), i < j comparing input indices (D_ij and D_ji: equal sets
// and demands).  Rule SE instead: D_ij = [e_i within e_j and f_i >= f_j].
// A block takes kPopDpRows superseders against 4,096 columns.  Incremental
// rounds: only row blocks with a hyperedge that lost a vertex.  With
// nshards > 1 only rows of 128-row blocks b with b % nshards == shard.
__global__ void __launch_bounds__(32 * kPopWarps, kPopDpBlocks)
    k_pop_dp(InstState *st, const Plan *plan, int shard, int nshards) {
    __shared__ int32_t ids_all[kPopWarps][kPopIds];
    __shared__ __align__(16) uint32_t fle[kPopT][128];  // [d - 1]: columns of demand <= d
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *ids = ids_all[warp];
    const int64_t total = plan->total_tiles;
    for (int64_t unit = blockIdx.x; unit < total; unit += gridDim.x) {
        const int b = find_owner(plan->tile_off, plan->count, unit);
        const InstState &s = st[b];
        const int32_t m = s.m, blocks = (m + 4095) / 4096;
        const int64_t local = unit - plan->tile_off[b];
        const int32_t i0 = (int32_t)(local / blocks) * kPopDpRows, jb = (int32_t)(local % blocks);
        if (nshards > 1 && (i0 / kTcM) % nshards != shard) continue;
        if (s.e_dirty_rb && !s.e_dirty_rb[i0 >> 7]) continue;
        __syncthreads();  // fle is free
#pragma unroll 4
        for (int w = warp; w < 128; w += kPopWarps) {
            const int32_t j = jb * 4096 + 32 * w + lane;
            const int32_t f = j < m ? s.e_f[j] : 0x7fffffff;
#pragma unroll
            for (int d = 0; d < kPopT; ++d) {
                const uint32_t bits = __ballot_sync(0xffffffffu, f <= d + 1);
                if (lane == d) fle[d][w] = bits;
            }
        }
        __syncthreads();
        const int32_t W = (s.n + 31) / 32, K = (m + 31) / 32, k = jb * 128 + 4 * lane;
        const uint32_t *const col = s.Atb + k;  // this lane's words of a vertex's bitmap
        bool large = false;  // the warp has a demand above kPopT
        for (int32_t i = i0 + warp; i < min(i0 + kPopDpRows, m); i += kPopWarps) {
            const PopRow r = {i, s.e_f[i], s.e_s[i], s.e_c2o[i]};
            if (r.f > kPopT) {
                large = true;
                continue;
            }
            const int t = s.edge_rule ? 0 : r.f - 1;
            const Quad valid = quad_rows(k * 32, m, i);
            Quad miss[kPopT], left = valid;  // [t]: columns that miss more than t; at most t
#pragma unroll
            for (int d = 0; d < kPopT; ++d) miss[d] = quad_fill(0);
            bool any = true;
            for (int32_t at = 0; at < W && any;) {
                const int32_t n = pop_ids(s.Ab + (int64_t)i * s.Ab_pitch, W, &at, ids, lane);
                for (int32_t q = 0; q < n && any; q += 4) {
                    Quad x[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        x[u] = quad_fill(~0u);
                        if (q + u < n && k < K)
                            x[u] = quad_load(col + (int64_t)ids[q + u] * s.Atb_pitch);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
#pragma unroll
                            for (int d = kPopT - 1; d > 0; --d)
                                miss[d].w[c] |= miss[d - 1].w[c] & ~x[u].w[c];
                            miss[0].w[c] |= ~x[u].w[c];
                        }
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        left.w[c] = valid.w[c] & ~(t == 0   ? miss[0].w[c]
                                                   : t == 1 ? miss[1].w[c]
                                                   : t == 2 ? miss[2].w[c]
                                                            : miss[3].w[c]);
                    any = __any_sync(0xffffffffu, left.any());
                }
            }
            if (!__any_sync(0xffffffffu, left.any())) continue;
            if (pop_gone(s, i)) continue;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t go = 0;
#pragma unroll
                for (int d = 0; d < kPopT; ++d)
                    if (d <= t && r.f - d >= 1) go |= ~miss[d].w[c] & fle[r.f - d - 1][4 * lane + c];
                go &= valid.w[c];
                if (__reduce_max_sync(0xffffffffu, __popc(go)) <= kPopFew) {
                    for (; go; go &= go - 1) {
                        const int bit = __ffs(go) - 1;
                        pop_delete(s, r, (k + c) * 32 + bit, miss[0].w[c] >> bit & 1u);
                    }
                    continue;
                }
                for (unsigned on = __ballot_sync(0xffffffffu, go != 0); on; on &= on - 1) {
                    const int l = __ffs(on) - 1;
                    const uint32_t word = __shfl_sync(0xffffffffu, go, l);
                    const uint32_t missed = __shfl_sync(0xffffffffu, miss[0].w[c], l);
                    const int32_t j = (jb * 128 + 4 * l + c) * 32 + lane;
                    if (word >> lane & 1u) pop_delete(s, r, j, missed >> lane & 1u);
                }
            }
        }
        if (!large) continue;
        for (int32_t i = i0 + warp; i < min(i0 + kPopDpRows, m); i += kPopWarps)
            if (s.e_f[i] > kPopT) pop_dp_planes(s, {i, s.e_f[i], s.e_s[i], s.e_c2o[i]}, jb, ids, lane);
    }
}

// Algorithm 2, D_ij = [x = d_j and (x != d_i or i < j)], i < j comparing
// input indices: C_j counts the other vertices of all of v_j's hyperedges,
// without those of equal incidence and a higher index.  A warp per vertex;
// incremental rounds: only vertices that lost a hyperedge.  (A vertex of no
// hyperedge goes whatever its count.)  Shares as in k_pop_dp.  A hyperedge's
// bitmap takes as many lanes as it has quads of words (a power of two), and the
// warp 4 x 32 / lanes hyperedges at a time: few vertices of high degree have
// only their own warps.  (n 66, m 100,000, two vertices in all hyperedges: the
// pass 6.4 ms with the whole warp on 4 hyperedges, 1.2 now; as tiles of bit
// counts 0.7, with a DP pass of 39 instead of 4.6.)
__global__ void __launch_bounds__(32 * kPopWarps, kPopMdBlocks)
    k_pop_md(InstState *st, const Plan *plan, int shard, int nshards) {
    __shared__ int32_t ids_all[kPopWarps][kPopIds];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *ids = ids_all[warp];
    const int64_t total = plan->total_tiles;
    for (int64_t unit = blockIdx.x; unit < total; unit += gridDim.x) {
        const int b = find_owner(plan->tile_off, plan->count, unit);
        InstState &s = st[b];
        const int32_t n = s.n;
        const int32_t j0 = (int32_t)(unit - plan->tile_off[b]) * kPopMdRows;
        if (nshards > 1 && (j0 / kTcM) % nshards != shard) continue;
        const int32_t W = (s.m + 31) / 32, K = (n + 31) / 32;
        for (int32_t j = j0 + warp; j < min(j0 + kPopMdRows, n); j += kPopWarps) {
            if (s.v_dirty && !s.md_full && !s.v_dirty[j]) continue;
            const int32_t dj = s.v_deg[j], oj = s.v_c2o[j];
            if (dj == 0) continue;
            int32_t count = 0;
            for (int32_t k0 = 0; k0 < K; k0 += 128) {
                const int quads = min((K - k0 + 3) / 4, 32);
                const int lanes = quads > 1 ? 1 << (32 - __clz(quads - 1)) : 1, sets = 32 / lanes;
                const int32_t k = k0 + 4 * (lane & (lanes - 1)), set = lane / lanes;
                Quad in = quad_rows(k * 32, n, j);
                bool any = true;
                for (int32_t at = 0; at < W && any;) {
                    const int32_t cnt = pop_ids(s.Atb + (int64_t)j * s.Atb_pitch, W, &at, ids, lane);
                    for (int32_t q = 0; q < cnt && any; q += 4 * sets) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int32_t id = q + u * sets + set;
                            if (id >= cnt || k >= K) continue;
                            const Quad x = quad_load(s.Ab + (int64_t)ids[id] * s.Ab_pitch + k);
#pragma unroll
                            for (int c = 0; c < 4; ++c) in.w[c] &= x.w[c];
                        }
                        __syncwarp();
                        for (int o = lanes; o < 32; o <<= 1)
#pragma unroll
                            for (int c = 0; c < 4; ++c) in.w[c] &= __shfl_xor_sync(0xffffffffu, in.w[c], o);
                        any = __any_sync(0xffffffffu, in.any());
                    }
                }
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    for (unsigned on = __ballot_sync(0xffffffffu, in.w[c] != 0 && set == 0); on; on &= on - 1) {
                        const int l = __ffs(on) - 1;
                        const uint32_t word = __shfl_sync(0xffffffffu, in.w[c], l);
                        const int32_t i = (k0 + 4 * l + c) * 32 + lane;
                        if (word >> lane & 1u) count += s.v_deg[i] != dj || s.v_c2o[i] < oj;
                    }
            }
            count = __reduce_add_sync(0xffffffffu, count);
            if (lane == 0) s.v_cnt[j] = count;
        }
    }
}

// --------------------------------------------------------------- results --

// Alive masks over the input ids; blockIdx.y = instance.  With `batch`
// set, instance b writes at its offsets v_base / e_base of the
// concatenated masks; otherwise at 0.
__global__ void k_alive_masks(const InstState *st, int count, bool batch, uint8_t *alive_v,
                              uint8_t *alive_e) {
    const int b = blockIdx.y;
    if (b >= count) return;
    const InstState &s = st[b];
    if (batch) {
        alive_v += s.v_base;
        alive_e += s.e_base;
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)s.n0 + s.m0;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (i < s.n0) alive_v[i] = s.v_o2c[i] >= 0;
        else alive_e[i - s.n0] = s.e_o2c[i - s.n0] >= 0;
    }
}

// ---- serving loop (device-resident; see server.cpp) ----

// One block per slot at a time.  The ready flag is read once per slot (by
// thread 0): the host may set it while this kernel runs.
__global__ void k_server_admit(InstState *live, const InstState *staged, volatile int32_t *ready,
                               int count) {
    __shared__ int32_t go;
    constexpr int kWords = (int)(sizeof(InstState) / 4);
    static_assert(sizeof(InstState) % 4 == 0, "state copied in words");
    for (int si = blockIdx.x; si < count; si += gridDim.x) {
        if (threadIdx.x == 0) go = ready[si];
        __syncthreads();
        if (go) {
            const int32_t *src = reinterpret_cast<const int32_t *>(staged + si);
            int32_t *dst = reinterpret_cast<int32_t *>(live + si);
            for (int w = threadIdx.x; w < kWords; w += blockDim.x) dst[w] = src[w];
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                ready[si] = 0;
                __threadfence_system();
            }
        }
        __syncthreads();
    }
}

// One block.  A slot is retired once: a finished instance is inactive (and
// its live slot zeroed here), a failed one is taken while still active.
__global__ void __launch_bounds__(256) k_server_retire(InstState *live, InstState *out,
                                                       const int32_t *done,
                                                       const BatchCounters *ctr,
                                                       volatile int32_t *ring,
                                                       volatile ServerFlags *flags,
                                                       ServerDev *dev, int count) {
    __shared__ int32_t fin[4096];  // max_slots <= 4096
    __shared__ int32_t nfin;
    constexpr int kWords = (int)(sizeof(InstState) / 4);
    if (threadIdx.x == 0) nfin = 0;
    __syncthreads();
    const int nd = min(ctr->n_done, count);
    for (int i = threadIdx.x; i < nd; i += blockDim.x) {
        const int si = done[i];
        if (si >= 0 && si < count) fin[atomicAdd(&nfin, 1) & 4095] = si;
    }
    for (int si = threadIdx.x; si < count; si += blockDim.x)
        if (live[si].active && live[si].status) fin[atomicAdd(&nfin, 1) & 4095] = si;
    __syncthreads();
    const int nf = min(nfin, count);  // each slot at most once
    for (int i = 0; i < nf; ++i) {
        const int si = fin[i];
        int32_t *src = reinterpret_cast<int32_t *>(live + si);
        int32_t *dst = reinterpret_cast<int32_t *>(out + si);
        for (int w = threadIdx.x; w < kWords; w += blockDim.x) dst[w] = src[w];
        __syncthreads();
        for (int w = threadIdx.x; w < kWords; w += blockDim.x) src[w] = 0;
        __syncthreads();
    }
    if (threadIdx.x == 0 && nf > 0) {
        __threadfence_system();  // the states in `out` before the ring entries
        const uint32_t head = dev->head;
        for (int i = 0; i < nf; ++i) ring[(head + (uint32_t)i) % (uint32_t)count] = fin[i];
        __threadfence_system();  // the entries before the head
        dev->head = head + (uint32_t)nf;
        flags->head = head + (uint32_t)nf;
        __threadfence_system();
    }
}

__global__ void k_server_cond(cudaGraphConditionalHandle h, const BatchCounters *ctr,
                              const int32_t *kerr, const Plan *plan, ServerDev *dev,
                              volatile ServerFlags *flags, volatile const int32_t *ready,
                              int count, int32_t cap) {
    __shared__ int32_t pending;
    if (threadIdx.x == 0) pending = 0;
    __syncthreads();
    for (int si = threadIdx.x; si < count; si += blockDim.x)
        if (ready[si]) pending = 1;
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (plan->any_active) dev->rounds += 1;
    const int32_t it = ++dev->iters;
    const int32_t err = *kerr;
    flags->rounds = dev->rounds;
    flags->kerr = err;
    __threadfence_system();
    const bool go = !flags->stop && err == 0 && it < cap && (ctr->active > 0 || pending);
    cudaGraphSetConditional(h, go ? 1u : 0u);
}

__global__ void k_loop_cond(cudaGraphConditionalHandle h, BatchCounters *ctr, int32_t *kerr,
                            int32_t round_cap) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int32_t it = ++ctr->loop_iters;
    bool go = ctr->active > 0 && *kerr == 0 && ctr->status_any == 0;
    if (go && it >= round_cap) {
        atomicOr(kerr, kErrRoundCap);
        go = false;
    }
    cudaGraphSetConditional(h, go ? 1u : 0u);
}

}  // namespace

// ------------------------------------------------------- host launchers --

cudaError_t launch_loop_cond(cudaGraphConditionalHandle h, BatchCounters *ctr, int32_t *kerr,
                             int32_t round_cap, cudaStream_t s) {
    k_loop_cond<<<1, 32, 0, s>>>(h, ctr, kerr, round_cap);
    return cudaGetLastError();
}

cudaError_t launch_server_admit(InstState *live, const InstState *staged, int32_t *ready,
                                int count, cudaStream_t s) {
    k_server_admit<<<count < 152 ? count : 152, 128, 0, s>>>(live, staged, ready, count);
    return cudaGetLastError();
}

cudaError_t launch_server_retire(InstState *live, InstState *out, const int32_t *done,
                                 const BatchCounters *ctr, int32_t *ring, ServerFlags *flags,
                                 ServerDev *dev, int count, cudaStream_t s) {
    if (count > 4096) return cudaErrorInvalidValue;  // one block lists the retirements
    k_server_retire<<<1, 256, 0, s>>>(live, out, done, ctr, ring, flags, dev, count);
    return cudaGetLastError();
}

cudaError_t launch_server_cond(cudaGraphConditionalHandle h, const BatchCounters *ctr,
                               const int32_t *kerr, const Plan *plan, ServerDev *dev,
                               ServerFlags *flags, const int32_t *ready, int count, int32_t cap,
                               cudaStream_t s) {
    k_server_cond<<<1, 256, 0, s>>>(h, ctr, kerr, plan, dev, flags, ready, count, cap);
    return cudaGetLastError();
}

static int grid_for(int sms, int per_sm) { return sms * per_sm; }

// Blocks per instance for a grid-stride kernel over `items` per instance:
// enough for the largest instance, but for a batch no more than about 16
// blocks per SM in all (a block that finds no work still costs a launch).
static int per_instance_grid(int64_t items, int count) {
    int64_t g = (items + 255) / 256;
    const int64_t cap = count > 1 ? (152 * 16 + count - 1) / count : 256;
    if (g > cap) g = cap;
    if (g > 256) g = 256;
    return g < 1 ? 1 : (int)g;
}

cudaError_t launch_validate(InstState *st, int count, cudaStream_t s) {
    k_validate<<<dim3(count > 1 ? per_instance_grid(1 << 20, count) : 256, count), 256, 0, s>>>(
        st, count);
    return cudaGetLastError();
}

cudaError_t launch_status_or(const InstState *st, int count, int32_t *out, cudaStream_t s) {
    k_status_or<<<(count + 255) / 256 < 64 ? (count + 255) / 256 : 64, 256, 0, s>>>(st, count, out);
    return cudaGetLastError();
}

cudaError_t launch_localize_ptr(InstState *st, int count, const int64_t *gptr, const int64_t *e0,
                                cudaStream_t s) {
    k_localize_ptr<<<dim3(16, count), 256, 0, s>>>(st, count, gptr, e0);
    return cudaGetLastError();
}

cudaError_t launch_gather_bounds(const int64_t *gptr, const int64_t *e0, int64_t *out, int count,
                                 cudaStream_t s) {
    k_gather_bounds<<<(count + 256) / 256, 256, 0, s>>>(gptr, e0, out, count);
    return cudaGetLastError();
}

cudaError_t launch_build(InstState *st, int count, int32_t max_rounds, int64_t max_nnz,
                         int64_t max_m, int64_t max_n, cudaStream_t s, int layout) {
    const int gx = per_instance_grid(max_m, count);
    const int gz = per_instance_grid(max_nnz, count);
    const int gr = per_instance_grid(max_m * kRankLanes, count);
    // a single instance splits its initial ranges over blocks
    const int gi = count > 1 ? 1 : (int)std::min<int64_t>((std::max(max_m, max_n) + 4095) / 4096, 152);
    k_init<<<dim3(gi > 0 ? gi : 1, count), 1024, 0, s>>>(st, count, max_rounds);
    if (layout == 2) {
        k_vertex_degrees<<<dim3(gz, count), 256, 0, s>>>(st, count);
        k_vertex_layout<<<count, 1024, 0, s>>>(st, count);
    }
    if (layout) {
        k_layout_keys<<<dim3(gx, count), 256, 0, s>>>(st, count);
        k_layout_scan<<<count, 1024, 0, s>>>(st, count);
        k_layout_place<<<dim3(gx, count), 256, 0, s>>>(st, count);
        k_layout_rank<<<dim3(gr, count), 256, 0, s>>>(st, count);
        k_layout_commit<<<dim3(gx, count), 256, 0, s>>>(st, count);
    }
    k_edge_rows<<<dim3(gx, count), 256, 0, s>>>(st, count);
    return cudaGetLastError();
}

// Set (or, phase 1, clear) pass of the operands: dense FP8 (tcgen05 path,
// sector writes) or bit-packed (popcount path).
template <int kPhase>
static void launch_scatter(InstState *st, const Plan *plan, bool set, bool dense, int sms,
                           cudaStream_t s) {
    if (dense) {  // blocks of 4 warps (17 KB of tables each): per SM 8 for the A set
                  // pass (its row-local sector writes lose with more), 12 for the MD
                  // set pass, 16 for the clear (measured)
        if (kPhase == 0) k_set_a_tc<<<grid_for(sms, 8), 32 * kSecWarps, 0, s>>>(st, plan);
        else if (set) k_set_md_tc<<<grid_for(sms, 12), 32 * kSecWarps, 0, s>>>(st, plan);
        else k_clear_at_tc<<<grid_for(sms, 16), 32 * kSecWarps, 0, s>>>(st, plan);
        return;
    }
    const int grid = grid_for(sms, 8);
    if (set) k_scatter<kPhase, true><<<grid, 256, 0, s>>>(st, plan);
    else k_scatter<kPhase, false><<<grid, 256, 0, s>>>(st, plan);
}

static void launch_pop(InstState *st, const Plan *plan, int phase, int shard, int nshards,
                       int sms, cudaStream_t s) {
    const int threads = 32 * kPopWarps;
    if (phase == 0) k_pop_dp<<<grid_for(sms, kPopDpBlocks), threads, 0, s>>>(st, plan, shard, nshards);
    else k_pop_md<<<grid_for(sms, kPopMdBlocks), threads, 0, s>>>(st, plan, shard, nshards);
}

cudaError_t launch_phase_prologue(InstState *st, Plan *plan, BatchCounters *ctr, int phase,
                                  int contraction, int sms, cudaStream_t s) {
    const bool tc = contraction == kFp8;
    k_plan<<<1, 1024, 0, s>>>(st, plan, phase, tc ? 1 : 0, ctr);
    if (phase == 0) launch_scatter<0>(st, plan, true, tc, sms, s);
    else launch_scatter<1>(st, plan, true, tc, sms, s);
    return cudaGetLastError();
}

cudaError_t launch_phase_contract(InstState *st, Plan *plan, BatchCounters *ctr, int phase,
                                  int contraction, int sms, int32_t *kerr, cudaStream_t s,
                                  int tile_n, int shard, int nshards) {
    const bool tc = contraction == kFp8;
    if (tc) {
        // each share builds its own list and hands it out from its start
        cudaError_t e = cudaMemsetAsync(&plan->list_count, 0, sizeof(int32_t), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(&plan->list_next, 0, sizeof(int32_t), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(&plan->list_light, 0, 2 * sizeof(int32_t), s);
        if (e == cudaSuccess) e = launch_tc_tile_list(st, plan, phase, sms, s, shard, nshards);
        if (e != cudaSuccess) return e;
        return launch_tc_contract(st, plan, ctr, phase, sms, tile_n, kerr, s);
    }
    launch_pop(st, plan, phase, shard, nshards, sms, s);
    return cudaGetLastError();
}

cudaError_t launch_phase_epilogue(InstState *st, Plan *plan, BatchCounters *ctr, int count,
                                  int phase, int contraction, int sms, cudaStream_t s,
                                  int32_t *done_list, int compact_blocks) {
    const bool tc = contraction == kFp8;
    // (the DP pass's clear of A runs inside the MD set pass, which walks the
    // same incidences)
    if (phase == 1) launch_scatter<1>(st, plan, false, tc, sms, s);
    // compact_blocks > 1: a single instance, one block per chunk of 1024 ids
    const dim3 cgrid(compact_blocks > 1 ? compact_blocks : 1, count);
    if (phase == 0) k_compact_edges<false><<<cgrid, 1024, 0, s>>>(st, count);
    else k_compact_vertices<<<cgrid, 1024, 0, s>>>(st, count, ctr, done_list);
    return cudaGetLastError();
}

// A sharded pass's partial output over INPUT ids (the replicas' layouts may
// order rows differently): phase 0 the DP/SE deletion flag of every
// hyperedge (0 if not alive), phase 1 the dominator count of every vertex.
// export: out[id] = value at the id's current position; import: the value at
// each alive id's position = in[id].
__global__ void k_pass_exchange(InstState *st, int phase, int import, void *buf) {
    InstState &s = st[0];
    const int32_t ids = phase == 0 ? s.m0 : s.n0;
    const int32_t rows = phase == 0 ? s.m : s.n;  // this pass's rows
    const int32_t *o2c = phase == 0 ? s.e_o2c : s.v_o2c;
    for (int32_t id = blockIdx.x * blockDim.x + threadIdx.x; id < ids;
         id += gridDim.x * blockDim.x) {
        const int32_t pos = o2c[id];
        const bool alive = pos >= 0 && pos < rows;
        if (phase == 0) {
            uint8_t *b = static_cast<uint8_t *>(buf);
            if (!import) b[id] = alive ? s.e_del[pos] : 0;
            else if (alive) s.e_del[pos] = b[id] ? 1 : 0;
        } else {
            int32_t *b = static_cast<int32_t *>(buf);
            if (!import) b[id] = alive ? s.v_cnt[pos] : 0;
            else if (alive) s.v_cnt[pos] = b[id];
        }
    }
}

cudaError_t launch_pass_exchange(InstState *st, int phase, int import, void *buf, int sms,
                                 cudaStream_t s) {
    k_pass_exchange<<<grid_for(sms, 2), 256, 0, s>>>(st, phase, import, buf);
    return cudaGetLastError();
}

cudaError_t launch_bounds(InstState *st, int count, int sms, cudaStream_t s, int compact_blocks) {
    const dim3 grid(count > 1 ? per_instance_grid(1 << 20, count) : grid_for(sms, 4), count);
    k_bounds<false><<<grid, 256, 0, s>>>(st, count);
    k_bounds<true><<<grid, 256, 0, s>>>(st, count);
    k_compact_edges<true>
        <<<dim3(compact_blocks > 1 ? compact_blocks : 1, count), 1024, 0, s>>>(st, count);
    return cudaGetLastError();
}

cudaError_t launch_round_phase(InstState *st, Plan *plan, BatchCounters *ctr, int count,
                               int phase, int contraction, int sms, int32_t *kerr,
                               cudaStream_t s, cudaEvent_t ev_contract_begin,
                               cudaEvent_t ev_contract_end, int32_t *done_list,
                               int compact_blocks, int tile_n) {
    const bool tc = contraction == kFp8;
    cudaError_t e0 = launch_phase_prologue(st, plan, ctr, phase, contraction, sms, s);
    if (e0 != cudaSuccess) return e0;
    if (tc) {
        cudaError_t e = launch_tc_tile_list(st, plan, phase, sms, s, 0, 1);
        if (e != cudaSuccess) return e;
    }
    // Timing events: external event nodes when the round is being captured
    // into a graph, plain records when it is launched directly.
    auto record = [s](cudaEvent_t ev) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive)
            cudaEventRecordWithFlags(ev, s, cudaEventRecordExternal);
        else
            cudaEventRecord(ev, s);
    };
    if (ev_contract_begin) record(ev_contract_begin);
    if (tc) {
        cudaError_t e = launch_tc_contract(st, plan, ctr, phase, sms, tile_n, kerr, s);
        if (e != cudaSuccess) return e;
    } else {
        launch_pop(st, plan, phase, 0, 1, sms, s);
    }
    if (ev_contract_end) record(ev_contract_end);
    return launch_phase_epilogue(st, plan, ctr, count, phase, contraction, sms, s, done_list,
                                 compact_blocks);
}

cudaError_t launch_alive_masks(const InstState *st, uint8_t *alive_v, uint8_t *alive_e,
                               cudaStream_t s) {
    k_alive_masks<<<dim3(152, 1), 256, 0, s>>>(st, 1, false, alive_v, alive_e);
    return cudaGetLastError();
}

cudaError_t launch_alive_masks_batch(const InstState *st, int count, uint8_t *alive_v,
                                     uint8_t *alive_e, cudaStream_t s) {
    k_alive_masks<<<dim3(4, count), 256, 0, s>>>(st, count, true, alive_v, alive_e);
    return cudaGetLastError();
}

}  // namespace mhs
