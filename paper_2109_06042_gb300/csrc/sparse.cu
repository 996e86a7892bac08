// sparse.cu -- Algorithm 3 by candidate lists instead of pair tiles.
//
// The contractions decide every pair (i, j) of a row block; of those pairs
// almost none can fire.  For sparse hypergraphs the pairs that can are found
// directly from the vertex -> hyperedge lists, and the result is the same
// set of deletions, pass by pass:
//
//  DP (Algorithm 1).  e_i supersedes e_j iff |e_i \ e_j| <= t, t = f_i - f_j,
//  i.e. iff they share at least need = |e_i| - t vertices.
//   * need >= 2: e_j holds one of any t + 1 vertices of e_i, so it is in the
//     list of one of its rarest ones.  The p-th rarest (p from 0) has to be
//     walked only for f_j <= f_i - p: an e_j that holds none of the p rarer
//     ones has missed p already.  The most popular vertex of e_i is never
//     walked (p <= |e_i| - 2).
//   * need = 1: every e_j holding a vertex v of e_i with f_j = f_i - |e_i| + 1
//     goes.  Per vertex the largest such bound is kept (m1), and every e_j
//     tests its own vertices.  Hyperedges of one vertex keep per vertex the
//     largest demand and, among equals, the lowest index (s1).
//   * need = 2 with both vertices heavy (192 hyperedges or more): the same
//     bound per pair of vertices, in a hash table.  What is left to walk in a
//     heavy vertex's list is need >= 3: 5.7 of 30 million entries on the
//     power-law instance.
//   * need <= 0 (only f_i > |e_i|, or an empty e_i): every e_j with
//     f_j <= f_i - |e_i| goes; one maximum over the instance (loose, empty).
//  A pair is mutual iff both sets and demands are equal; the lower input
//  index stays.  "Supersedes or wins the tie" is transitive and acyclic, so a
//  hyperedge that is deleted need not be tested as a superseder: whatever it
//  supersedes, a surviving one does too.  Deleted hyperedges are therefore
//  skipped as soon as they are flagged, in any order, with the same result.
//  Rule SE is the case t = 0 whatever the demands, with f_i >= f_j.
//
//  MD (Algorithm 2).  A dominator of v_j is in every hyperedge of v_j, so only
//  the members of its smallest one are tested; fewer members than the
//  largest demand decide at once.
//
// Pairs are filtered by 64-bit signatures (a set bit of e_i missing in e_j
// is a vertex missed; a set bit of v_j missing in v_i rules v_i out), then
// decided exactly by searching the sorted rows.  After the first round only
// hyperedges that lost a vertex are superseders and only vertices that lost
// a hyperedge are tested (the incremental argument of the contractions).
//
// What bounds it: latency.  A pass reads a few megabytes from L2 in chains of
// two or three dependent loads, so the whole fixpoint runs in ONE kernel: a
// team of CTAs per instance with a barrier between the phases (a cooperative
// launch), or one CTA per instance of a batch.  Eight lanes share a
// hyperedge or vertex, a warp's four groups in step; lists longer than
// kHeavyList become tasks for whole warps, vertices with more than kHeavyDeg
// hyperedges are handled by whole CTAs.
// Measured on one GB300, the rounds alone (load, kernelization and result
// through the C ABI beside the FP8 contraction's):
//   power law 20,000 x 40,000: 225 us (400 / 1,240)
//   interval 50,000 x 100,000: 358 us (600 / 5,900)
//   uniform 16,000 x 32,000, |e| 2..16: 70 us (200 / 4,150)
#include <algorithm>

#include <cuda_runtime.h>

#include "bounded_wait.cuh"
#include "kernels.h"
#include "mhs_internal.h"

namespace mhs {

namespace {

typedef unsigned long long u64;

constexpr int kG = 8;                  // lanes per hyperedge / vertex
// Loads in flight per lane, in the phases, a task and the build.  Small: the
// phases are short and each round runs through all of them, so what they
// cost most is their code (at 4 throughout, and with the helpers inlined, the
// kernel was 236 KB and every phase waited 5 to 10 us for instructions).
constexpr int kU = 2;
constexpr int kTaskU = 4;
constexpr int kRowU = 2;
// Longer lists become tasks of whole warps, in parts: eight lanes take 0.6 us
// per 16 entries, up to four lists in turn.  At 192 and parts of 1,024, the
// walk of a round with 880 tasks took 32 us, the tasks 18 (power law; 24 and
// below gain nothing).  Where lists are that long on average, tasks only cost
// their barrier (|e| 64 over 2,000 x 4,000: DP 179 us, 200 with tasks from 96
// entries on), so a list also has to be twice as long as the mean, or 4 times
// kHeavyList (Shared::heavy_list).  Parts grow with the mean too, up to 1,024:
// with 256, the tasks of 20,000 hyperedges over 64 vertices do not all find
// room, and eight lanes walk the rest (load and kernelization 531 us; 292 now).
constexpr int kHeavyList = 48;
constexpr int kTaskLen = 256;
// The same for a vertex's bounds, whose entries are read four in flight, like
// the members of a deleted hyperedge (rule SE: tasks of 72 us in a second
// round with 1,024 entries, one at a time; 20 now).
constexpr int kBoundList = 32, kBoundLen = 128;
constexpr int kHeavyDeg = 256;         // vertices of a higher degree: whole CTAs
constexpr int32_t kNoTask = -1, kBoundTask = -2;  // Task.x: unused; a vertex's bounds
constexpr int32_t kGone = 0;           // demand of a deleted hyperedge: no legal one (they are >= 1)
constexpr int kSpThreads = 1024;       // threads of a CTA of a team
constexpr int kMaxTeam = 256;          // CTAs of a team, at most
constexpr int kSpBatchThreads = 512;   // threads of a CTA of a batch
constexpr int kSpBatchBlocks = 2;      // such CTAs per SM
constexpr int64_t kSpTeamNnz = 512;    // incidences per CTA of a team
constexpr int64_t kSpTeamItems = 256;  // hyperedges and vertices per CTA of a team
constexpr uint64_t kTeamWaitNs = 4000000000ull;  // 4 s bound on a team barrier
// Self-test (mhs_selftest_team_wait): this thread's launches wait so long for a
// CTA that never comes; 0: off.
thread_local uint64_t t_absent_ns = 0;

__device__ __forceinline__ u64 sig_bit(int32_t id) {
    return 1ull << (((uint32_t)id * 2654435761u) >> 26);
}
__device__ __forceinline__ u64 rec_sig(int4 r) {
    return (u64)(uint32_t)r.x | ((u64)(uint32_t)r.y << 32);
}
// Rows hold keys: the vertex's degree at load, in 8 bits (exact below 16,
// then 8 steps per octave), above its id.  A row in key order is sorted by one
// order common to all rows, its rarest vertices first.
constexpr uint32_t kIdMask = 0xffffffu;
__device__ __forceinline__ uint32_t row_key(int32_t id, int32_t deg) {
    const uint32_t d = (uint32_t)deg;
    uint32_t q = d;
    if (d >= 16) {
        const int lg = 31 - __clz((int)d);
        q = 16u + 8u * (uint32_t)(lg - 4) + ((d >> (lg - 3)) & 7u);
    }
    return (q << 24) | (uint32_t)id;
}
// Heavy: a degree of 192 or more at load (class 44 starts there).
constexpr uint32_t kHeavyKey = 44u << 24;
__device__ __forceinline__ int32_t key_id(uint32_t key) { return (int32_t)(key & kIdMask); }

// An entry of a vertex's list: hyperedge id (24 bits), demand and size (4
// bits each, 15: that or more), signature folded to 32 bits.  Almost every
// entry of a walk is ruled out by these alone, without a load of the
// hyperedge's record.  Sizes and signatures may be those of an earlier round
// (never smaller than the present ones, so nothing is ruled out wrongly).
__device__ __forceinline__ u64 make_entry(int32_t e, int32_t f, int32_t len, uint32_t fold) {
    return (u64)(uint32_t)e | ((u64)(uint32_t)min(f, 15) << 24) |
           ((u64)(uint32_t)min(len, 15) << 28) | ((u64)fold << 32);
}
__device__ __forceinline__ int32_t entry_id(u64 x) { return (int32_t)((uint32_t)x & kIdMask); }
constexpr u64 kNoEntry = ~0ull;  // (no hyperedge has id 2^24 - 1)
__device__ __forceinline__ uint32_t fold_sig(u64 sig) { return (uint32_t)sig | (uint32_t)(sig >> 32); }
__device__ __forceinline__ int4 make_rec(u64 sig, int32_t z, int32_t w) {
    return make_int4((int32_t)(uint32_t)sig, (int32_t)(uint32_t)(sig >> 32), z, w);
}
__device__ __forceinline__ int32_t vload(const int32_t *p) {
    return *reinterpret_cast<const volatile int32_t *>(p);
}

// The instance's arrays.
struct View {
    const int32_t *eptr;
    uint32_t *row;
    u64 *vedge;
    int32_t *e_o2c, *v_o2c, *estamp, *vstamp, *tstamp;
    int4 *erec, *vrec, *vaux;
    SpAgg *agg;
    int32_t *bound;
    uint32_t *gone;
    SpCtl *ctl;
    View() = default;
    __device__ __forceinline__ explicit View(const InstState &s)
        : eptr(s.eptr), row(s.sp_row), vedge(s.sp_vedge), e_o2c(s.e_o2c), v_o2c(s.v_o2c),
          estamp(s.sp_estamp), vstamp(s.sp_vstamp), tstamp(s.sp_tstamp), erec(s.sp_erec),
          vrec(s.sp_vrec), vaux(s.sp_vaux), agg(s.sp_vagg), bound(s.sp_bound),
          gone(s.sp_gone), ctl(s.sp_ctl) {}
};

// The round state of an instance.
struct Progress {
    int32_t n, m, rounds, changed, dp, md, fe_passes, max_rounds, fe;
    int32_t active, full;
    int64_t k;
    uint64_t t_dp, t_md, t_all;  // ns (kept by the team's first thread)
};

// A CTA's shared memory.  What a phase needs to start (the arrays, the
// round) is kept here: every team barrier empties L1, and a pointer or a
// stack slot fetched again from L2 costs as much as the work itself.
struct Shared {
    View view;
    InstState *s;
    const int32_t *heavy;
    SpPair *pair_tab;
    uint32_t pair_mask;
    int4 *task;
    int32_t task_cap, n0, m0, rule;
    // The threads that reduce the instance: `size` CTAs, this one the `rank`-th.
    int32_t rank, size;
    uint32_t *bar;        // arrivals so far, over all launches (size > 1)
    uint32_t target;      // arrivals that complete the last barrier begun
    uint32_t absent;      // self-test: arrivals waited for in vain
    uint64_t wait_ns;     // bound on a barrier
    int32_t epoch;        // round being executed, from 1
    int32_t par;          // counter parity
    int32_t full;         // every hyperedge and vertex is a candidate
    int32_t ok;           // the last barrier
    int32_t local;        // there is room for degrees (build of a batch)
    int32_t demands;      // (build) some demand is above kFewMisses
    int32_t heavy_list;   // longer lists are walked as tasks,
    int32_t task_len;     // of so many entries
    SpRound got;          // counters read right after it
    Progress g;           // the instance's rounds, as every CTA of the team knows them
    int32_t del, del2;    // deletions of this phase
    int32_t next;         // batch: the instance taken from the queue
    int32_t mf, pos;      // md_lists: one high-degree vertex
    u64 cost, open, sig, small;
    int2 *pairs;          // this instance's pairs (i, j) to be decided exactly
    int32_t pair_cap;
};
// Behind it, for every warp of the CTA:
struct WarpShared {
    int32_t ids[32];             // flagged ids of a chunk
    int2 buf[32 * (kTaskU + 1)]; // pairs not yet listed (decide_pairs: not yet decided)
};
constexpr size_t kSharedBytes = (sizeof(Shared) + 15) / 16 * 16;
constexpr size_t shared_bytes(int threads) { return kSharedBytes + threads / 32 * sizeof(WarpShared); }
extern __shared__ __align__(16) uint8_t sp_smem[];
__device__ __forceinline__ Shared *shared() { return reinterpret_cast<Shared *>(sp_smem); }
// And behind that, in the build of a batch, the degrees of up to kLocalVertices
// vertices, and the places of their lists: a CTA that has an instance to
// itself counts them there (a batch of 4,096 instances with 56 M incidences:
// the load takes 2.9 ms, 3.8 with returning atomics on L2; the places 0.08).
// 3,072: the CTAs' shared memory stays below 48 KB.
constexpr int32_t kLocalVertices = 3072;
__device__ __forceinline__ int32_t *local_degrees() {
    return reinterpret_cast<int32_t *>(sp_smem + shared_bytes(blockDim.x));
}
static_assert(shared_bytes(kSpThreads) <= 48 * 1024 &&
                  shared_bytes(kSpBatchThreads) + 8 * kLocalVertices <= 48 * 1024,
              "more needs cudaFuncAttributeMaxDynamicSharedMemorySize");
__device__ __forceinline__ WarpShared *warp_shared() {
    return reinterpret_cast<WarpShared *>(sp_smem + kSharedBytes) + (threadIdx.x >> 5);
}

// Barrier over the team; false if it timed out.  The CTAs are resident
// together (cooperative launch), and each wait gives up after kTeamWaitNs,
// after which every CTA of the team leaves and the kernel tells the host.  p:
// counters that are complete once every CTA has arrived, read into `got`.
__device__ __noinline__ bool team_sync(const SpRound *p = nullptr) {
    Shared *sh = shared();
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t good = 1;
        if (sh->size > 1) {
            uint32_t *bar = sh->bar;
            const uint32_t target = sh->target + (uint32_t)sh->size;
            sh->target = target;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
            uint64_t t0 = 0;
            for (uint32_t it = 1;; ++it) {
                uint32_t now;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(bar) : "memory");
                if ((int32_t)(now - target - sh->absent) >= 0) break;
                if ((it & 255u) == 0) {
                    const uint64_t t = globaltimer();
                    if (t0 == 0) t0 = t;
                    else if (t - t0 > sh->wait_ns) {
                        atomicOr(&sh->s->status, kErrTimeout);
                        good = 0;
                        break;
                    }
                }
            }
        }
        sh->ok = good;
        if (p) {
            sh->got.dp = vload(&p->dp);
            sh->got.md = vload(&p->md);
            sh->got.ntask = vload(&p->ntask);
            sh->got.npair[0] = vload(&p->npair[0]);
            sh->got.npair[1] = vload(&p->npair[1]);
            sh->got.nbig = vload(&p->nbig);
        }
    }
    __syncthreads();
    return sh->ok != 0;
}

// A thread's place and the round, from shared memory.
struct Ctx {
    Shared *sh;
    int lane, warp, sub, lead;  // lane in the warp, warp in the CTA, lane in the group, its first lane
    int gw, nw;                 // warp of the team, and their number
    int32_t epoch, par;
    bool full;
    __device__ __forceinline__ Ctx() {
        sh = shared();
        lane = threadIdx.x & 31;
        warp = threadIdx.x >> 5;
        sub = lane & (kG - 1);
        lead = lane & ~(kG - 1);
        gw = warp * sh->size + sh->rank;  // neighbours in the id range on different SMs
        nw = (int)(blockDim.x >> 5) * sh->size;
        epoch = sh->epoch;
        par = sh->par;
        full = sh->full != 0;
    }
};

// Reductions over a group; every lane of the warp takes part.
__device__ __forceinline__ u64 group_min(u64 x) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) {
        const u64 y = __shfl_xor_sync(0xffffffffu, x, o);
        x = y < x ? y : x;
    }
    return x;
}
__device__ __forceinline__ u64 group_or(u64 x) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) x |= __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
__device__ __forceinline__ int32_t group_max(int32_t x) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
__device__ __forceinline__ int32_t group_sum(int32_t x) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
// The lanes of this group whose flag is set (bit 0: the group's first lane).
__device__ __forceinline__ unsigned group_ballot(const Ctx &c, bool x) {
    return (__ballot_sync(0xffffffffu, x) >> c.lead) & ((1u << kG) - 1u);
}

// Runs fn(id) for every id in [0, n) with flag(id): a group of lanes per id,
// the warp's four groups in step (an idle group gets id -1), so that a list
// that is longer in one group than in the others costs its excess only once.
// A warp takes chunks of ids; the chunk shrinks to 4 (one per group) when
// there are more warps than work.
template <typename Flag, typename Fn>
__device__ __forceinline__ void for_flagged(const Ctx &c, int32_t n, Flag &&flag, Fn &&fn) {
    int chunk = 32;
    while (chunk > 32 / kG && (int64_t)n < (int64_t)c.nw * chunk) chunk >>= 1;
    int32_t *ids = warp_shared()->ids;
    const int g = c.lane / kG;
#pragma unroll 1
    for (int64_t base = (int64_t)c.gw * chunk; base < n; base += (int64_t)c.nw * chunk) {
        const int32_t id = (int32_t)base + c.lane;
        const bool on = c.lane < chunk && id < n && flag(id);
        const unsigned mk = __ballot_sync(0xffffffffu, on);
        if (!mk) continue;
        if (on) ids[__popc(mk & ((1u << c.lane) - 1u))] = id;
        __syncwarp();
        const int cnt = __popc(mk);
#pragma unroll 1
        for (int q = 0; q < cnt; q += 32 / kG) fn(q + g < cnt ? ids[q + g] : -1);
        __syncwarp();
    }
}

// ------------------------------------------------------------------ bounds --

// The slot of the pair of heavy vertices a < b, or the free one for it.
constexpr int kProbes = 16;
__device__ __forceinline__ SpPair *pair_slot(const Shared *sh, uint32_t a, uint32_t b, int probe) {
    const uint32_t h = a * 0x9e3779b1u ^ (b * 0x85ebca77u + 0x165667b1u);
    return sh->pair_tab + ((((h ^ (h >> 15)) * 0x2c1b3c6du >> 8) + (uint32_t)probe) & sh->pair_mask);
}
__device__ __forceinline__ u64 pair_key(uint32_t a, uint32_t b) { return ((u64)a << 24 | b) + 1; }

// Hyperedge e's bound for the pair of its heavy vertices x and y.
__device__ __forceinline__ void add_pair_bound(Shared *sh, int32_t e, int32_t f, int32_t len,
                                               uint32_t x, uint32_t y) {
    SpAgg *agg = sh->view.agg;
    const uint32_t lo = min(x, y), hi = max(x, y);
    const u64 key = pair_key(lo, hi);
    SpPair *slot = nullptr;
#pragma unroll 1
    for (int q = 0; q < kProbes && !slot; ++q) {
        SpPair *p = pair_slot(sh, lo, hi, q);
        u64 cur = *reinterpret_cast<volatile u64 *>(&p->key);
        if (cur == 0) cur = atomicCAS(&p->key, 0ull, key);
        if (cur == 0 || cur == key) slot = p;
    }
    if (!slot) {
        sh->view.ctl->pairs_full = 1;  // the walks must find what the bounds miss
        return;
    }
    // (popular pairs have hundreds of writers: look before an atomic)
    const int32_t bound = len == 2 ? f : f - len + 2;
    const uint32_t most = (uint32_t)bound << 1;  // (bit 0: for whole CTAs)
    const uint32_t hx = *reinterpret_cast<volatile uint32_t *>(&agg[x].heavy);
    const uint32_t hy = *reinterpret_cast<volatile uint32_t *>(&agg[y].heavy);
    if ((hx & ~1u) < most) atomicMax(&agg[x].heavy, most | (hx & 1u));
    if ((hy & ~1u) < most) atomicMax(&agg[y].heavy, most | (hy & 1u));
    if (len == 2) {
        const u64 s2 = ((u64)(uint32_t)f << 32) | (0xffffffffu - (uint32_t)e);
        if (*reinterpret_cast<volatile u64 *>(&slot->s2) < s2) atomicMax(&slot->s2, s2);
    } else if (vload(&slot->m2) < bound) {
        atomicMax(&slot->m2, bound);
    }
}

// True if e_j goes by the bound of its heavy vertices x and y.
__device__ __forceinline__ bool pair_hit(const Shared *sh, uint32_t x, uint32_t y, int32_t j,
                                         int32_t fj, int32_t lenj) {
    const uint32_t lo = min(x, y), hi = max(x, y);
    const u64 key = pair_key(lo, hi);
#pragma unroll 1
    for (int q = 0; q < kProbes; ++q) {
        const SpPair *p = pair_slot(sh, lo, hi, q);
        const u64 cur = p->key;
        if (cur == 0) return false;
        if (cur != key) continue;
        if (p->m2 >= fj) return true;
        const u64 s2 = p->s2;
        return s2 && fj <= (int32_t)(s2 >> 32) &&
               (lenj >= 3 || (int32_t)(0xffffffffu - (uint32_t)s2) != j);
    }
    return false;
}

// Rows of many heavy vertices, whose pairs grow with the square: above kPairRow
// a superseder sets no pair bounds and walks its heavy lists whole; above
// kPairTest a hyperedge is not tested against them, and every walk is whole.
// Every pair of every row, as far as the table had room, took (load and
// kernelization, us; so / now / by the contraction):
//   one hyperedge of 600, demand 600, among 20,000 of 10 over 700 vertices
//                                                          124,935 /  721 / 549
//   20,000 of 30 over 1,000 vertices, of demand |e|          3,650 /  858 / 652
constexpr int32_t kPairRow = 6, kPairTest = 64;
__device__ __forceinline__ bool many_heavy(const uint32_t *row, int32_t len, int32_t most) {
    return len > most && row[len - 1 - most] >= kHeavyKey;  // (they end the row)
}

// What hyperedge e (row: its keys) contributes to the tests with need <= 1,
// and in full rounds to those of pairs of heavy vertices.  One group, without
// the others.
__device__ __noinline__ void contribute(int32_t e, int32_t f, int32_t len, const uint32_t *row) {
    Shared *sh = shared();
    const int sub = threadIdx.x & (kG - 1);
    SpAgg *agg = sh->view.agg;
    int32_t *tstamp = sh->view.tstamp;
    SpCtl *ctl = sh->view.ctl;
    const int32_t epoch = sh->epoch;
    if (len <= 1) {
        if (sub != 0) return;
        const u64 key = ((u64)(uint32_t)f << 32) | (0xffffffffu - (uint32_t)e);
        if (len == 0) {
            if (atomicMax(&ctl->empty, key) < key) ctl->c[sh->par].scan_all = 1;
            return;
        }
        const int32_t x = key_id(row[0]);
        if (*reinterpret_cast<volatile u64 *>(&agg[x].s1) < key && atomicMax(&agg[x].s1, key) < key) {
            tstamp[x] = epoch;
            atomicMax(&sh->view.bound[x], f);
        }
        if (!sh->rule && f > 1 && atomicMax(&ctl->loose, f - 1) < f - 1) ctl->c[sh->par].scan_all = 1;
        return;
    }
    if (sh->rule) return;
    if (sh->full && many_heavy(row, len, kPairTest)) ctl->pairs_full = 1;
    if (f < len - 1) return;
    const int32_t m1 = f - len + 1;
    if (m1 >= 1)
#pragma unroll 1
        for (int32_t k = sub; k < len; k += kG) {
            const int32_t x = key_id(row[k]);
            if (vload(&agg[x].m1) < m1 && atomicMax(&agg[x].m1, m1) < m1) {
                tstamp[x] = epoch;
                atomicMax(&sh->view.bound[x], m1);
            }
        }
    if (f > len && sub == 0 && atomicMax(&ctl->loose, f - len) < f - len)
        ctl->c[sh->par].scan_all = 1;
    if (!sh->full || many_heavy(row, len, kPairRow) || vload(&ctl->pairs_full)) return;
    // every two heavy ones: they end the row, and most rows have fewer
    int32_t a = len - 1;
    while (a > 0 && row[a - 1] >= kHeavyKey) --a;
#pragma unroll 1
    for (; a < len - 1; ++a) {
        const uint32_t ka = row[a];
#pragma unroll 1
        for (int32_t k = a + 1 + sub; k < len; k += kG)
            add_pair_bound(sh, e, f, len, ka & kIdMask, row[k] & kIdMask);
    }
}

// ---------------------------------------------------------------- DP pass --

// Flag hyperedge x as deleted (once), and its vertices as MD candidates.
// One thread.
__device__ __noinline__ void delete_edge(int32_t x) {
    Shared *sh = shared();
    const View &v = sh->view;
    if (atomicExch(&v.erec[x].z, kGone) == kGone) return;
    atomicAdd(&sh->del, 1);
    const int32_t epoch = sh->epoch;
    v.e_o2c[x] = -1 - epoch;
    atomicOr(&v.gone[x >> 5], 1u << (x & 31));
    if (sh->full) return;  // every vertex is a candidate
    const int32_t len = v.erec[x].w;
    const uint32_t *row = v.row + v.eptr[x];
    // (a store waits for its own load, a serial chain of L2 latencies, unless
    // several are in flight)
#pragma unroll 4
    for (int32_t k = 0; k < len; ++k) v.vstamp[key_id(row[k])] = epoch;
}

// True if e_j goes by the need <= 1 bounds of one of its vertices.
__device__ __forceinline__ bool agg_hit(int4 a, int32_t j, int32_t fj, int32_t lenj) {
    if (a.x >= fj) return true;                      // m1
    if (a.w == 0) return false;                      // s1: demand a.w, ~index a.z
    return fj <= a.w && (lenj >= 2 || (int32_t)(0xffffffffu - (uint32_t)a.z) != j);
}
// True if e_j goes by the instance-wide bounds.
__device__ __forceinline__ bool global_hit(int32_t loose, u64 empty, int32_t j, int32_t fj,
                                           int32_t lenj) {
    if (fj <= loose) return true;
    return empty && fj <= (int32_t)(empty >> 32) &&
           (lenj > 0 || (int32_t)(0xffffffffu - (uint32_t)empty) != j);
}
__device__ __forceinline__ int4 load_agg(const SpAgg *p) {
    return *reinterpret_cast<const int4 *>(p);
}

// The counters of the task and pair lists must not wrap, however much finds no
// room: a reservation wholly behind the end is given back, so that beside the
// one that crossed it at most one per warp of the team is counted at a time.
// (Looking at the counter before each addition costs a chain of two L2
// latencies: power law 396 -> 410 us, with SE and FE 1,134 -> 1,217.)
constexpr int32_t kMaxReserve = 1 << 17;  // places a warp reserves at once, at most
static_assert((int64_t)kMaxTeam * (kSpThreads / 32) * kMaxReserve + kMaxListed < (1ll << 31),
              "the lists' counters cannot wrap");

// Reserve tasks for the list of vertex x, in the lanes with want set (the
// whole warp, one atomic); false if there is no room (the caller walks the
// list itself).
__device__ __noinline__ bool push_tasks(bool want, int32_t i, int32_t x, int32_t p, int32_t deg,
                                        int32_t part) {
    if (!__any_sync(0xffffffffu, want)) return false;
    Shared *sh = shared();
    const int lane = threadIdx.x & 31;
    const int32_t cap = sh->task_cap;
    const int32_t parts = want ? (deg + part - 1) / part : 0;
    int32_t inc = parts;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    // (the lanes before the first that does not fit are a prefix; 65,536 parts, the
    // most of one lane, fit)
    const int32_t total = __reduce_max_sync(0xffffffffu, inc <= kMaxReserve ? inc : 0);
    int32_t *const ntask = &sh->view.ctl->c[sh->par].ntask;
    int32_t at = 0;
    if (lane == 31) {
        at = atomicAdd(ntask, total);
        if (at >= cap) atomicSub(ntask, total);
    }
    at = __shfl_sync(0xffffffffu, at, 31) + inc - parts;
    if (inc > kMaxReserve) return false;
    const bool fits = at <= cap - parts;
#pragma unroll 1
    for (int32_t q = 0; q < parts; ++q)
        if (at + q < cap)
            sh->task[at + q] = fits ? make_int4(i, x, p, q) : make_int4(kNoTask, 0, 0, 0);
    return want && fits;
}

// The hyperedges of vertex x that its bounds delete: entries k0, k0 + step, ... < k1.
__device__ __noinline__ void bound_list(int32_t x, int32_t k0, int32_t k1, int32_t step, int shard,
                                        int nshards) {
    const View &v = shared()->view;
    const int4 a = load_agg(v.agg + x);
    const u64 *list = v.vedge + v.vrec[x].w;
#pragma unroll 1
    for (int32_t k = k0; k < k1; k += kTaskU * step) {
        int32_t j[kTaskU];
        int4 r[kTaskU];
#pragma unroll
        for (int u = 0; u < kTaskU; ++u) {
            j[u] = k + u * step < k1 ? entry_id(list[k + u * step]) : -1;
            if (nshards > 1 && j[u] >= 0 && (j[u] >> 7) % nshards != shard) j[u] = -1;
        }
#pragma unroll
        for (int u = 0; u < kTaskU; ++u) r[u] = j[u] >= 0 ? v.erec[j[u]] : make_int4(0, 0, kGone, 0);
#pragma unroll
        for (int u = 0; u < kTaskU; ++u)
            if (r[u].z != kGone && agg_hit(a, j[u], r[u].z, r[u].w)) delete_edge(j[u]);
    }
}

// The tests with need <= 1 (and of pairs of heavy vertices) for every
// hyperedge: full rounds, or an instance-wide bound rose.
__device__ __noinline__ void dp_bounds_all(int shard, int nshards) {
    const Ctx c;
    const View &v = c.sh->view;
    const int32_t loose = vload(&v.ctl->loose);
    const u64 empty = *reinterpret_cast<volatile u64 *>(&v.ctl->empty);
    const int32_t *const e_o2c = v.e_o2c, *const eptr = v.eptr;
    const int4 *const erec = v.erec;
    const uint32_t *const rows = v.row;
    const SpAgg *const agg = v.agg;
    const int32_t *const bound = v.bound;
    for_flagged(
        c, c.sh->m0,
        [&](int32_t j) { return e_o2c[j] >= 0 && (nshards == 1 || (j >> 7) % nshards == shard); },
        [&](int32_t j) {
            const int4 r = j >= 0 ? erec[j] : make_int4(0, 0, kGone, 0);
            const uint32_t *row = j >= 0 ? rows + eptr[j] : nullptr;
            const int32_t fj = r.z, len = fj == kGone ? 0 : r.w;
            bool hit = fj != kGone && global_hit(loose, empty, j, fj, r.w);
            int32_t heavy = 0;  // heavy vertices
            const int32_t maxlen = c.full ? __reduce_max_sync(0xffffffffu, len) : 0;
#pragma unroll 1
            for (int32_t k0 = 0; k0 < maxlen; k0 += kU * kG) {
                uint32_t x[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int32_t k = k0 + u * kG + c.sub;
                    x[u] = k < len ? row[k] : 0xffffffffu;
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    if (x[u] == 0xffffffffu || bound[key_id(x[u])] < fj) continue;
                    // (by its own bound, a hyperedge of one vertex does not go)
                    hit |= r.w >= 2 || agg_hit(load_agg(agg + key_id(x[u])), j, fj, r.w);
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) heavy += x[u] >= kHeavyKey && x[u] != 0xffffffffu;
            }
            hit = hit && fj != kGone;
            // every two heavy ones, unless decided
            int32_t end = 0;
            if (__any_sync(0xffffffffu, heavy != 0)) {
                heavy = group_sum(heavy);
                end = group_ballot(c, hit) == 0 && heavy > 1 && heavy <= kPairTest ? len : 0;
                end = __shfl_sync(0xffffffffu, end, c.lead);
            }
            const int32_t maxend = __reduce_max_sync(0xffffffffu, end);
#pragma unroll 1
            for (int32_t a = 0; a < maxend; ++a) {
                const uint32_t ka = a < end ? row[a] : 0;
                bool on = ka >= kHeavyKey;
                if (!__any_sync(0xffffffffu, on)) continue;
                on = on && (int32_t)(agg[ka & kIdMask].heavy >> 1) >= fj;
                if (on)
#pragma unroll 1
                    for (int32_t k = a + 1 + c.sub; k < end && !hit; k += kG) {
                        const uint32_t y = row[k] & kIdMask;
                        if ((int32_t)(agg[y].heavy >> 1) >= fj) hit = pair_hit(c.sh, ka & kIdMask, y, j, fj, r.w);
                    }
                __syncwarp();
                if (group_ballot(c, hit)) end = 0;
            }
            if (group_ballot(c, hit) && c.sub == 0 && fj != kGone) delete_edge(j);
            __syncwarp();
        });
}

// The same for the hyperedges of the vertices whose bounds rose.
__device__ __noinline__ void dp_bounds_touched(int shard, int nshards) {
    const Ctx c;
    const View &v = c.sh->view;
    const int32_t *const tstamp = v.tstamp, *const v_o2c = v.v_o2c;
    const int4 *const vrec = v.vrec;
    for_flagged(
        c, c.sh->n0, [&](int32_t x) { return tstamp[x] == c.epoch && v_o2c[x] >= 0; },
        [&](int32_t x) {
            const int32_t deg = x >= 0 ? vrec[x].z : 0;
            bool later = push_tasks(deg > kBoundList && c.sub == 0, kBoundTask, x, 0, deg, kBoundLen);
            later = __shfl_sync(0xffffffffu, later, c.lead);
            if (x >= 0 && !later) bound_list(x, c.sub, deg, kG, shard, nshards);
            __syncwarp();
        });
}

__device__ __forceinline__ void dp_bounds(int shard, int nshards) {
    const Shared *sh = shared();
    if (sh->full || vload(&sh->view.ctl->c[sh->par].scan_all)) dp_bounds_all(shard, nshards);
    if (!sh->full) dp_bounds_touched(shard, nshards);
}

// Vertices of a row to be walked: need >= 2 leaves out the most popular.
__device__ __forceinline__ int32_t walk_count(int32_t rule, int32_t f, int32_t len) {
    if (len < 2) return 0;
    return rule ? 1 : min(f, len - 1);
}

// What a walk of `entries` list entries counts as open (SpTotals).  Where the demand allows as many missed vertices as the 64-bit signatures show of
// two unrelated sets (less a standard deviation), most entries become pairs that
// are searched row by row: 45 ps each at |e| 12, 950 at 60 (8 to 14 ps an entry
// that is ruled out at once).  Demands up to 4 never do.
constexpr int32_t kFewMisses = 4;
__device__ __forceinline__ float open_walk(float entries, int32_t f, int32_t len) {
    const float unset = __expf((float)len * (-1.f / 64.f));  // share of a signature's bits
    const float missed = 64.f * unset * (1.f - unset);
    const float dev = sqrtf(missed * (1.f - unset));
    return (float)f - 1.f >= missed - dev ? entries * 1.5f * (float)len : 0.f;
}
// And a walk of many lists, which one group takes one after the other (one
// hyperedge of demand and size 300 among 20,000 of 10 over 3,000 vertices: 1.4 ms
// in all, 0.86 by the contraction; 3,000: 14 and 1.0).
constexpr int32_t kManyLists = 128;
constexpr float kPerListSquared = 4096.f;

struct Walker {  // the superseder of a walk
    int32_t i, f, len, rule;
    uint32_t fold;
};

// May e_i supersede the hyperedge of entry x of its p-th rarest vertex's
// list?  (Demands and sizes of 15 stand for larger ones: decide_pairs looks.)
// p carries kNeed3 in the lists of heavy vertices that only pairs with
// need >= 3 are taken from.
constexpr int32_t kNeed3 = 1 << 30;
__device__ __forceinline__ bool may_supersede(const uint32_t *gone, const Walker &w, int32_t p,
                                              u64 x) {
    const int32_t fj = (int32_t)((uint32_t)x >> 24) & 15, lenj = (int32_t)((uint32_t)x >> 28);
    const int32_t t = w.rule ? 0 : w.f - fj;
    // the strongest test first
    if (__popc(w.fold & ~(uint32_t)(x >> 32)) > t) return false;
    if (fj > w.f - (p & ~kNeed3) || entry_id(x) == w.i) return false;
    // need <= 1 (2): dp_bounds
    if (!w.rule && fj < 15 && w.len - t < (p & kNeed3 ? 3 : 2)) return false;
    if (lenj < 15 && lenj < w.len - t) return false;
    // lists keep the hyperedges deleted since they were last rewritten: most
    // of what gets here in a first round (power-law: 3.07 of 3.25 million)
    const int32_t j = entry_id(x);
    return !((gone[j >> 5] >> (j & 31)) & 1u);
}

// Can the pair (i, j) fire, by the records as they are now?  Leaves the
// slack in *t.
__device__ __forceinline__ bool pair_open(int32_t rule, int4 ri, int4 rj, int32_t *t) {
    if (ri.z == kGone || rj.z == kGone || rj.z > ri.z) return false;
    *t = rule ? 0 : ri.z - rj.z;
    return rj.w >= ri.w - *t && __popcll(rec_sig(ri) & ~rec_sig(rj)) <= *t;
}

// Place of `key` in a row of len keys, or of the next larger one.
__device__ __forceinline__ int32_t find_key(const uint32_t *row, int32_t len, uint32_t key) {
    int32_t lo = 0, hi = len;
#pragma unroll 1
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (row[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Decide the pair (i, j) of each group (i < 0: none) exactly: |e_i \ e_j| <= t.
// Each lane looks for one vertex of e_i at a time (rows are in key order).
// The whole warp.
__device__ __noinline__ void decide_group(int2 ij) {
    const Ctx c;
    const View &v = c.sh->view;
    const int32_t rule = c.sh->rule;
    const int4 gone = make_int4(0, 0, kGone, 0);
    const int4 ri = ij.x >= 0 ? v.erec[ij.x] : gone;
    const int4 rj = ij.x >= 0 ? v.erec[ij.y] : gone;
    const uint32_t *rowi = ij.x >= 0 ? v.row + v.eptr[ij.x] : nullptr;
    const uint32_t *rowj = ij.x >= 0 ? v.row + v.eptr[ij.y] : nullptr;
    int32_t t = 0;
    const bool mine = pair_open(rule, ri, rj, &t);
    // (one lane's view: the records may change under the others)
    const bool open = __shfl_sync(0xffffffffu, mine, c.lead);
    t = __shfl_sync(0xffffffffu, t, c.lead);
    const int32_t leni = open ? ri.w : 0, lenj = rj.w;
    const int32_t maxi = __reduce_max_sync(0xffffffffu, leni);
    int32_t miss = 0;
#pragma unroll 1
    for (int32_t k0 = 0; k0 < maxi; k0 += kG) {
        const int32_t k = k0 + c.sub;
        bool lost = false;
        if (k < leni && miss <= t) {
            const uint32_t a = rowi[k];
            const int32_t at = find_key(rowj, lenj, a);
            lost = at >= lenj || rowj[at] != a;
        }
        __syncwarp();
        miss += __popc(group_ballot(c, lost));
        if (!__any_sync(0xffffffffu, miss <= t && k0 + kG < leni)) break;
    }
    if (open && miss <= t && c.sub == 0) {
        // mutual (equal sets and demands): the lower index stays
        const bool eq = miss == 0 && leni == lenj && ri.z == rj.z;
        delete_edge(eq && ij.y < ij.x ? ij.x : ij.y);
    }
    __syncwarp();
}

// The pairs that may fire are few, and the walks find them very unevenly (a
// warp hundreds, most none), so they are listed, and decided by all threads
// of the team alike once the walks are done.  A warp gathers them in shared
// memory and lists 32 or more at a time.
__device__ __noinline__ void list_pairs(int32_t which, int32_t base, int32_t n) {
    const Ctx c;
    Shared *sh = c.sh;
    int2 *const buf = warp_shared()->buf;
    __syncwarp();
    int32_t *const npair = &sh->view.ctl->c[c.par].npair[which];
    int32_t at = 0;
    if (c.lane == 0) {
        at = atomicAdd(npair, n);
        if (at >= sh->pair_cap - base) atomicSub(npair, n);
    }
    const int64_t to = (int64_t)base + __shfl_sync(0xffffffffu, at, 0);
#pragma unroll 1
    for (int32_t k = c.lane; k < n; k += 32)
        if (to + k < sh->pair_cap) sh->pairs[to + k] = buf[k];
    __syncwarp();
    if (to + n <= sh->pair_cap) return;
    // no room: decided here, as in decide_pairs by one lane's look at the records
    // first (without: n 300, m 4,000, |e| 2..16, all demands 50, 855 us; 358 with)
    const View &v = sh->view;
    int32_t open = 0;
#pragma unroll 1
    for (int32_t k0 = 0; k0 < n; k0 += 32) {
        const int32_t k = k0 + c.lane;
        const int2 ij = k < n && to + k >= sh->pair_cap ? buf[k] : make_int2(-1, -1);
        int32_t t;
        const bool on = ij.x >= 0 && pair_open(sh->rule, v.erec[ij.x], v.erec[ij.y], &t);
        const unsigned mk = __ballot_sync(0xffffffffu, on);
        if (on) buf[open + __popc(mk & ((1u << c.lane) - 1u))] = ij;
        open += __popc(mk);
        __syncwarp();
    }
#pragma unroll 1
    for (int32_t k0 = 0; k0 < open; k0 += 32 / kG) {
        const int32_t k = k0 + c.lane / kG;
        decide_group(k < open ? buf[k] : make_int2(-1, -1));
    }
    __syncwarp();
}
struct Pairs {
    int2 *buf;
    int32_t which;  // the walks' list (0), or the tasks' behind it (1)
    int32_t base;   // its first place
    int32_t n = 0;  // pairs in the buffer, the same in every lane
    __device__ __forceinline__ Pairs(const Ctx &c, int32_t w)
        : buf(warp_shared()->buf), which(w), base(w ? min(c.sh->got.npair[0], c.sh->pair_cap) : 0) {}
    // At most kTaskU times between two calls of list().
    __device__ __forceinline__ void push(const Ctx &c, bool want, int32_t i, int32_t j) {
        const unsigned mk = __ballot_sync(0xffffffffu, want);
        if (want) buf[n + __popc(mk & ((1u << c.lane) - 1u))] = make_int2(i, j);
        n += __popc(mk);
    }
    __device__ __forceinline__ void list(int32_t least) {
        if (n < least) return;
        list_pairs(which, base, n);
        n = 0;
    }
};

// After the barrier that ends a walk: decide the pairs of a list.  First
// each lane looks at one pair's records (most pairs fall here: the hyperedge
// is deleted by now, or its whole signature rules it out); the rest goes to
// groups of lanes.  (One thread per pair to the end: 103 us for the 220,000
// pairs of the 2,000 x 4,000 interval instance, in chains of 100 loads.)
__device__ __noinline__ void decide_pairs(int32_t which) {
    const Ctx c;
    Shared *sh = c.sh;
    const View &v = sh->view;
    const int2 *pairs = sh->pairs;
    const int32_t rule = sh->rule;
    const int32_t from = which ? min(sh->got.npair[0], sh->pair_cap) : 0;
    const int64_t to = min((int64_t)from + sh->got.npair[which], (int64_t)sh->pair_cap);
    int2 *buf = warp_shared()->buf;
    int32_t n = 0;  // pairs in the buffer
    int32_t chunk = 32;  // fewer per warp when there are more warps than work
    while (chunk > 32 / kG && to - from < (int64_t)c.nw * chunk) chunk >>= 1;
#pragma unroll 1
    for (int64_t base = from + (int64_t)c.gw * chunk;; base += (int64_t)c.nw * chunk) {
        const bool last = base >= to;
        if (!last) {
            const bool on = c.lane < chunk && base + c.lane < to;
            const int2 ij = on ? pairs[base + c.lane] : make_int2(-1, -1);
            int32_t t;
            const bool open = on && pair_open(rule, v.erec[ij.x], v.erec[ij.y], &t);
            const unsigned mk = __ballot_sync(0xffffffffu, open);
            if (open) buf[n + __popc(mk & ((1u << c.lane) - 1u))] = ij;
            n += __popc(mk);
            __syncwarp();
        }
        // whole sets of four, then the rest at the end
#pragma unroll 1
        while (n >= (last ? 1 : 32 / kG)) {
            const int32_t q = n - 1 - c.lane / kG;
            decide_group(q >= 0 ? buf[q] : make_int2(-1, -1));
            n = max(n - 32 / kG, 0);
        }
        if (last) break;
    }
}

// The tests with need >= 2: short lists at once, long ones as tasks.
__device__ __noinline__ void dp_walk(int shard, int nshards) {
    const Ctx c;
    const View &v = c.sh->view;
    const int32_t rule = c.sh->rule;
    const bool bounded = c.full && !rule && !vload(&v.ctl->pairs_full);
    const int32_t *const e_o2c = v.e_o2c, *const estamp = v.estamp, *const eptr = v.eptr;
    const int4 *const erec = v.erec, *const vrec = v.vrec;
    const uint32_t *const rows = v.row, *const gone = v.gone;
    const u64 *const vedge = v.vedge;
    const int32_t heavy_list = c.sh->heavy_list, task_len = c.sh->task_len;
    Pairs pairs(c, 0);
    for_flagged(
        c, c.sh->m0,
        [&](int32_t i) {
            return (c.full ? e_o2c[i] >= 0 : estamp[i] == c.epoch) &&
                   (nshards == 1 || (i >> 7) % nshards == shard);
        },
        [&](int32_t i) {
            const int4 r = i >= 0 ? erec[i] : make_int4(0, 0, kGone, 0);
            const uint32_t *row = i >= 0 ? rows + eptr[i] : nullptr;
            Walker w;
            w.i = i;
            // one lane's view of the flag: another might read it later
            w.f = __shfl_sync(0xffffffffu, r.z, c.lead);
            w.len = r.w;
            w.fold = fold_sig(rec_sig(r));
            w.rule = rule;
            const int32_t np = w.f == kGone ? 0 : walk_count(rule, w.f, w.len);
            const int32_t npmax = __reduce_max_sync(0xffffffffu, np);
            // (a smaller demand leaves need >= 3 in any case)
            const bool mine = bounded && !(np > 0 && w.f >= w.len - 1 && many_heavy(row, w.len, kPairRow));
#pragma unroll 1
            for (int32_t p0 = 0; p0 < npmax; p0 += kG) {
                // one of the next 8 vertices per lane
                int32_t p = p0 + c.sub;
                const uint32_t key = p < np ? row[p] : 0;
                int32_t x = p < np ? key_id(key) : -1;
                if (mine && key >= kHeavyKey) {  // its pairs with need 2 went by the bounds
                    if (p > w.len - 3) x = -1;
                    p |= kNeed3;
                }
                const int4 vr = x >= 0 ? vrec[x] : make_int4(0, 0, 0, 0);
                int32_t deg = vr.z;
                if (push_tasks(deg > heavy_list, i, x, p, deg, task_len)) deg = 0;
                const int32_t lists = min(npmax - p0, kG);
#pragma unroll 1
                for (int q = 0; q < lists; ++q) {
                    const int32_t dq = __shfl_sync(0xffffffffu, deg | (p & kNeed3), q, kG);
                    const int32_t b = __shfl_sync(0xffffffffu, vr.w, q, kG);
                    const int32_t d = dq & ~kNeed3, lp = (p0 + q) | (dq & kNeed3);
                    const int32_t maxd = __reduce_max_sync(0xffffffffu, d);
#pragma unroll 1
                    for (int32_t o = c.sub; o - c.sub < maxd; o += kU * kG) {
                        u64 ent[kU];
                        bool may[kU];
#pragma unroll
                        for (int u = 0; u < kU; ++u)
                            ent[u] = o + u * kG < d ? vedge[b + o + u * kG] : kNoEntry;
#pragma unroll
                        for (int u = 0; u < kU; ++u)
                            may[u] = ent[u] != kNoEntry && may_supersede(gone, w, lp, ent[u]);
                        bool any = false;
#pragma unroll
                        for (int u = 0; u < kU; ++u) any |= may[u];
                        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
                        for (int u = 0; u < kU; ++u) pairs.push(c, may[u], i, entry_id(ent[u]));
                        pairs.list(32);
                    }
                }
            }
        });
    pairs.list(1);
}

// The tasks: one warp per task_len entries of a long list.
__device__ __noinline__ void dp_tasks(int shard, int nshards) {
    const Ctx c;
    const View &v = c.sh->view;
    const int32_t nt = min(c.sh->got.ntask, c.sh->task_cap);
    const uint32_t *const gone = v.gone;
    Pairs pairs(c, 1);
#pragma unroll 1
    for (int32_t t = c.gw; t < nt; t += c.nw) {
        const int4 tk = c.sh->task[t];
        if (tk.x == kNoTask) continue;
        const int4 vr = v.vrec[tk.y];
        const int4 r = tk.x >= 0 ? v.erec[tk.x] : make_int4(0, 0, 0, 0);
        const int32_t part = tk.x == kBoundTask ? kBoundLen : c.sh->task_len;
        const int32_t k0 = tk.w * part, k1 = min(k0 + part, vr.z);
        if (tk.x == kBoundTask) {
            bound_list(tk.y, k0 + c.lane, k1, 32, shard, nshards);
            __syncwarp();
            continue;
        }
        Walker w;
        w.i = tk.x;
        w.f = __shfl_sync(0xffffffffu, r.z, 0);
        if (w.f == kGone) continue;
        w.len = r.w;
        w.fold = fold_sig(rec_sig(r));
        w.rule = c.sh->rule;
        const u64 *list = v.vedge + vr.w;
#pragma unroll 1
        for (int32_t k = k0 + c.lane; k - c.lane < k1; k += kTaskU * 32) {
            u64 ent[kTaskU];
            unsigned may = 0;
#pragma unroll
            for (int u = 0; u < kTaskU; ++u) ent[u] = k + u * 32 < k1 ? list[k + u * 32] : kNoEntry;
#pragma unroll
            for (int u = 0; u < kTaskU; ++u)
                may |= (ent[u] != kNoEntry && may_supersede(gone, w, tk.z, ent[u]) ? 1u : 0u) << u;
            if (!__any_sync(0xffffffffu, may != 0)) continue;
#pragma unroll
            for (int u = 0; u < kTaskU; ++u) pairs.push(c, (may >> u) & 1u, tk.x, entry_id(ent[u]));
            pairs.list(32);
        }
    }
    pairs.list(1);
}

// Rows of the candidates without the vertices MD deleted, their signatures
// and contributions.
__device__ __noinline__ void dp_rows() {
    const Ctx c;
    const View &v = c.sh->view;
    const int32_t *const e_o2c = v.e_o2c, *const estamp = v.estamp, *const v_o2c = v.v_o2c;
    for_flagged(
        c, c.sh->m0, [&](int32_t e) { return e_o2c[e] >= 0 && (c.full || estamp[e] == c.epoch); },
        [&](int32_t e) {
            const int4 r = e >= 0 ? v.erec[e] : make_int4(0, 0, 0, 0);
            uint32_t *row = e >= 0 ? v.row + v.eptr[e] : nullptr;
            u64 sig = 0;
            int32_t w = 0;
            const int32_t maxlen = __reduce_max_sync(0xffffffffu, r.w);
#pragma unroll 1
            for (int32_t k0 = 0; k0 < maxlen; k0 += kG) {
                const int32_t k = k0 + c.sub;
                const uint32_t x = k < r.w ? row[k] : 0;
                const bool keep = k < r.w && v_o2c[key_id(x)] >= 0;
                const unsigned b = group_ballot(c, keep);
                if (keep) {
                    sig |= sig_bit(key_id(x));
                    row[w + __popc(b & ((1u << c.sub) - 1u))] = x;
                }
                w += __popc(b);
            }
            sig = group_or(sig);
            __syncwarp();
            if (e >= 0) {
                if (c.sub == 0) v.erec[e] = make_rec(sig, r.z, w);
                contribute(e, r.z, w, row);
            }
            __syncwarp();
        });
}

// ---------------------------------------------------------------- MD pass --

__device__ __forceinline__ bool vertex_candidate(const Ctx &c, const View &v, int32_t x) {
    return v.v_o2c[x] >= 0 && (c.full || v.vstamp[x] == c.epoch);
}

// Lists of the candidates without the hyperedges DP deleted; degree,
// signature, largest demand and smallest hyperedge.
__device__ __noinline__ void md_lists() {
    const Ctx c;
    const View &v = c.sh->view;
    const int4 *const erec = v.erec;
    for_flagged(
        c, c.sh->n0, [&](int32_t x) { return vertex_candidate(c, v, x) && !(v.agg[x].heavy & 1); },
        [&](int32_t x) {
            const int4 vr = x >= 0 ? v.vrec[x] : make_int4(0, 0, 0, 0);
            u64 *list = v.vedge + vr.w;
            u64 sig = 0, small = ~0ull;
            int32_t w = 0, mf = 0;
            const int32_t maxdeg = __reduce_max_sync(0xffffffffu, vr.z);
#pragma unroll 1
            for (int32_t k0 = 0; k0 < maxdeg; k0 += kU * kG) {
                u64 ent[kU];
                int4 r[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int32_t k = k0 + u * kG + c.sub;
                    ent[u] = k < vr.z ? list[k] : kNoEntry;
                }
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    r[u] = ent[u] != kNoEntry ? erec[entry_id(ent[u])] : make_int4(0, 0, kGone, 0);
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const bool keep = r[u].z != kGone;
                    const unsigned b = group_ballot(c, keep);
                    if (keep) {
                        const int32_t e = entry_id(ent[u]);
                        sig |= sig_bit(e);
                        mf = max(mf, r[u].z);
                        const u64 key = ((u64)(uint32_t)r[u].w << 32) | (uint32_t)e;
                        small = key < small ? key : small;
                        list[w + __popc(b & ((1u << c.sub) - 1u))] =
                            make_entry(e, r[u].z, r[u].w, fold_sig(rec_sig(r[u])));
                    }
                    w += __popc(b);
                }
            }
            sig = group_or(sig);
            small = group_min(small);
            mf = group_max(mf);
            if (x >= 0 && c.sub == 0) {
                v.vrec[x] = make_rec(sig, w, vr.w);
                const int32_t e0 = (int32_t)(uint32_t)small;
                v.vaux[x] = make_int4(e0, mf, w > 0 ? v.eptr[e0] : 0, (int32_t)(small >> 32));
            }
        });
    // the vertices whose degree at load was above kHeavyDeg: one CTA each
    Shared *sh = c.sh;
    const int32_t nh = vload(&v.ctl->n_heavy);
#pragma unroll 1
    for (int32_t h = sh->rank; h < nh; h += sh->size) {
        const int32_t x = sh->heavy[h];
        if (!vertex_candidate(c, v, x)) continue;
        const int4 vr = v.vrec[x];
        u64 *list = v.vedge + vr.w;
        __syncthreads();  // every thread has the record before it is replaced
        if (threadIdx.x == 0) { sh->pos = 0; sh->mf = 0; sh->sig = 0; sh->small = ~0ull; }
        __syncthreads();
        u64 sig = 0, small = ~0ull;
        int32_t mf = 0;
#pragma unroll 1
        for (int32_t k0 = 0; k0 < vr.z; k0 += kU * blockDim.x) {
            int32_t e[kU];
            int4 r[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int32_t k = k0 + u * blockDim.x + threadIdx.x;
                e[u] = k < vr.z ? entry_id(list[k]) : -1;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                r[u] = e[u] >= 0 ? erec[e[u]] : make_int4(0, 0, kGone, 0);
            __syncthreads();  // the chunk is read: the kept ones move to the front
            int32_t kept = 0;
#pragma unroll
            for (int u = 0; u < kU; ++u) kept += __popc(__ballot_sync(0xffffffffu, r[u].z != kGone));
            int32_t at = 0;
            if (c.lane == 0 && kept) at = atomicAdd(&sh->pos, kept);
            at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const bool keep = r[u].z != kGone;
                const unsigned b = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    sig |= sig_bit(e[u]);
                    mf = max(mf, r[u].z);
                    const u64 key = ((u64)(uint32_t)r[u].w << 32) | (uint32_t)e[u];
                    small = key < small ? key : small;
                    list[at + __popc(b & ((1u << c.lane) - 1u))] =
                        make_entry(e[u], r[u].z, r[u].w, fold_sig(rec_sig(r[u])));
                }
                at += __popc(b);
            }
            __syncthreads();
        }
        mf = __reduce_max_sync(0xffffffffu, mf);
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) {
            sig |= __shfl_xor_sync(0xffffffffu, sig, o);
            const u64 y = __shfl_xor_sync(0xffffffffu, small, o);
            small = y < small ? y : small;
        }
        if (c.lane == 0) {
            atomicMax(&sh->mf, mf);
            atomicOr(&sh->sig, sig);
            atomicMin(&sh->small, small);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            v.vrec[x] = make_rec(sh->sig, sh->pos, vr.w);
            const int32_t e0 = (int32_t)(uint32_t)sh->small;
            v.vaux[x] = make_int4(e0, sh->mf, sh->pos > 0 ? v.eptr[e0] : 0,
                                  (int32_t)(sh->small >> 32));
        }
        __syncthreads();
    }
}

// The vertex of key i in the row of hyperedge e?
__device__ __forceinline__ bool in_row(const View &v, int32_t e, uint32_t i) {
    const uint32_t *r = v.row + v.eptr[e];
    const int32_t len = v.erec[e].w;
    const int32_t at = find_key(r, len, i);
    return at < len && r[at] == i;
}

// Can vertex i dominate j, by degree, signature and tie-break?
__device__ __forceinline__ bool may_dominate(int32_t i, int4 ri, int32_t j, int4 rj) {
    if (i == j || ri.z < rj.z) return false;
    if (rec_sig(rj) & ~rec_sig(ri)) return false;
    return ri.z > rj.z || i < j;  // equal degrees: contained means equal, the lower index dominates
}

// Delete vertex j (lane `sub` of `step` lanes): its hyperedges are the next
// round's candidates.
__device__ __forceinline__ void delete_vertex(Shared *sh, int32_t j, int4 rj, int32_t sub,
                                              int32_t step) {
    const View &v = sh->view;
    if (sub == 0) {
        v.v_o2c[j] = -1;
        atomicAdd(&sh->del2, 1);
    }
    const int32_t next = sh->epoch + 1;
#pragma unroll 1
    for (int32_t q = sub; q < rj.z; q += step) v.estamp[entry_id(v.vedge[rj.w + q])] = next;
}

// The test of vertex j (below), by the whole CTA: of high degree, or left by a group.
__device__ __noinline__ void md_whole(int32_t j, bool count) {
    const Ctx c;
    Shared *sh = c.sh;
    const View &v = sh->view;
    const int4 rj = v.vrec[j], aux = v.vaux[j];
    const int32_t e0 = aux.x, len0 = rj.z > 0 ? aux.w : 0;
    if (rj.z > 0 && !count && len0 - 1 < aux.y) return;
    const uint32_t *row = v.row + aux.z;
    const u64 *list = v.vedge + rj.w;
    if (threadIdx.x == 0) sh->pos = 0;
    __syncthreads();
    // one member per warp, 32 hyperedges at a time
#pragma unroll 1
    for (int32_t k = c.warp; k < len0; k += blockDim.x >> 5) {
        const uint32_t i = row[k];
        bool ok = may_dominate(key_id(i), v.vrec[key_id(i)], j, rj);  // (all lanes alike)
#pragma unroll 1
        for (int32_t q0 = 0; q0 < rj.z && ok; q0 += 32) {
            const int32_t q = q0 + c.lane;
            const int32_t e = q < rj.z ? entry_id(list[q]) : e0;
            const bool in = e == e0 || in_row(v, e, i);
            __syncwarp();
            ok = !__any_sync(0xffffffffu, !in);
        }
        if (ok && c.lane == 0) atomicAdd(&sh->pos, 1);
        __syncwarp();
        const bool decided = !count && vload(&sh->pos) >= aux.y;
        if (__any_sync(0xffffffffu, decided)) break;
    }
    __syncthreads();
    const int32_t cnt = sh->pos;
    __syncthreads();  // (reset for the next)
    if (count) {
        if (threadIdx.x == 0) sh->s->v_cnt[j] = cnt;
    } else if (rj.z == 0 || cnt >= aux.y) {
        delete_vertex(sh, j, rj, threadIdx.x, blockDim.x);
    }
}

// A group gives up a vertex after so many hyperedges looked at by a lane, if the
// list of such vertices has room: whole CTAs take them, 32 hyperedges of a member
// at a time.  (Every vertex in all hyperedges but one, 250 of each, beside 4,000
// small ones, load and kernelization: 5.3 ms by groups alone, which look through
// half of them for every member; 0.92 so, 1.17 by the contraction.)
constexpr int32_t kMdBudget = 96;
__device__ __noinline__ bool leave_to_cta(bool want, int32_t j) {
    const Ctx c;
    int32_t at = c.sh->task_cap;
    if (want && c.sub == 0) {
        at = atomicAdd(&c.sh->view.ctl->c[c.par].nbig, 1);
        if (at < c.sh->task_cap) c.sh->task[at] = make_int4(j, 0, 0, 0);
    }
    return __shfl_sync(0xffffffffu, at, c.lead) < c.sh->task_cap;
}

// The dominators of the candidates (count: into v_cnt; else a vertex with
// at least as many as its largest demand is deleted, and its hyperedges
// become the next round's candidates).
__device__ __noinline__ void md_test(bool count, int shard, int nshards) {
    const Ctx c;
    Shared *sh = c.sh;
    const View &v = sh->view;
    const int4 *const vrec = v.vrec;
    int32_t *const v_cnt = sh->s->v_cnt;
    for_flagged(
        c, sh->n0,
        [&](int32_t x) {
            return vertex_candidate(c, v, x) && !(v.agg[x].heavy & 1) &&
                   (!count || nshards == 1 || (x >> 7) % nshards == shard);
        },
        [&](int32_t j) {
            const int4 rj = j >= 0 ? vrec[j] : make_int4(0, 0, 0, 0);
            const int4 aux = j >= 0 ? v.vaux[j] : make_int4(0, 0, 0, 0);
            const int32_t e0 = aux.x;
            int32_t len0 = rj.z > 0 ? aux.w : 0;
            if (!count && len0 - 1 < aux.y) len0 = 0;  // too few members to dominate
            const uint32_t *row = v.row + aux.z;
            const u64 *list = v.vedge + rj.w;
            int32_t cnt = 0, spent = 0;
            bool mine = j >= 0;
            const int32_t maxlen = __reduce_max_sync(0xffffffffu, len0);
#pragma unroll 1
            for (int32_t k = c.sub; k - c.sub < maxlen; k += kG) {
                const uint32_t i = k < len0 ? row[k] : 0;
                bool ok = k < len0 && may_dominate(key_id(i), vrec[key_id(i)], j, rj);
#pragma unroll 1
                for (int32_t q = 0; q < rj.z && ok; ++q) {
                    const int32_t e = entry_id(list[q]);
                    ok = e == e0 || in_row(v, e, i);
                    ++spent;
                }
                __syncwarp();
                cnt += __popc(group_ballot(c, ok));
                if (!count && cnt >= aux.y) len0 = 0;  // decided
                const bool more = k - c.sub + kG < len0;
                if (!__any_sync(0xffffffffu, more)) break;
                const unsigned far = group_ballot(c, spent > kMdBudget);
                const bool big = more && !count && far;
                if (__any_sync(0xffffffffu, big)) {
                    const bool left = leave_to_cta(big, j);
                    if (big && left) {
                        mine = false;
                        len0 = 0;
                    } else if (big) {
                        spent = INT32_MIN / 2;  // (no room: go on)
                    }
                }
            }
            if (mine) {
                if (count) {
                    if (c.sub == 0) v_cnt[j] = cnt;
                } else if (rj.z == 0 || cnt >= aux.y) {
                    delete_vertex(sh, j, rj, c.sub, kG);
                }
            }
            __syncwarp();
        });
    const int32_t nh = vload(&v.ctl->n_heavy);
#pragma unroll 1
    for (int32_t h = sh->rank; h < nh; h += sh->size) {
        const int32_t j = sh->heavy[h];
        const bool mine = vertex_candidate(c, v, j) &&
                          (!count || nshards == 1 || (j >> 7) % nshards == shard);
        __syncthreads();  // (v_o2c[j] is written below)
        if (!mine) continue;
        md_whole(j, count);
    }
}

// The vertices whose groups gave up.
__device__ __noinline__ void md_big() {
    const Shared *sh = shared();
    const int32_t nb = min(sh->got.nbig, sh->task_cap);
#pragma unroll 1
    for (int32_t t = sh->rank; t < nb; t += sh->size) md_whole(sh->task[t].x, false);
}

// Sharded passes: the decision from the (merged) counts.
__device__ __noinline__ void md_decide() {
    const Ctx c;
    const View &v = c.sh->view;
    const int32_t *const v_cnt = c.sh->s->v_cnt;
    for_flagged(
        c, c.sh->n0, [&](int32_t x) { return vertex_candidate(c, v, x); },
        [&](int32_t j) {
            if (j >= 0) {
                const int4 rj = v.vrec[j];
                if (rj.z == 0 || v_cnt[j] >= v.vaux[j].y) delete_vertex(c.sh, j, rj, c.sub, kG);
            }
            __syncwarp();
        });
}

// ---------------------------------------------------------------- rule FE --

// Full hyperedges go, their vertices into the solution.
__device__ __noinline__ void fe_mark() {
    const Ctx c;
    const View &v = c.sh->view;
    uint8_t *const forced = c.sh->s->forced;
    for_flagged(
        c, c.sh->m0, [&](int32_t e) { return v.e_o2c[e] >= 0; },
        [&](int32_t e) {
            const int4 r = e >= 0 ? v.erec[e] : make_int4(0, 0, 0, -1);
            __syncwarp();  // read by every lane before it is written
            if (r.w == r.z) {
                const uint32_t *row = v.row + v.eptr[e];
#pragma unroll 1
                for (int32_t k = c.sub; k < r.w; k += kG) {
                    const int32_t x = key_id(row[k]);
                    if (atomicExch(&v.v_o2c[x], -1) >= 0) {
                        forced[x] = 1;
                        atomicAdd(&c.sh->del2, 1);
                    }
                }
                if (c.sub == 0) {
                    v.erec[e].z = kGone;
                    v.e_o2c[e] = -1;
                    atomicOr(&v.gone[e >> 5], 1u << (e & 31));
                    atomicAdd(&c.sh->del, 1);
                }
            }
            __syncwarp();
        });
}

// The others lose one unit of demand per vertex taken; the bounds restart.
__device__ __noinline__ void fe_apply() {
    const Ctx c;
    const View &v = c.sh->view;
    int32_t *const f = c.sh->s->f;
    for_flagged(
        c, c.sh->m0, [&](int32_t e) { return v.e_o2c[e] >= 0; },
        [&](int32_t e) {
            const int4 r = e >= 0 ? v.erec[e] : make_int4(0, 0, 0, 0);
            const uint32_t *row = e >= 0 ? v.row + v.eptr[e] : nullptr;
            int32_t lost = 0;
#pragma unroll 1
            for (int32_t k = c.sub; k < r.w; k += kG) lost += v.v_o2c[key_id(row[k])] < 0;
            __syncwarp();
            lost = group_sum(lost);
            if (lost > 0 && c.sub == 0) {
                const int32_t left = r.z - lost;
                f[e] = left;
                v.erec[e].z = left > 0 ? left : kGone;
                if (left <= 0) {
                    v.e_o2c[e] = -1;
                    atomicOr(&v.gone[e >> 5], 1u << (e & 31));
                    atomicAdd(&c.sh->del, 1);
                }
            }
            __syncwarp();
        });
    const int32_t t0 = c.sh->rank * blockDim.x + threadIdx.x, ts = c.sh->size * blockDim.x;
#pragma unroll 1
    for (int32_t x = t0; x < c.sh->n0; x += ts) {
        v.agg[x].m1 = 0;
        v.bound[x] = 0;
        v.agg[x].heavy &= 1;
        v.agg[x].s1 = 0;
    }
#pragma unroll 1
    for (uint32_t q = t0; q <= c.sh->pair_mask; q += ts) c.sh->pair_tab[q] = SpPair{};
    if (t0 == 0) {
        v.ctl->loose = 0;
        v.ctl->empty = 0;
        v.ctl->pairs_full = 0;
    }
}

// ------------------------------------------------------------------ build --

// 256 counters of a warp become the first places of their classes.
__device__ __forceinline__ void first_places(int32_t *at, int lane) {
    constexpr int kPer = 256 / 32;
    int32_t sum = 0;
#pragma unroll 1
    for (int c = 0; c < kPer; ++c) sum += at[lane * kPer + c];
    int32_t inc = sum;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    int32_t first = inc - sum;
    __syncwarp();
#pragma unroll 1
    for (int c = 0; c < kPer; ++c) {
        const int32_t n = at[lane * kPer + c];
        at[lane * kPer + c] = first;
        first += n;
    }
    __syncwarp();
}

// Rows that are not strictly ascending: up to kRankRow ids their eight lanes rank
// each id by counting, up to kSortRow the warp sorts them by bytes of the id, and
// with a longer one the load leaves this path (kLeave), as for one that does not
// pay.  One such row among 20,000 of 10 ids over 40,000 vertices, load and
// kernelization (us), all by counting / so / by the contraction:
//   2,000 ids  21,035 / 640 / 21,237     32,768 ids  (not run) / 3,944 / 21,472
// 10,000 ids among 300 rows over 10,000 vertices: 1,196 / 1,225 by the contraction.
constexpr int32_t kRankRow = 64;
constexpr int32_t kSortRow = 65536;
constexpr int32_t kLeave = 1 << 30;  // (of the status, beside the kErr* bits)
constexpr int32_t kLongRow = 1 << 29;
constexpr int32_t kInOrder = -1;

// A row of more than kRankRow ids, by the warp: kInOrder if `in` ascends, else
// its ids in order, without repeats, into row, and their number (ids outside
// [0, n0) may come out anywhere; one of each remains).  Too long for that:
// kLeave, and kErrBadVertex if it has such an id.
__device__ __noinline__ int32_t long_row(const int32_t *in, int32_t *tmp, int32_t *row, int32_t len,
                                         int32_t n0) {
    const int lane = threadIdx.x & 31;
    int32_t back = 0, out = 0;  // entries not below their right neighbour; outside
#pragma unroll 4
    for (int32_t k = lane; k < len; k += 32) {
        const int32_t x = in[k];
        back |= k + 1 < len && x >= in[k + 1 < len ? k + 1 : k];
        out |= x < 0 || x >= n0;
    }
    if (!__any_sync(0xffffffffu, back)) return kInOrder;
    if (len > kSortRow) return kLeave | (__any_sync(0xffffffffu, out) ? kErrBadVertex : 0);
    int32_t *const at = reinterpret_cast<int32_t *>(warp_shared()->buf);
    constexpr int kAhead = 4;  // loads in flight
    const int passes = n0 <= 1 << 8 ? 1 : n0 <= 1 << 16 ? 2 : 3;
    const int32_t *from = in;
    int32_t *to = passes == 2 ? tmp : row;
#pragma unroll 1
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        for (int c = lane; c < 256; c += 32) at[c] = 0;
        __syncwarp();
#pragma unroll 4
        for (int32_t k = lane; k < len; k += 32) atomicAdd(&at[((uint32_t)from[k] >> shift) & 255u], 1);
        __syncwarp();
        first_places(at, lane);
#pragma unroll 1
        for (int32_t k0 = 0; k0 < len; k0 += kAhead * 32) {
            int32_t x[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int32_t k = k0 + u * 32 + lane;
                x[u] = k < len ? from[k] : 0;
            }
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const bool on = k0 + u * 32 + lane < len;
                const uint32_t digit = on ? ((uint32_t)x[u] >> shift) & 255u : 256u;
                const unsigned peers = __match_any_sync(0xffffffffu, digit);
                const int32_t q = on ? at[digit] + __popc(peers & ((1u << lane) - 1u)) : 0;
                __syncwarp();
                if (on) {
                    if (lane == 31 - __clz(peers)) at[digit] = q + 1;
                    to[q] = x[u];
                }
                __syncwarp();
            }
        }
        from = to;
        to = to == row ? tmp : row;
    }
    int32_t w = 0;
#pragma unroll 1
    for (int32_t k0 = 0; k0 < len; k0 += 32) {
        const int32_t k = k0 + lane;
        const int32_t x = k < len ? row[k] : 0;
        const bool keep = k < len && (k == 0 || row[k - 1] != x);
        const unsigned mk = __ballot_sync(0xffffffffu, keep);  // (read before it is written)
        if (keep) row[w + __popc(mk & ((1u << lane) - 1u))] = x;
        w += __popc(mk);
        __syncwarp();
    }
    return w;
}

// Hyperedge e of the input: its checks, the vertices' degrees and the
// incidences' places in their lists.  A row that is not strictly ascending is
// sorted, without repeats, into v.row (its ids; noted in the record).
// Rows above kRankRow are left to count_long_rows (kLongRow).  Returns the error
// bits found.  The whole warp.
__device__ __forceinline__ int32_t count_row(const Ctx &c, const View &v, const int32_t *evtx,
                                             const int32_t *f, int32_t *place, int32_t *local,
                                             int32_t n0, int64_t nnz0, int32_t e) {
    int32_t p0 = 0, len = 0, fe = 1, bad = 0;
    if (e >= 0) {
        p0 = v.eptr[e];
        len = v.eptr[e + 1] - p0;
        fe = f[e];
        if (fe < 1) bad |= kErrBadDemand;
        if (fe > kFewMisses) c.sh->demands = 1;
        if (p0 < 0 || len < 0 || (int64_t)p0 + len > nnz0) { bad |= kErrBadPtr; len = 0; }
        if (len > kRankRow) { bad |= kLongRow; len = 0; }
    }
    const int32_t *in = evtx + p0;
    int32_t *row = reinterpret_cast<int32_t *>(v.row) + p0;
    const int32_t maxlen = __reduce_max_sync(0xffffffffu, len);
    // first the entries, in order? (each against its right neighbour)
    bool asc = true;
#pragma unroll 1
    for (int32_t k = c.sub; k + 1 < len; k += kG) asc = asc && in[k] < in[k + 1];
    __syncwarp();
    const bool sorted = group_ballot(c, !asc) == 0;
    if (__any_sync(0xffffffffu, !sorted)) {
        // rank sort (ties by place), then drop repeats
        if (!sorted)
#pragma unroll 1
            for (int32_t k = c.sub; k < len; k += kG) {
                const int32_t y = in[k];
                int32_t rank = 0;
#pragma unroll 1
                for (int32_t l = 0; l < len; ++l) rank += in[l] < y || (in[l] == y && l < k);
                row[rank] = y;
            }
        __syncwarp();
        int32_t w = len;
        if (!sorted && c.sub == 0) {
            int32_t last = row[0];
            w = 1;
#pragma unroll 1
            for (int32_t k = 1; k < len; ++k) {
                const int32_t y = row[k];
                if (y != last) row[w++] = y;
                last = y;
            }
        }
        len = __shfl_sync(0xffffffffu, w, c.lead);
        __syncwarp();
    }
    const int32_t *ids = sorted ? in : row;
#pragma unroll 1
    for (int32_t k0 = 0; k0 < maxlen; k0 += kRowU * kG) {
        int32_t x[kRowU], at[kRowU];
#pragma unroll
        for (int u = 0; u < kRowU; ++u) {
            const int32_t k = k0 + u * kG + c.sub;
            x[u] = k < len ? ids[k] : 0;
        }
        // (the atomics of a batch are under way together)
#pragma unroll
        for (int u = 0; u < kRowU; ++u) {
            const bool on = k0 + u * kG + c.sub < len;
            const bool ok = x[u] >= 0 && x[u] < n0;
            if (on && !ok) bad |= kErrBadVertex;
            at[u] = !on || !ok ? 0 : atomicAdd(local ? &local[x[u]] : &v.vrec[x[u]].z, 1);
        }
#pragma unroll
        for (int u = 0; u < kRowU; ++u)
            if (k0 + u * kG + c.sub < len) place[p0 + k0 + u * kG + c.sub] = at[u];
    }
    if (e >= 0 && c.sub == 0) v.erec[e] = make_int4(sorted ? 0 : 1, 0, fe, len);
    return bad;
}

// The degrees of a CTA's instance in shared memory, or null.
__device__ __forceinline__ int32_t *local_table(const Shared *sh) {
    return sh->local && sh->n0 <= kLocalVertices ? local_degrees() : nullptr;
}

// The same for the rows above kRankRow, a warp for each, after the others.
__device__ __noinline__ int32_t count_long_rows() {
    const Ctx c;
    const View &v = c.sh->view;
    const InstState &s = *c.sh->s;
    const int32_t *const evtx = s.evtx, *const f = s.f;
    int32_t *const place = s.sp_pos;
    uint32_t *const tmp = s.sp_tmp;
    const int32_t n0 = c.sh->n0, m0 = c.sh->m0;
    const int64_t nnz0 = s.nnz0;
    int32_t *const local = local_table(c.sh);
    int32_t bad = 0, chunk = 32;  // the ids that for_flagged gives this warp
    while (chunk > 32 / kG && (int64_t)m0 < (int64_t)c.nw * chunk) chunk >>= 1;
#pragma unroll 1
    for (int64_t base = (int64_t)c.gw * chunk; base < m0; base += (int64_t)c.nw * chunk) {
        const int32_t e0 = (int32_t)base + c.lane;
        int32_t p0 = 0, len = 0;
        if (c.lane < chunk && e0 < m0) {
            p0 = v.eptr[e0];
            len = v.eptr[e0 + 1] - p0;
            if (p0 < 0 || len < 0 || (int64_t)p0 + len > nnz0) len = 0;
        }
        unsigned longs = __ballot_sync(0xffffffffu, len > kRankRow);
#pragma unroll 1
        while (longs) {
            const int l = __ffs(longs) - 1;
            longs &= longs - 1;
            const int32_t e = (int32_t)base + l, p = __shfl_sync(0xffffffffu, p0, l);
            int32_t n = __shfl_sync(0xffffffffu, len, l);
            int32_t *const row = reinterpret_cast<int32_t *>(v.row) + p;
            const int32_t got = long_row(evtx + p, reinterpret_cast<int32_t *>(tmp) + p, row, n, n0);
            if (got != kInOrder && (got & kLeave)) {
                bad |= got;
                continue;
            }
            if (got != kInOrder) n = got;
            const int32_t *const ids = got == kInOrder ? evtx + p : row;
#pragma unroll 2
            for (int32_t k = c.lane; k < n; k += 32) {
                const int32_t x = ids[k];
                const bool ok = x >= 0 && x < n0;
                if (!ok) bad |= kErrBadVertex;
                place[p + k] = ok ? atomicAdd(local ? &local[x] : &v.vrec[x].z, 1) : 0;
            }
            if (c.lane == 0) v.erec[e] = make_int4(got == kInOrder ? 0 : 1, 0, f[e], n);
            __syncwarp();
        }
    }
    return bad;
}

// The row of hyperedge e in key order, and its entries in its vertices'
// lists, by kW lanes (8 or 32; `lane` of them)
// that hold the row (len <= kRowU * kW) in registers and rank each key by
// counting.  Adds to *cost the lengths of the lists of its np rarest
// vertices; returns the signature.  The whole warp calls it.
template <int kW>
__device__ __forceinline__ u64 fill_row(const Ctx &c, const View &v, const int32_t *local,
                                        const int32_t *ids, const int32_t *place, uint32_t *row,
                                        int32_t e, int32_t f, int32_t len, int32_t np, int lane,
                                        u64 *cost) {
    const int32_t maxlen = kW == 32 ? len : __reduce_max_sync(0xffffffffu, len);
    uint32_t key[kRowU];
    int32_t at[kRowU], deg[kRowU], rank[kRowU];
    u64 sig = 0;
#pragma unroll
    for (int u = 0; u < kRowU; ++u) {
        const int32_t k = u * kW + lane;
        const int32_t x = k < len ? ids[k] : -1;
        int2 vr = make_int2(0, 0);  // degree, place of the list
        if (x >= 0)
            vr = local ? make_int2(local[x], local[kLocalVertices + x])
                       : *reinterpret_cast<const int2 *>(&v.vrec[x].z);
        key[u] = x >= 0 ? row_key(x, vr.x) : 0xffffffffu;
        at[u] = x >= 0 ? vr.y + place[k] : 0;
        deg[u] = vr.x;
        rank[u] = 0;
        if (x >= 0) sig |= sig_bit(x);
    }
    sig = group_or(sig);
    if (kW == 32) {
        sig |= __shfl_xor_sync(0xffffffffu, sig, 8);
        sig |= __shfl_xor_sync(0xffffffffu, sig, 16);
    }
#pragma unroll
    for (int w = 0; w < kRowU; ++w) {
        // (eight lanes: without loop control.  A batch is bound by what its
        // warps issue; this and the sum of costs kept in registers take 0.3
        // of its load's 2.8 ms)
        if (kW == kG) {
            if (w * kW >= maxlen) break;
#pragma unroll
            for (int l = 0; l < kW; ++l) {
                const uint32_t y = __shfl_sync(0xffffffffu, key[w], l, kW);
#pragma unroll
                for (int u = 0; u < kRowU; ++u) rank[u] += y < key[u];
            }
            continue;
        }
        const int32_t n = min(kW, maxlen - w * kW);
#pragma unroll 1
        for (int l = 0; l < n; ++l) {
            const uint32_t y = __shfl_sync(0xffffffffu, key[w], l);
#pragma unroll
            for (int u = 0; u < kRowU; ++u) rank[u] += y < key[u];
        }
    }
    __syncwarp();  // (ids may lie where the row goes)
    const uint32_t fold = fold_sig(sig);
#pragma unroll
    for (int u = 0; u < kRowU; ++u) {
        if (u * kW + lane >= len) continue;
        row[rank[u]] = key[u];
        v.vedge[at[u]] = make_entry(e, f, len, fold);
        if (rank[u] < np) *cost += (uint32_t)deg[u];
    }
    return sig;
}

// The same for any length, by the warp: a counting sort of the keys by their
// degree class, in order inside a class (ids ascend).  place becomes the
// entries' places in the lists.  (Gathering class by class cost a scan of the
// row per class, and the longest row of an instance is what its load waits for:
// intervals of 64 over 2,000 x 4,000, 137 us; 115 now.  Few registers: with
// twice the loads in flight the batch's rows, which never come here, spill, 2.46
// -> 2.60 ms.)
__device__ __noinline__ u64 fill_long_row(const int32_t *ids, int32_t *place, uint32_t *tmp,
                                          uint32_t *row, int32_t e, int32_t f, int32_t len,
                                          int32_t np, u64 *cost) {
    constexpr int kClasses = 256, kPer = kClasses / 32;
    static_assert(sizeof(WarpShared::buf) >= kClasses * sizeof(int32_t), "a counter per class");
    const View &v = shared()->view;
    const int lane = threadIdx.x & 31;
    int32_t *const at = reinterpret_cast<int32_t *>(warp_shared()->buf);
#pragma unroll
    for (int c = 0; c < kPer; ++c) at[c * 32 + lane] = 0;
    __syncwarp();
    u64 sig = 0;
#pragma unroll 2
    for (int32_t k = lane; k < len; k += 32) {
        const int32_t x = ids[k];
        const int4 vr = v.vrec[x];
        const uint32_t key = row_key(x, vr.z);
        tmp[k] = key;
        place[k] += vr.w;
        sig |= sig_bit(x);
        atomicAdd(&at[key >> 24], 1);
    }
    __syncwarp();
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) sig |= __shfl_xor_sync(0xffffffffu, sig, o);
    const u64 entry = make_entry(e, f, len, fold_sig(sig));
    first_places(at, lane);
#pragma unroll 1
    for (int32_t k0 = 0; k0 < len; k0 += 32) {
        const int32_t k = k0 + lane;
        const uint32_t key = k < len ? tmp[k] : 0xffffffffu;  // (class 255 cannot occur)
        const unsigned peers = __match_any_sync(0xffffffffu, key >> 24);
        const int32_t to = k < len ? at[key >> 24] + __popc(peers & ((1u << lane) - 1u)) : 0;
        __syncwarp();
        if (k < len) {
            if (lane == 31 - __clz(peers)) at[key >> 24] = to + 1;
            row[to] = key;
            v.vedge[place[k]] = entry;
            if (to < np) *cost += (uint32_t)v.vrec[key_id(key)].z;
        }
        __syncwarp();
    }
    return sig;
}

// ------------------------------------------------------------ round driver --

// Add this CTA's deletions of a phase to the instance's counter.
__device__ __forceinline__ void flush(int32_t *sh_ctr, int32_t *to) {
    __syncthreads();
    if (threadIdx.x == 0) {
        if (*sh_ctr) atomicAdd(to, *sh_ctr);
        *sh_ctr = 0;
    }
}

// Shared memory for one instance.
__device__ __noinline__ void start(InstState *s, int rank, int size, uint64_t absent_ns,
                                   bool local = false) {
    Shared *sh = shared();
    if (threadIdx.x == 0) {
        sh->view = View(*s);
        sh->s = s;
        sh->heavy = s->sp_heavy;
        sh->pair_tab = s->sp_pair_tab;
        sh->pair_mask = s->sp_pair_mask;
        sh->task = s->sp_task;
        sh->task_cap = s->sp_task_cap;
        sh->n0 = s->n0;
        sh->m0 = s->m0;
        sh->rule = s->edge_rule;
        sh->rank = rank;
        sh->local = local;
        const int32_t twice = 2 * (int32_t)min(s->nnz0 / max(s->n0, 1), (int64_t)1 << 29);
        sh->heavy_list = max(kHeavyList, min(twice, 4 * kHeavyList));
        sh->task_len = max(kTaskLen, min(twice, 4 * kTaskLen));
        sh->size = size;
        sh->absent = absent_ns != 0;
        sh->wait_ns = absent_ns ? absent_ns : kTeamWaitNs;
        sh->epoch = 1;
        sh->par = 0;
        sh->full = 1;
        sh->del = sh->del2 = 0;
        sh->cost = sh->open = 0;
        sh->demands = 0;
        sh->pairs = s->sp_pairs;
        sh->pair_cap = s->sp_pair_cap;
        sh->bar = &s->sp_ctl->bar;
        // no barrier can complete without this CTA, so the arrivals seen
        // beyond a multiple of the team's size are this launch's first
        const uint32_t now = *reinterpret_cast<volatile uint32_t *>(sh->bar);
        sh->target = now / (uint32_t)size * (uint32_t)size;
    }
    __syncthreads();
}

// What the walks of the hyperedges with demands above kFewMisses count as open
// (rows and degrees are in place).  Apart from the fill, whose loop keeps fewer
// registers with it (the batch of 4,096: 2.52 ms instead of 2.47).
__device__ __noinline__ void open_walks() {
    const Ctx c;
    Shared *sh = c.sh;
    const View &v = sh->view;
    if (sh->rule) return;
    const int32_t *const f = sh->s->f;
    float open = 0.f;
    for_flagged(
        c, sh->m0, [&](int32_t e) { return f[e] > kFewMisses; },
        [&](int32_t e) {
            if (e >= 0) {
                const int4 r = v.erec[e];
                const int32_t np = walk_count(0, r.z, r.w);
                const uint32_t *row = v.row + v.eptr[e];
                float entries = 0.f;
#pragma unroll 1
                for (int32_t k = c.sub; k < np && np <= kManyLists; k += kG)
                    entries += (float)v.vrec[key_id(row[k])].z;
                open += open_walk(entries, r.z, r.w);
                if (np > kManyLists && c.sub == 0) open += kPerListSquared * (float)np * (float)np;
            }
            __syncwarp();
        });
    if (open > 0.f) atomicAdd(&sh->open, (u64)open);
}

// Structural checks, rows and lists of one instance; !kLong: if it has no row above
// kRankRow (else its status says kLongRow).  False if a barrier timed out.
template <bool kLong>
__device__ __noinline__ bool build_instance(int32_t max_rounds, SpTotals *out) {
    const Ctx c;
    InstState &s = *c.sh->s;
    const View v = c.sh->view;
    const int32_t n0 = s.n0, m0 = s.m0;
    const int64_t nnz0 = s.nnz0;
    const int32_t *const evtx = s.evtx;
    const int32_t *const f = s.f;
    int32_t *const place = s.sp_pos;
    uint32_t *const tmp = s.sp_tmp;
    const int32_t t0 = c.sh->rank * blockDim.x + threadIdx.x, ts = c.sh->size * blockDim.x;
    int32_t *const local = local_table(c.sh);
    if (local) {
#pragma unroll 1
        for (int32_t x = threadIdx.x; x < n0; x += blockDim.x) local[x] = 0;
        __syncthreads();
    }
    if (t0 == 0) {
        s.n = s.n0; s.m = s.m0; s.m_dp = s.m0; s.n_next = s.n0;
        s.rounds = 0; s.active = 1; s.max_rounds = max_rounds; s.changed = 0;
        s.dp_deleted = 0; s.md_deleted = 0; s.fe_stage = 0; s.fe_passes = 0;
        v.ctl->full = 1;
        if (s.eptr[0] != 0 || (int64_t)s.eptr[s.m0] != s.nnz0) atomicOr(&s.status, kErrBadPtr);
    }
    // (the records, bounds and stamps are zero: cleared with the control words)
    int32_t bad = 0;
    uint8_t *const forced = s.forced;
#pragma unroll 1
    for (int32_t x = t0; x < n0; x += ts) {
        v.v_o2c[x] = x;
        if (forced) forced[x] = 0;
    }
#pragma unroll 1
    for (int32_t e = t0; e < m0; e += ts) v.e_o2c[e] = e;
    for_flagged(
        c, m0, [](int32_t) { return true; },
        [&](int32_t e) { bad |= count_row(c, v, evtx, f, place, local, n0, nnz0, e); });
    if (kLong && __any_sync(0xffffffffu, bad & kLongRow))
        bad = (bad & ~kLongRow) | count_long_rows();
    if (bad) atomicOr(&s.status, bad);
    if (!team_sync()) return false;
    if (const int32_t st = vload(&s.status)) {
        if (t0 == 0 && !(st & kLongRow)) {
            if (st == kLeave) out->leave = 1;
            else atomicOr(&out->status, st & ~kLeave);
        }
        return true;
    }
    // a place for every vertex's list (in any order): one atomic per warp
    int32_t *const heavy = s.sp_heavy;
#pragma unroll 1
    for (int32_t x0 = t0 - c.lane; x0 < n0; x0 += ts) {
        const int32_t x = x0 + c.lane;
        const int32_t d = x >= n0 ? 0 : local ? local[x] : v.vrec[x].z;
        int32_t inc = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (c.lane >= o) inc += y;
        }
        int32_t at = 0;
        if (c.lane == 31) at = (int32_t)atomicAdd(&v.ctl->cursor, (uint32_t)inc);
        at = __shfl_sync(0xffffffffu, at, 31);
        if (x < n0) {
            v.vrec[x] = make_int4(0, 0, d, at + inc - d);
            if (local) local[kLocalVertices + x] = at + inc - d;
        }
        if (d > kHeavyDeg) {
            v.agg[x].heavy = 1;
            heavy[atomicAdd(&v.ctl->n_heavy, 1)] = x;
        }
    }
    if (!team_sync()) return false;
    const int32_t rule = s.edge_rule;
    u64 cost = 0;  // the entries that walking this lane's hyperedges may visit
    for_flagged(
        c, m0, [](int32_t) { return true; },
        [&](int32_t e) {
            const int4 r = e >= 0 ? v.erec[e] : make_int4(0, 0, 0, 0);
            const int32_t p0 = e >= 0 ? v.eptr[e] : 0, len = r.w;
            const int32_t *ids = r.x ? reinterpret_cast<const int32_t *>(v.row) + p0 : evtx + p0;
            uint32_t *row = v.row + p0;
            const int32_t np = e >= 0 ? walk_count(rule, r.z, len) : 0;
            u64 sig = 0;
            // rows up to 16: the group ranks each key among the row's
            const bool small = len <= kRowU * kG;
            if (__any_sync(0xffffffffu, small && len > 0)) {
                sig = fill_row<kG>(c, v, local, ids, place + p0, row, e, r.z, small ? len : 0, np, c.sub,
                                   &cost);
                if (small && c.sub == 0 && e >= 0) v.erec[e] = make_rec(sig, r.z, len);
            }
            // longer ones, one after the other: the whole warp
            unsigned longs = __ballot_sync(0xffffffffu, !small && c.sub == 0);
#pragma unroll 1
            while (longs) {
                const int l = __ffs(longs) - 1;
                longs &= longs - 1;
                const int32_t le = __shfl_sync(0xffffffffu, e, l);
                const int32_t lp = __shfl_sync(0xffffffffu, p0, l);
                const int32_t llen = __shfl_sync(0xffffffffu, len, l);
                const int32_t lf = __shfl_sync(0xffffffffu, r.z, l);
                const int32_t lnp = __shfl_sync(0xffffffffu, np, l);
                const bool sorted = __shfl_sync(0xffffffffu, r.x, l) == 0;
                const int32_t *lids =
                    sorted ? evtx + lp : reinterpret_cast<const int32_t *>(v.row) + lp;
                u64 ls;
                if (llen <= kRowU * 32)
                    ls = fill_row<32>(c, v, local, lids, place + lp, v.row + lp, le, lf, llen, lnp, c.lane,
                                      &cost);
                else
                    ls = fill_long_row(lids, place + lp, tmp + lp, v.row + lp, le, lf, llen, lnp, &cost);
                if (c.lane == 0) v.erec[le] = make_rec(ls, lf, llen);
                __syncwarp();
            }
            cost += (u64)(uint32_t)(c.sub == 0 ? np : 0);
            __syncwarp();
            if (e >= 0) contribute(e, r.z, len, row);
            __syncwarp();
        });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cost += __shfl_xor_sync(0xffffffffu, cost, o);
    if (c.lane == 0 && cost) atomicAdd(&c.sh->cost, cost);
    if (c.sh->demands) open_walks();
    __syncthreads();
    if (threadIdx.x == 0 && c.sh->cost) atomicAdd(&out->cost, c.sh->cost);
    if (threadIdx.x == 0 && c.sh->open) atomicAdd(&out->open, c.sh->open);
    return true;
}

// A batch's instance with a row above kRankRow: the build anew.  (A branch of its
// own: with a call more in it, the function that builds most instances keeps less
// in registers, and the batch of 4,096 loads in 2.51 to 2.80 ms instead of 2.45.)
__device__ __noinline__ void build_again(int32_t max_rounds, SpTotals *out) {
    Shared *sh = shared();
    if (threadIdx.x == 0) sh->s->status = 0;
#pragma unroll 1
    for (int32_t x = threadIdx.x; x < sh->n0; x += blockDim.x) sh->view.vrec[x].z = 0;
    __syncthreads();
    build_instance<true>(max_rounds, out);
}

// Thread 0 of every CTA: the state at the start of a launch.
__device__ void load_progress(Progress &g, const InstState &s) {
    g.n = s.n; g.m = s.m; g.rounds = s.rounds; g.changed = s.changed;
    g.dp = s.dp_deleted; g.md = s.md_deleted; g.fe_passes = s.fe_passes;
    g.max_rounds = s.max_rounds; g.fe = s.full_edges; g.k = s.k;
    g.active = s.active && !s.status;
    g.full = s.sp_ctl->full;
    g.t_dp = g.t_md = 0;
    g.t_all = globaltimer();
}

// One thread of the team: the state at its end.
__device__ void store_progress(const Progress &g, InstState &s, BatchCounters *ctr) {
    s.n = g.n; s.n_next = g.n; s.m = g.m; s.m_dp = g.m; s.rounds = g.rounds;
    s.changed = g.changed; s.dp_deleted = g.dp; s.md_deleted = g.md;
    s.fe_passes = g.fe_passes; s.k = g.k; s.active = g.active;
    s.sp_ctl->full = g.full;
    if (!ctr) return;
    atomicAdd(&ctr->active, g.active);
    atomicAdd(&ctr->n_alive, g.n);
    atomicAdd(&ctr->m_alive, g.m);
    atomicAdd(&ctr->dp_deleted, g.dp);
    atomicAdd(&ctr->md_deleted, g.md);
    atomicMax(&ctr->max_rounds_seen, g.rounds);
    atomicOr(&ctr->changed_any, g.changed);
    atomicOr(&ctr->status_any, vload(&s.status));
}

__device__ __forceinline__ void begin_round() {
    Shared *sh = shared();
    if (threadIdx.x == 0) {
        sh->epoch = sh->g.rounds + 1;
        sh->par = sh->g.rounds & 1;
        sh->full = sh->g.full;
    }
    __syncthreads();
}

// The end of a round that deleted dp hyperedges and md vertices: the books,
// rule FE at a fixpoint, and whether there is more to do.  False if a
// barrier timed out.
__device__ __noinline__ bool finish_round(int32_t dp, int32_t md) {
    Shared *sh = shared();
    SpCtl *ctl = sh->view.ctl;
    Progress &g = sh->g;
    const bool fe = dp + md == 0 && g.fe && g.max_rounds == 0;
    __syncthreads();  // g is read above by every thread
    if (threadIdx.x == 0) {
        if (sh->rank == 0 && g.rounds < kTraceRounds) {
            int32_t *row = sh->s->trace[g.rounds];
            row[0] = g.m;
            row[1] = g.n;
            row[2] = g.m - dp;
        }
        g.dp = dp;
        g.md = md;
        g.m -= dp;
        g.n -= md;
        g.full = 0;
        g.changed = dp + md > 0;
        ++g.rounds;
        if (!fe && (!g.changed || (g.max_rounds > 0 && g.rounds >= g.max_rounds))) g.active = 0;
    }
    __syncthreads();
    if (!fe) return true;
    fe_mark();
    flush(&sh->del, &ctl->fe.dp);
    flush(&sh->del2, &ctl->fe.md);
    if (!team_sync()) return false;
    fe_apply();
    flush(&sh->del, &ctl->fe.dp);
    if (!team_sync(&ctl->fe)) return false;
    const int32_t de = sh->got.dp, dv = sh->got.md;
    if (!team_sync()) return false;  // every CTA has read them
    if (threadIdx.x == 0) {
        if (sh->rank == 0) ctl->fe = SpRound{};
        ++g.fe_passes;
        g.m -= de;
        g.n -= dv;
        g.k -= dv;
        // lowered demands make every hyperedge and vertex a candidate again
        if (de + dv > 0) g.full = g.changed = 1;
        else g.active = 0;
    }
    __syncthreads();
    return true;
}

// Rounds of Algorithm 3 (and FE at its fixpoints) until the fixpoint or
// `limit` rounds (0: no limit).  False if a barrier timed out.
__device__ __noinline__ bool run_instance(int32_t limit, BatchCounters *ctr, SpTimes *times) {
    Shared *sh = shared();
    if (threadIdx.x == 0) load_progress(sh->g, *sh->s);
    // one CTA must not publish the final state before all have read this one
    if (!team_sync()) return false;
    for (int32_t done = 0; sh->g.active && (limit <= 0 || done < limit); ++done) {
        begin_round();
        SpRound *rc = &sh->view.ctl->c[sh->par], *nx = &sh->view.ctl->c[sh->par ^ 1];
        const bool lead = sh->rank == 0 && threadIdx.x == 0;
        int32_t dp = 0, md = 0;
        if (sh->full || sh->g.md > 0) {
            if (sh->epoch > 1) {  // (the first round's rows are the load's)
                dp_rows();
                if (!team_sync()) return false;
                if (sh->full) {  // FE lowered demands, which the lists repeat
                    md_lists();
                    if (!team_sync()) return false;
                }
            }
            if (lead) sh->g.t_dp -= globaltimer();
            dp_bounds(0, 1);
            // full rounds: the walks skip what the bounds deleted (a matter of
            // time only: 40 M list entries become 14 M on the power-law instance)
            if (sh->full && !team_sync()) return false;
            dp_walk(0, 1);
            flush(&sh->del, &rc->dp);
            if (!team_sync(rc)) return false;
            // (each list has a counter that is final at the barrier before it is
            // read: the CTAs must agree on the barriers that follow)
            if (sh->got.npair[0] > 0) {
                decide_pairs(0);
                flush(&sh->del, &rc->dp);
                if (!team_sync(rc)) return false;
            }
            if (sh->got.ntask > 0) {  // (after the pairs: a hyperedge found deleted needs no walk)
                dp_tasks(0, 1);
                flush(&sh->del, &rc->dp);
                if (!team_sync(rc)) return false;
                if (sh->got.npair[1] > 0) {
                    decide_pairs(1);
                    flush(&sh->del, &rc->dp);
                    if (!team_sync(rc)) return false;
                }
            }
            if (lead) sh->g.t_dp += globaltimer();
            dp = sh->got.dp;
            // every CTA is past the previous round: its counters serve the next one
            if (lead) *nx = SpRound{};
            if (sh->full || dp > 0) {
                md_lists();
                if (!team_sync()) return false;
                if (lead) sh->g.t_md -= globaltimer();
                md_test(false, 0, 1);
                flush(&sh->del2, &rc->md);
                if (!team_sync(rc)) return false;
                if (sh->got.nbig > 0) {
                    md_big();
                    flush(&sh->del2, &rc->md);
                    if (!team_sync(rc)) return false;
                }
                if (lead) sh->g.t_md += globaltimer();
                md = sh->got.md;
            }
        } else if (lead) {
            // no hyperedge lost a vertex: both passes are empty.  (The last
            // round's md is 0, so resetting its counters loses nothing.)
            *nx = SpRound{};
        }
        if (!finish_round(dp, md)) return false;
    }
    if (sh->rank == 0 && threadIdx.x == 0) {
        const Progress &g = sh->g;
        store_progress(g, *sh->s, ctr);
        atomicAdd(&times->dp, (u64)g.t_dp);
        atomicAdd(&times->md, (u64)g.t_md);
        atomicAdd(&times->all, (u64)(globaltimer() - g.t_all));
    }
    return true;
}

// One part of a sharded round (mhs_pass_*).  False if a barrier timed out.
__device__ bool run_pass(int op, int shard, int nshards, BatchCounters *ctr, void *buf) {
    Shared *sh = shared();
    InstState &s = *sh->s;
    if (threadIdx.x == 0) load_progress(sh->g, s);
    if (!team_sync()) return false;
    begin_round();
    const bool lead = sh->rank == 0 && threadIdx.x == 0;
    const int32_t t0 = sh->rank * blockDim.x + threadIdx.x, ts = sh->size * blockDim.x;
    if (!sh->g.active && op != kSpExport0 && op != kSpExport1) {
        if (lead && op == kSpEnd1) store_progress(sh->g, s, ctr);
        return true;
    }
    const Ctx c;
    const View v = sh->view;
    SpRound *rc = &v.ctl->c[sh->par], *nx = &v.ctl->c[sh->par ^ 1];
    switch (op) {
        case kSpBegin0:
            if (lead) *nx = SpRound{};
            if (c.epoch > 1) {
                dp_rows();
                if (c.full) {  // FE lowered demands, which the lists repeat
                    if (!team_sync()) return false;
                    md_lists();
                }
            }
            break;
        case kSpContract0:
            if (lead) rc->ntask = rc->npair[0] = rc->npair[1] = 0;
            if (!team_sync()) return false;
            dp_bounds(shard, nshards);
            if (!team_sync()) return false;
            dp_walk(shard, nshards);
            if (!team_sync(rc)) return false;
            dp_tasks(shard, nshards);
            if (!team_sync(rc)) return false;
            decide_pairs(0);
            decide_pairs(1);
            flush(&sh->del, &rc->dp);
            break;
        case kSpExport0:
#pragma unroll 1
            for (int32_t e = t0; e < s.m0; e += ts)
                static_cast<uint8_t *>(buf)[e] = v.e_o2c[e] == -1 - c.epoch;
            break;
        case kSpImport0:
#pragma unroll 1
            for (int32_t e = t0; e < s.m0; e += ts)
                if (static_cast<const uint8_t *>(buf)[e] && v.e_o2c[e] >= 0) delete_edge(e);
            flush(&sh->del, &rc->dp);
            break;
        case kSpBegin1:
#pragma unroll 1
            for (int32_t x = t0; x < s.n0; x += ts) s.v_cnt[x] = 0;
            md_lists();
            break;
        case kSpContract1:
            md_test(true, shard, nshards);
            break;
        case kSpExport1:
#pragma unroll 1
            for (int32_t x = t0; x < s.n0; x += ts)
                static_cast<int32_t *>(buf)[x] = v.v_o2c[x] >= 0 ? s.v_cnt[x] : 0;
            break;
        case kSpImport1:
#pragma unroll 1
            for (int32_t x = t0; x < s.n0; x += ts) s.v_cnt[x] = static_cast<const int32_t *>(buf)[x];
            break;
        case kSpEnd1: {
            md_decide();
            flush(&sh->del2, &rc->md);
            if (!team_sync(rc)) return false;
            const int32_t dp = sh->got.dp, md = sh->got.md;
            if (!finish_round(dp, md)) return false;
            if (lead) store_progress(sh->g, s, ctr);
            break;
        }
        default:
            break;
    }
    return true;
}

// Team of CTAs per instance (team > 0, all CTAs resident: a cooperative
// launch), or one CTA per instance taken from a queue (team = 0).
// The last CTA of the launch hands `words` words over to the host and zeroes
// them for the next launch (a copy and a memset in the stream took 5 us of a
// call with a small instance).  host null: they stay.  Thread 0.
__device__ __noinline__ void report(SpQueue *q, int32_t *from, volatile int32_t *host, int words) {
    if (!host) return;
    __threadfence();
    if (atomicAdd(&q->done, 1) != (int32_t)gridDim.x - 1) return;
    __threadfence();
#pragma unroll 1
    for (int w = 0; w < words; ++w) {
        host[w] = __ldcg(from + w);
        from[w] = 0;
    }
    q->next = q->done = 0;
}

template <int kThreads, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_sparse_build(InstState *st, int count, int team, int32_t max_rounds, SpQueue *queue,
                   SpTotals *out, SpTotals *host, uint64_t absent_ns) {
    Shared *sh = shared();
    bool ok = true;
    if (team > 0) {
        start(st + blockIdx.x / team, blockIdx.x % team, team, absent_ns);
        ok = build_instance<true>(max_rounds, out);
    } else {
        for (;;) {
            __syncthreads();
            if (threadIdx.x == 0) sh->next = atomicAdd(&queue->next, 1);
            __syncthreads();
            if (sh->next >= count) break;
            start(st + sh->next, 0, 1, 0, true);
            build_instance<false>(max_rounds, out);
            __syncthreads();
            const bool again = (vload(&sh->s->status) & kLongRow) != 0;
            __syncthreads();
            if (again) build_again(max_rounds, out);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && !ok) atomicOr(&out->status, kErrTimeout);
    if (threadIdx.x == 0)
        report(queue, reinterpret_cast<int32_t *>(out), reinterpret_cast<int32_t *>(host),
               sizeof(SpTotals) / 4);
}

template <int kThreads, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_sparse_rounds(InstState *st, int count, int team, int32_t limit, BatchCounters *ctr,
                    SpQueue *queue, SpTimes *times, BatchCounters *host, SpMasks masks,
                    uint64_t absent_ns) {
    Shared *sh = shared();
    bool ok = true;
    if (masks.built) {  // (all words on their way together)
        const SpTotals b = *masks.built;
        if ((b.status | b.leave) | (int)(b.cost + b.open > masks.max_cost)) return;
    }
    if (team > 0) {
        start(st + blockIdx.x / team, blockIdx.x % team, team, absent_ns);
        ok = run_instance(limit, ctr, times);
        if (masks.built && ok) {  // (every CTA is past the last round's barrier)
            const int32_t t0 = sh->rank * blockDim.x + threadIdx.x, ts = sh->size * blockDim.x;
#pragma unroll 1
            for (int32_t x = t0; x < sh->n0; x += ts) masks.v[x] = sh->view.v_o2c[x] >= 0;
#pragma unroll 1
            for (int32_t e = t0; e < sh->m0; e += ts) masks.e[e] = sh->view.e_o2c[e] >= 0;
        }
    } else {
        for (;;) {
            __syncthreads();
            if (threadIdx.x == 0) sh->next = atomicAdd(&queue->next, 1);
            __syncthreads();
            if (sh->next >= count) break;
            start(st + sh->next, 0, 1, 0);
            run_instance(limit, ctr, times);
        }
    }
    __syncthreads();
    // (a CTA that gave up has not stored the state, and no other may)
    if (threadIdx.x == 0 && !ok) atomicOr(&ctr->status_any, kErrTimeout);
    if (threadIdx.x == 0)
        report(queue, reinterpret_cast<int32_t *>(ctr), reinterpret_cast<int32_t *>(host),
               sizeof(BatchCounters) / 4);
}

__global__ void __launch_bounds__(kSpThreads, 1)
    k_sparse_pass(InstState *st, int team, int op, int shard, int nshards, BatchCounters *ctr,
                  void *buf, uint64_t absent_ns) {
    start(st, blockIdx.x, team, absent_ns);
    // (a pass that ends early leaves its status for the round's last)
    if (!run_pass(op, shard, nshards, ctr, buf) && ctr && threadIdx.x == 0)
        atomicOr(&ctr->status_any, kErrTimeout);
}

}  // namespace

// ------------------------------------------------------- host launchers --

int sparse_team(int count, int64_t nnz, int64_t items, int sms) {
    // one CTA of kSpThreads threads per SM at most; about one hyperedge or
    // vertex, and a few incidences, per group of lanes
    const int64_t want = std::max<int64_t>((nnz + kSpTeamNnz - 1) / kSpTeamNnz,
                                           (items + kSpTeamItems - 1) / kSpTeamItems);
    const int64_t cap = std::min(sms, kMaxTeam) / std::max(count, 1);
    if (count > 1 && cap < 2) return 0;  // a batch: one CTA each, from a queue
    return (int)std::max<int64_t>(1, std::min(want, cap));
}

template <typename... A, typename... B>
static cudaError_t launch_team(void (*k)(A...), int ctas, cudaStream_t s, B... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kSpThreads);
    cfg.dynamicSmemBytes = shared_bytes(kSpThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, A(args)...);
}

cudaError_t launch_sparse_build(InstState *st, int count, int team, int32_t max_rounds,
                                SpQueue *queue, SpTotals *out, SpTotals *host, int sms,
                                cudaStream_t s) {
    if (team > 0)
        return launch_team(k_sparse_build<kSpThreads, 1>, count * team, s, st, count, team,
                           max_rounds, queue, out, host, t_absent_ns);
    const size_t smem = shared_bytes(kSpBatchThreads) + 8 * kLocalVertices;
    k_sparse_build<kSpBatchThreads, kSpBatchBlocks>
        <<<std::min(count, sms * kSpBatchBlocks), kSpBatchThreads, smem, s>>>(
            st, count, 0, max_rounds, queue, out, host, 0);
    return cudaGetLastError();
}

cudaError_t launch_sparse_rounds(InstState *st, int count, int team, int32_t limit,
                                 BatchCounters *ctr, SpQueue *queue, SpTimes *times,
                                 BatchCounters *host, const SpMasks &masks, int sms,
                                 cudaStream_t s) {
    if (team > 0)
        return launch_team(k_sparse_rounds<kSpThreads, 1>, count * team, s, st, count, team, limit,
                           ctr, queue, times, host, masks, t_absent_ns);
    k_sparse_rounds<kSpBatchThreads, kSpBatchBlocks>
        <<<std::min(count, sms * kSpBatchBlocks), kSpBatchThreads, shared_bytes(kSpBatchThreads), s>>>(
            st, count, 0, limit, ctr, queue, times, host, masks, 0);
    return cudaGetLastError();
}

cudaError_t launch_sparse_pass(InstState *st, int team, int op, int shard, int nshards,
                               BatchCounters *ctr, void *buf, cudaStream_t s) {
    return launch_team(k_sparse_pass, team, s, st, team, op, shard, nshards, ctr, buf, t_absent_ns);
}

void set_team_absent(uint64_t ns) { t_absent_ns = ns; }
uint64_t team_absent() { return t_absent_ns; }

}  // namespace mhs
