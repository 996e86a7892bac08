// noalloc.cu -- mhs_kernelize_noalloc: a complete kernelization of one small
// instance whose working memory is a fixed, file-scope device array, so the
// call allocates nothing.
//
// Who needs it: callers that may not allocate device memory while they run
// -- code inside a custom or fixed-budget allocator, real-time loops that
// forbid cudaMalloc/cudaFree (both can synchronise the device), or plug-ins
// embedded in a host that owns all device memory.  They pass device inputs
// and device outputs; everything else (id maps, bit-packed operands, flags,
// counters, the per-instance state) lives in kScratch below.
//
// The array is kScratchBytes (6 MiB) and every GPU that loads this library
// holds it until the process exits.  It fits instances with n <= 4096,
// m <= 4096 and at most 65,536 incidences; larger ones are rejected with
// MHS_EINVAL.  It takes the candidate lists (sparse.cu: one launch to load, one
// for all rounds), or, where their first round would walk too much, the
// bit-packed passes with the encode / compaction kernels of the main path.
//
// All calls share the one array and it keeps the last call's contents, so
// everything that must start from zero is cleared by each call.  Calls whose
// GPU work overlaps (different streams or threads at the same time) race on
// the array and give wrong results: serialise them.
//
// Set-up: every call looks up the array's device address with
// cudaGetSymbolAddress, with the caller's device current.  No address is
// cached, so a context torn down and created again (cudaDeviceReset) cannot
// leave a stale one behind.  The first call on a device, and the first that
// takes the other form, may load the library's device code into the context;
// make them before any stream capture.
//
// Pointers: every device array the caller passes is checked with
// cudaPointerGetAttributes (device or managed memory of the current device)
// before any kernel touches it; anything else is MHS_EINVAL.
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdio>
#include <cstring>

#include "kernels.h"
#include "mhs.h"
#include "mhs_internal.h"

namespace mhs {
namespace {

constexpr int32_t kNoAllocMaxN = 4096;
constexpr int32_t kNoAllocMaxM = 4096;
constexpr int64_t kNoAllocMaxNnz = 65536;
constexpr size_t kScratchBytes = (size_t)6 << 20;  // 6 MiB

static __device__ __align__(256) uint8_t kScratch[kScratchBytes];

inline int64_t up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }
inline int64_t words(int64_t K) { return up(((K + 31) / 32) > 0 ? (K + 31) / 32 : 1, 4); }

// The candidate lists are taken for rows of this mean length at most, and while
// their first round visits no more list entries than this (with what the pairs
// found in them cost, in such units).  Measured, a call
// by lists / by bits alone (us); bits after a build that did not pay: + 50.
//   n 1,000, m 2,000, |e| 2..16:       cost 55 K     83 / 254
//   n 256, m 4,096, |e| 14..16:        cost 1.8 M   117 / 180
//   n 32, m 4,096, |e| 14..16:         cost 15 M    308 / 292
//   n 8, m 4,096, |e| 1..8:            cost 20 M     87 / 381
//   n 16, m 4,096, |e| 8..16:          cost 25 M   1280 / 370
//   n 1,000, m 300, |e| 150..200:      mean 175     169 / 201
//   n 2,000, m 200, |e| 300..320:      mean 310     275 / 237
constexpr unsigned long long kNoAllocCost = 20000000;
constexpr int64_t kNoAllocMeanSize = 200;
// Not even built above this: a list of mean length per hyperedge (n 16, m 4,096,
// |e| 8..16: 12.6 M, 400 us with the build, 370 without; n 8: 9.3 M).
constexpr int64_t kNoAllocEstimate = 10000000;

// What the candidate lists' two launches start with at zero, and what the host
// reads back (the first two).
struct Words {
    SpTotals totals;
    BatchCounters ctr;
    SpTimes times;
    SpQueue queue;
};
struct Found {
    SpTotals totals;
    BatchCounters ctr;
};
static_assert(offsetof(Words, ctr) == offsetof(Found, ctr), "one copy");

struct Take {
    int64_t bytes = 0;
    int64_t operator()(int64_t n) {
        int64_t o = bytes;
        bytes += up(n > 0 ? n : 1, 256);
        return o;
    }
};

mhs_status err(char *buf, size_t cap, mhs_status st, const char *msg) {
    if (buf && cap) {
        std::strncpy(buf, msg, cap - 1);
        buf[cap - 1] = '\0';
    }
    return st;
}

// True if p is device (or managed) memory that device `dev` can use; a
// pointer of no kind CUDA knows (plain host memory) is rejected.
bool on_device(const void *p, int dev) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();  // the failed query's error is not sticky: clear it
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

}  // namespace
}  // namespace mhs

using namespace mhs;

extern "C" mhs_status mhs_kernelize_noalloc(int32_t n, int32_t m, const int32_t *edge_ptr,
                                            const int32_t *edge_vtx, const int32_t *demand,
                                            int32_t nnz, uint8_t *alive_v, uint8_t *alive_e,
                                            int32_t *rounds_out, void *cuda_stream,
                                            char *err_buf, size_t err_cap) {
    if (n < 0 || m < 0 || nnz < 0)
        return err(err_buf, err_cap, MHS_EINVAL, "n, m and nnz must be >= 0");
    if (n > kNoAllocMaxN || m > kNoAllocMaxM || nnz > kNoAllocMaxNnz)
        return err(err_buf, err_cap, MHS_EINVAL,
                   "instance too large for the static scratch (n, m <= 4096, nnz <= 65536)");
    if (!edge_ptr || (m > 0 && !demand) || (nnz > 0 && !edge_vtx) ||
        (n > 0 && !alive_v) || (m > 0 && !alive_e))
        return err(err_buf, err_cap, MHS_EINVAL, "NULL array");
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0)
        return err(err_buf, err_cap, MHS_ECUDA, "no current CUDA device");
    if (!on_device(edge_ptr, dev) || (m > 0 && !on_device(demand, dev)) ||
        (nnz > 0 && !on_device(edge_vtx, dev)) || (n > 0 && !on_device(alive_v, dev)) ||
        (m > 0 && !on_device(alive_e, dev)))
        return err(err_buf, err_cap, MHS_EINVAL,
                   "an array is not device memory of the current device");
    void *base_v = nullptr;
    if (cudaGetSymbolAddress(&base_v, kScratch) != cudaSuccess || !base_v)
        return err(err_buf, err_cap, MHS_ECUDA, "cudaGetSymbolAddress(scratch) failed");
    uint8_t *base = static_cast<uint8_t *>(base_v);
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        sms <= 0)
        return err(err_buf, err_cap, MHS_ECUDA, "cannot read the SM count");

    // layout inside the scratch (same roles as the main path's arena)
    Take take;
    const int64_t o_state = take(sizeof(InstState));
    const int64_t o_vo2c = take(4 * (int64_t)n), o_eo2c = take(4 * (int64_t)m);
    const int64_t o_vcnt = take(4 * ((int64_t)n + 1));
    // the two forms of the rest lie over one another
    Take bits = take;
    const int64_t o_plan = bits(sizeof(Plan));
    const int64_t o_rowoff = bits(2 * sizeof(int32_t));
    const int64_t o_tileoff = bits(2 * sizeof(int64_t));
    const int64_t o_ctr = bits(sizeof(BatchCounters));
    const int64_t o_kerr = bits(sizeof(int32_t));
    const int64_t o_vc2o = bits(4 * (int64_t)n), o_ec2o = bits(4 * (int64_t)m);
    const int64_t o_eprev = bits(4 * (int64_t)m);
    const int64_t o_ef = bits(4 * (int64_t)m), o_es = bits(4 * (int64_t)m);
    const int64_t o_vdeg = bits(4 * ((int64_t)n + 1)), o_vmaxf = bits(4 * (int64_t)n);
    const int64_t o_edel = bits(m), o_vdel = bits(n);
    const int64_t arows = up(m > 0 ? m : 1, kRowAlign), atrows = up(n > 0 ? n : 1, kRowAlign);
    const int64_t o_ab = bits(arows * words(n) * 4);
    const int64_t o_atb = bits(atrows * words(m) * 4);
    const int64_t o_row = take(4 * (int64_t)nnz), o_pos = take(4 * (int64_t)nnz);
    const int64_t o_tmp = take(4 * (int64_t)nnz), o_vedge = take(8 * (int64_t)nnz);
    const int64_t o_erec = take(16 * (int64_t)m), o_vaux = take(16 * (int64_t)n);
    const int64_t o_heavy = take(4 * sp_heavy_cap(nnz));
    const int32_t task_cap = 8192, pair_cap = 131072;
    const int64_t o_task = take(16 * (int64_t)task_cap), o_pairs = take(8 * (int64_t)pair_cap);
    const int64_t o_words = take(sizeof(Words));  // from here on zero at the start
    const int64_t o_ctl = take(sizeof(SpCtl)), o_vrec = take(16 * (int64_t)n);
    const int64_t o_vagg = take(16 * (int64_t)n);
    const int64_t slots = sp_pair_slots(m), o_tab = take((int64_t)sizeof(SpPair) * slots);
    const int64_t o_bound = take(4 * (int64_t)n), o_gone = take(4 * (((int64_t)m + 31) / 32));
    const int64_t o_estamp = take(4 * (int64_t)m);
    const int64_t o_vstamp = take(4 * (int64_t)n), o_tstamp = take(4 * (int64_t)n);
    if (take.bytes > (int64_t)kScratchBytes || bits.bytes > (int64_t)kScratchBytes)
        return err(err_buf, err_cap, MHS_EINVAL, "instance does not fit the static scratch");

    InstState st;
    std::memset(&st, 0, sizeof(st));
    st.n0 = n;
    st.m0 = m;
    st.nnz0 = nnz;
    st.eptr = edge_ptr;  // inputs are read in place
    st.evtx = edge_vtx;
    st.f = const_cast<int32_t *>(demand);  // read only: rule FE is off here
    st.v_o2c = reinterpret_cast<int32_t *>(base + o_vo2c);
    st.v_c2o = reinterpret_cast<int32_t *>(base + o_vc2o);
    st.e_o2c = reinterpret_cast<int32_t *>(base + o_eo2c);
    st.e_c2o = reinterpret_cast<int32_t *>(base + o_ec2o);
    st.e_prev = reinterpret_cast<int32_t *>(base + o_eprev);
    st.e_f = reinterpret_cast<int32_t *>(base + o_ef);
    st.e_s = reinterpret_cast<int32_t *>(base + o_es);
    st.v_deg = reinterpret_cast<int32_t *>(base + o_vdeg);
    st.v_maxf = reinterpret_cast<int32_t *>(base + o_vmaxf);
    st.v_cnt = reinterpret_cast<int32_t *>(base + o_vcnt);
    st.e_del = base + o_edel;
    st.v_del = base + o_vdel;
    st.Ab = reinterpret_cast<uint32_t *>(base + o_ab);
    st.Atb = reinterpret_cast<uint32_t *>(base + o_atb);
    st.Ab_pitch = (int32_t)words(n);
    st.Atb_pitch = (int32_t)words(m);
    st.A_rows = (int32_t)arows;
    st.At_rows = (int32_t)atrows;

    st.sp_row = reinterpret_cast<uint32_t *>(base + o_row);
    st.sp_pos = reinterpret_cast<int32_t *>(base + o_pos);
    st.sp_tmp = reinterpret_cast<uint32_t *>(base + o_tmp);
    st.sp_vedge = reinterpret_cast<unsigned long long *>(base + o_vedge);
    st.sp_erec = reinterpret_cast<int4 *>(base + o_erec);
    st.sp_vrec = reinterpret_cast<int4 *>(base + o_vrec);
    st.sp_vagg = reinterpret_cast<SpAgg *>(base + o_vagg);
    st.sp_vaux = reinterpret_cast<int4 *>(base + o_vaux);
    st.sp_bound = reinterpret_cast<int32_t *>(base + o_bound);
    st.sp_gone = reinterpret_cast<uint32_t *>(base + o_gone);
    st.sp_estamp = reinterpret_cast<int32_t *>(base + o_estamp);
    st.sp_vstamp = reinterpret_cast<int32_t *>(base + o_vstamp);
    st.sp_tstamp = reinterpret_cast<int32_t *>(base + o_tstamp);
    st.sp_task = reinterpret_cast<int4 *>(base + o_task);
    st.sp_task_cap = task_cap;
    st.sp_pair_tab = reinterpret_cast<SpPair *>(base + o_tab);
    st.sp_pair_mask = (uint32_t)slots - 1;
    st.sp_pairs = reinterpret_cast<int2 *>(base + o_pairs);
    st.sp_pair_cap = pair_cap;
    st.sp_heavy = reinterpret_cast<int32_t *>(base + o_heavy);
    st.sp_ctl = reinterpret_cast<SpCtl *>(base + o_ctl);

    Plan pl;
    std::memset(&pl, 0, sizeof(pl));
    pl.count = 1;
    pl.row_off = reinterpret_cast<int32_t *>(base + o_rowoff);
    pl.tile_off = reinterpret_cast<int64_t *>(base + o_tileoff);

    InstState *dst = reinterpret_cast<InstState *>(base + o_state);
    Plan *dplan = reinterpret_cast<Plan *>(base + o_plan);
    BatchCounters *dctr = reinterpret_cast<BatchCounters *>(base + o_ctr);
    int32_t *dkerr = reinterpret_cast<int32_t *>(base + o_kerr);

    // pageable sources: each copy returns once the source has been staged
    Words *dw = reinterpret_cast<Words *>(base + o_words);
    const int team = sparse_team(1, nnz, (int64_t)n + m, sms);
    cudaError_t e = cudaMemcpyAsync(dst, &st, sizeof(st), cudaMemcpyHostToDevice, s);
    const bool lists = nnz <= kNoAllocMeanSize * m && (int64_t)nnz * m <= kNoAllocEstimate * n;
    Found found;
    std::memset(&found, 0, sizeof(found));
    BatchCounters &ctr = found.ctr;
    if (lists) {
        if (e == cudaSuccess)
            e = cudaMemsetAsync(base + o_words, 0, (size_t)(take.bytes - o_words), s);
        if (e == cudaSuccess)
            e = launch_sparse_build(dst, 1, team, 0, &dw->queue, &dw->totals, nullptr, sms, s);
        // (whether they are to run is decided on the device: one wait, not two)
        if (e == cudaSuccess)
            e = launch_sparse_rounds(dst, 1, team, 0, &dw->ctr, &dw->queue, &dw->times, nullptr,
                                     {&dw->totals, kNoAllocCost, alive_v, alive_e}, sms, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&found, dw, sizeof(found), cudaMemcpyDeviceToHost, s);
    } else {
        if (e == cudaSuccess) e = launch_validate(dst, 1, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&found.totals.status, &dst->status, sizeof(int32_t),
                                cudaMemcpyDeviceToHost, s);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return err(err_buf, err_cap, MHS_ECUDA, cudaGetErrorString(e));
    if (found.totals.status & (kErrTimeout | kErrCapacity))
        return err(err_buf, err_cap, MHS_EDEVICE, "kernel reported an error status");
    if (found.totals.status)
        return err(err_buf, err_cap, MHS_EINVAL, "malformed instance (bad edge_ptr or vertex id)");
    if (lists && !found.totals.leave && found.totals.cost + found.totals.open <= kNoAllocCost) {
        if (ctr.status_any || ctr.active)
            return err(err_buf, err_cap, MHS_EDEVICE, "kernel reported an error status");
        if (rounds_out) *rounds_out = ctr.max_rounds_seen;
        return MHS_OK;
    }

    // the bit-packed passes, from the input again
    e = cudaMemcpyAsync(dst, &st, sizeof(st), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dplan, &pl, sizeof(pl), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(dkerr, 0, sizeof(int32_t), s);
    if (e != cudaSuccess) return err(err_buf, err_cap, MHS_ECUDA, cudaGetErrorString(e));
    // the bit-packed operands must start all-zero (a call that stopped early
    // may have left incidences set)
    e = cudaMemsetAsync(base + o_ab, 0, (size_t)(o_atb - o_ab + atrows * words(m) * 4), s);
    if (e == cudaSuccess) e = launch_build(dst, 1, 0, nnz, m, n, s, 0);
    if (e != cudaSuccess) return err(err_buf, err_cap, MHS_ECUDA, cudaGetErrorString(e));
    int32_t kerr = 0;
    // every changing round deletes an item, so n + m + 1 rounds always suffice
    for (int32_t r = 0; r <= n + m + 1; ++r) {
        e = launch_round_phase(dst, dplan, dctr, 1, 0, kPopcount, sms, dkerr, s, nullptr, nullptr);
        if (e == cudaSuccess)
            e = launch_round_phase(dst, dplan, dctr, 1, 1, kPopcount, sms, dkerr, s, nullptr,
                                   nullptr);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&ctr, dctr, sizeof(ctr), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&kerr, dkerr, sizeof(kerr), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return err(err_buf, err_cap, MHS_ECUDA, cudaGetErrorString(e));
        if (kerr || ctr.status_any)
            return err(err_buf, err_cap, MHS_EDEVICE, "kernel reported an error status");
        if (ctr.active == 0) break;
    }
    if (ctr.active != 0)  // unreachable with correct kernels: never report a partial result
        return err(err_buf, err_cap, MHS_EDEVICE, "round cap reached before fixpoint");
    if (n > 0 || m > 0) {
        e = launch_alive_masks(dst, n > 0 ? alive_v : nullptr, m > 0 ? alive_e : nullptr, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return err(err_buf, err_cap, MHS_ECUDA, cudaGetErrorString(e));
    }
    if (rounds_out) *rounds_out = ctr.max_rounds_seen;
    return MHS_OK;
}
