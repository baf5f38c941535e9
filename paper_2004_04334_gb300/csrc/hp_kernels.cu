// sm_103a kernels of libhp: silicon-pixel local reconstruction.
//
// One launch reconstructs a batch of E independent events (a single event is
// E = 1).  The unit of clustering work is an item = (event, module); there
// are E * M items, in (event, module) order.
//
//   hist_kernel     module histogram: count[item] (shared-memory bins over a
//                   block's range of digis, flushed with global atomics);
//                   validates module ids
//   scan_kernel     one block per event: exclusive prefix sum of the event's
//                   M counts -> bucket start of every item (the event's digi
//                   offset is the base, so events scan independently)
//   scatter_kernel  bucket scatter: each digi's word and in-event index go to
//                   its item's bucket (block-local ranks in shared memory,
//                   positions reserved by the histogram or by one global
//                   atomic per non-empty bin); scatter_wide_kernel for many
//                   digis on many modules
//   cc_kernel       persistent clustering: groups of threads take tickets of
//                   up to kGroup consecutive items (the count is a tuning
//                   parameter); a ticket's small items go together through
//                   the packed tier (bitmaps of the words they touch), larger
//                   ones one by one through the run tier (bitmaps of the
//                   module, union-find over horizontal runs), in shared
//                   memory, or in global scratch if their runs do not fit;
//                   items too large for a group's share by the whole block;
//                   cc_hash_kernel (the hash label store, a tuning choice)
//                   has groups of 128-512 threads cluster the items between
//                   on a hash table each; kept clusters are staged per item
//                   in id order
//   offsets_kernel  each item's first output position (prefix over the items'
//                   kept-cluster counts, chained across chunks)
//   copy_kernel     staged clusters to their ordered output positions; per-event
//                   status codes
//
// Launches of few digis run three kernels instead: bucket_kernel (the first
// three in one), the clustering kernel and finish_kernel (the last two).
//
// Labels are unique and the order of clusters fixed, so every tier gives the
// same result: the id of a cluster is its smallest linear pixel index, the
// root of its tree in every union-find here; charge, pixel count and the two
// moments sum(q * row), sum(q * col) accumulate per root in 32 bits (the
// charge always fits: the configuration bounds every cluster's), and an item
// with a cluster heavy enough to overflow the moments sums them again in 64
// bits.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <type_traits>

#include "hp_internal.h"

namespace hp {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Programmatic dependent launch between the pass's kernels: each kernel lets
// the next one launch as soon as all its own blocks are running (the next
// kernel's blocks then take free SM slots and wait), and each dependent
// kernel waits, before it reads anything but the call's inputs, until the
// previous grid has completed and its writes are visible.  (A launch's first
// kernel is an ordinary launch, so the inputs are in place by then.)  The
// waits are the hardware's, not spins.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
constexpr uint32_t kSpinLimit = 1u << 24;          // iterations of a blocking wait, at most
constexpr unsigned long long kWaitNs = 1000000000ull; // and at most one second of it

struct ItemCtx {
    uint32_t b, n;
    int32_t gain, ped;
    int32_t *label_e;    // label of the event's first digi, or null
    uint16_t *label16_e; // compact label of the event's first digi, or null (then label_e is null)
    uint32_t *err_e;     // the event's error bits
};

// Compact labels: the rank of the digi's cluster among the kept clusters of
// its item (= its staging ordinal), or these two markers.
constexpr uint16_t kLab16Below = 0xFFFFu;   // pixel below threshold (label -1)
constexpr uint16_t kLab16Dropped = 0xFFFEu; // cluster below threshold (label -2)

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t sm_id()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void st_relaxed(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void st_release(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Exclusive scan of one value per thread over a block of T threads with a
// single barrier: warp scans, then every warp scans the warp totals in
// registers.  tmp must not be rewritten before the caller's next barrier.
template <int T>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *tmp, uint32_t *total)
{
    static_assert(T / 32 <= 32, "one warp scans the warp totals");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) tmp[warp] = x;
    __syncthreads();
    const uint32_t wt = lane < T / 32 ? tmp[lane] : 0u;
    uint32_t ws = wt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, ws, o);
        if (lane >= o) ws += y;
    }
    *total = __shfl_sync(kFull, ws, T / 32 - 1);
    return __shfl_sync(kFull, ws - wt, warp) + x - v;
}

// Event and module of work item `item` (one division, by the thread that
// sets up the item's record).
__device__ __forceinline__ void item_coords(uint64_t item, uint32_t M, uint32_t *e, uint32_t *m)
{
    if (item <= 0xFFFFFFFFull) {
        const uint32_t i32 = (uint32_t)item;
        *e = i32 / M;
        *m = i32 - *e * M;
    } else {
        *e = (uint32_t)(item / M);
        *m = (uint32_t)(item - (uint64_t)*e * M);
    }
}

// Per-item record of a ticket, set up once in shared memory by one thread
// (the division by the module count and the calibration loads happen there,
// not in every thread of the block).
struct ItemRec {
    uint32_t e;
    int32_t gain, ped;
    uint32_t label_off; // the event's first digi (a launch has fewer than 2^32)
};

__device__ __forceinline__ ItemRec make_rec(const Launch &L, uint64_t item)
{
    ItemRec r;
    uint32_t m;
    item_coords(item, L.g.M, &r.e, &m);
    r.gain = L.g.gain[m];
    r.ped = L.g.ped[m];
    r.label_off = (uint32_t)L.offsets[r.e];
    return r;
}

__device__ __forceinline__ ItemCtx make_item(const Launch &L, const ItemRec &rec, uint32_t b, uint32_t n)
{
    ItemCtx it;
    it.b = b;
    it.n = n;
    it.gain = rec.gain;
    it.ped = rec.ped;
    it.label_e = L.out.label ? L.out.label + rec.label_off : nullptr;
    it.label16_e = L.out.label16 ? L.out.label16 + rec.label_off : nullptr;
    it.err_e = L.ws.event_err + rec.e;
    return it;
}

// ---------------------------------------------------------------- histogram / scatter

// Thread t of a histogram/scatter block owns the kPerThread consecutive digis
// [c0 + kPerThread * t, ...) of the block's chunk; module ids and words are
// read with 16-byte vector loads when the arrays are 16-byte aligned.
constexpr int kPerThread = kChunk / kHistThreads;
static_assert(kPerThread == 8, "vector loads below assume 8 digis per thread");

__device__ __forceinline__ void load_modules(const Launch &L, uint64_t k0, uint64_t c1, uint32_t m[kPerThread])
{
    if (((reinterpret_cast<uintptr_t>(L.modules) & 15) == 0) && k0 + kPerThread <= c1) {
        const uint4 a = *reinterpret_cast<const uint4 *>(L.modules + k0);
        m[0] = a.x & 0xFFFFu, m[1] = a.x >> 16, m[2] = a.y & 0xFFFFu, m[3] = a.y >> 16;
        m[4] = a.z & 0xFFFFu, m[5] = a.z >> 16, m[6] = a.w & 0xFFFFu, m[7] = a.w >> 16;
    } else {
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) m[j] = k0 + j < c1 ? (uint32_t)L.modules[k0 + j] : 0xFFFFFFFFu;
    }
}

__device__ __forceinline__ void load_words(const Launch &L, uint64_t k0, uint64_t c1, uint32_t w[kPerThread])
{
    if (((reinterpret_cast<uintptr_t>(L.words) & 15) == 0) && k0 + kPerThread <= c1) {
        const uint4 a = *reinterpret_cast<const uint4 *>(L.words + k0);
        const uint4 b = *reinterpret_cast<const uint4 *>(L.words + k0 + 4);
        w[0] = a.x, w[1] = a.y, w[2] = a.z, w[3] = a.w, w[4] = b.x, w[5] = b.y, w[6] = b.z, w[7] = b.w;
    } else {
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) w[j] = k0 + j < c1 ? L.words[k0 + j] : 0u;
    }
}

// Asynchronous 16-byte copies global -> shared (cp.async), committed as one
// group and waited for by the issuing thread only.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Prefetch of the thread's next kPerThread digis (starting at k0, all before
// c1 and 16-byte aligned) into its own slots of pf_m / pf_w; false (nothing
// issued) for a partial or unaligned group, which is then loaded directly.
__device__ __forceinline__ bool prefetch_digis(const Launch &L, uint64_t k0, uint64_t c1, uint16_t *pf_m, uint32_t *pf_w)
{
    if (k0 + kPerThread > c1 || ((reinterpret_cast<uintptr_t>(L.modules) | reinterpret_cast<uintptr_t>(L.words)) & 15))
        return false;
    const uint32_t t = threadIdx.x * kPerThread;
    cp_async16(pf_m + t, L.modules + k0);
    cp_async16(pf_w + t, L.words + k0);
    cp_async16(pf_w + t + 4, L.words + k0 + 4);
    cp_async_commit();
    return true;
}

__device__ __forceinline__ void take_prefetched(const uint16_t *pf_m, const uint32_t *pf_w, uint32_t m[kPerThread],
                                                uint32_t w[kPerThread])
{
    cp_async_wait_all();
    const uint32_t t = threadIdx.x * kPerThread;
    const uint4 a = *reinterpret_cast<const uint4 *>(pf_m + t);
    m[0] = a.x & 0xFFFFu, m[1] = a.x >> 16, m[2] = a.y & 0xFFFFu, m[3] = a.y >> 16;
    m[4] = a.z & 0xFFFFu, m[5] = a.z >> 16, m[6] = a.w & 0xFFFFu, m[7] = a.w >> 16;
    const uint4 b = *reinterpret_cast<const uint4 *>(pf_w + t);
    const uint4 c = *reinterpret_cast<const uint4 *>(pf_w + t + 4);
    w[0] = b.x, w[1] = b.y, w[2] = b.z, w[3] = b.w, w[4] = c.x, w[5] = c.y, w[6] = c.z, w[7] = c.w;
}

// Event of each of the thread's digis: a binary search over the block's
// event offsets (in shared memory when they fit), then a forward walk.
constexpr uint32_t kChunkEvents = 512; // event offsets a block keeps in shared memory

__device__ __forceinline__ void digi_events(const Launch &L, const uint64_t *s_off, uint32_t ef, uint32_t el,
                                            uint64_t k0, uint32_t e_of[kPerThread])
{
    uint32_t e = ef;
    if (ef != el) {
        const bool in_sh = el - ef + 1 < kChunkEvents;
        uint32_t lo = ef, hi = el;
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1) >> 1;
            const uint64_t o = in_sh ? s_off[mid - ef] : L.offsets[mid];
            if (o <= k0)
                lo = mid;
            else
                hi = mid - 1;
        }
        e = lo;
    }
    uint64_t next = e < el ? (el - ef + 1 < kChunkEvents ? s_off[e + 1 - ef] : L.offsets[e + 1]) : ~0ull;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
        while (k0 + j >= next) {
            ++e;
            next = e < el ? L.offsets[e + 1] : ~0ull;
        }
        e_of[j] = e;
    }
}

// Largest e in [lo, hi] with off[e] <= k (requires off[lo] <= k), by one
// full warp: 32 probes per round shrink the interval 32-fold.
__device__ __forceinline__ uint32_t find_event_warp(const uint64_t *off, uint32_t lo, uint32_t hi, uint64_t k)
{
    const uint32_t lane = threadIdx.x & 31;
    while (lo < hi) {
        const uint32_t step = (hi - lo + 31) / 32;
        const uint32_t p = min(hi, lo + (lane + 1) * step);
        const uint32_t le = __ballot_sync(kFull, off[p] <= k);
        if (le == 0) {
            hi = lo + step - 1;
        } else {
            const uint32_t t = 31 - __clz(le);
            const uint32_t pt = min(hi, lo + (t + 1) * step);
            if (t < 31) hi = min(hi, lo + (t + 2) * step) - 1;
            lo = pt;
            if (hi < lo) hi = lo;
        }
    }
    return lo;
}

struct ChunkInfo {
    uint64_t c0, c1, keybase;
    uint32_t ef, el, nkeys;
    bool use_sh;
};

// Digis [c0, c1) of block b of nb: contiguous ranges cut at multiples of
// kPerThread digis (so every thread's group of digis is 16-byte aligned).
__device__ __forceinline__ void block_range(uint64_t N, uint32_t b, uint32_t nb, uint64_t *c0, uint64_t *c1)
{
    const uint64_t ng = (N + kPerThread - 1) / kPerThread;
    *c0 = min(N, (uint64_t)b * ng / nb * kPerThread);
    *c1 = min(N, (uint64_t)(b + 1) * ng / nb * kPerThread);
}

// Events and (event, module) keys of the digis [c0, c1) (c0 < c1): the first
// and last event by a warp search, the events' offsets in shared memory when
// they fit, and whether the keys fit a shared-memory histogram.
template <int kThreads = kHistThreads>
__device__ __forceinline__ ChunkInfo chunk_info(const Launch &L, uint64_t c0, uint64_t c1, uint32_t *s_ev,
                                                uint64_t *s_off)
{
    ChunkInfo ci;
    ci.c0 = c0;
    ci.c1 = c1;
    if (threadIdx.x < 32) {
        const uint32_t ef = find_event_warp(L.offsets, 0, L.E - 1, ci.c0);
        const uint32_t el = find_event_warp(L.offsets, ef, L.E - 1, ci.c1 - 1);
        if (threadIdx.x == 0) {
            s_ev[0] = ef;
            s_ev[1] = el;
        }
    }
    __syncthreads();
    ci.ef = s_ev[0];
    ci.el = s_ev[1];
    if (ci.el - ci.ef + 1 < kChunkEvents)
        for (uint32_t i = threadIdx.x; i <= ci.el - ci.ef + 1; i += kThreads) s_off[i] = L.offsets[ci.ef + i];
    const uint64_t nk = (uint64_t)(ci.el - ci.ef + 1) * L.g.M;
    ci.use_sh = nk <= (uint64_t)kHistCap;
    ci.nkeys = ci.use_sh ? (uint32_t)nk : 0u;
    ci.keybase = (uint64_t)ci.ef * L.g.M;
    return ci;
}

// Shared-memory histogram of a block: with few (event, module) keys every
// warp counts into its own sub-histogram (atomics collide only inside a
// warp), else one shared histogram.
constexpr uint32_t kHistWarps = kHistThreads / 32;
constexpr uint32_t kSubKeys = kHistCap / kHistWarps; // keys per warp sub-histogram

// The thread's group of module ids at k0, packed (absent ones 0).
__device__ __forceinline__ uint4 load_packed(const Launch &L, uint64_t k0, uint64_t c1)
{
    if (((reinterpret_cast<uintptr_t>(L.modules) & 15) == 0) && k0 + kPerThread <= c1)
        return *reinterpret_cast<const uint4 *>(L.modules + k0);
    uint32_t m[kPerThread];
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) m[j] = k0 + j < c1 ? (uint32_t)L.modules[k0 + j] : 0u;
    return make_uint4(m[0] | m[1] << 16, m[2] | m[3] << 16, m[4] | m[5] << 16, m[6] | m[7] << 16);
}

// Histogram, persistent: block b counts the digis of its contiguous range
// (one event search a block), 8 module ids a thread per step with the next
// two steps' ids loaded ahead, into a shared histogram over the range's keys, flushed once with one global atomic per non-empty key; the
// atomic's return value (the block's offset inside the key's bucket) is
// kept in blk_off for the scatter kernel.  A group of digis of a step that
// lies in one event (most do), all valid, is counted without a look at its
// digis' events: three instructions a digi, which bound this kernel, instead of
// a dozen (27.7M digis in 256 events: 45.7 -> 29.7 us, 1.9 TB/s).
__global__ void __launch_bounds__(kHistThreads, 3) hist_kernel(const __grid_constant__ Launch L)
{
    extern __shared__ uint32_t sh[];
    __shared__ uint32_t s_ev[2];
    pdl_trigger();
    __shared__ uint64_t s_off[kChunkEvents + 1];
    // the event offsets must run 0 = o[0] <= o[1] <= ... <= o[E] = N (the
    // device entry points take them from the caller); each block checks a
    // slice, and a violation makes every later kernel skip its writes and
    // every event report HP_EINVAL
    {
        const uint64_t e0 = (uint64_t)blockIdx.x * L.E / gridDim.x, e1 = (uint64_t)(blockIdx.x + 1) * L.E / gridDim.x;
        bool bad = false;
        for (uint64_t e = e0 + threadIdx.x; e < e1; e += kHistThreads) bad |= L.offsets[e] > L.offsets[e + 1];
        if (threadIdx.x == 0 && blockIdx.x == 0) bad |= L.offsets[0] != 0 || L.offsets[L.E] != L.N;
        if (bad) atomicOr(&L.ws.ctl[1], kErrBadOffsets);
    }
    uint64_t c0, c1;
    block_range(L.N, blockIdx.x, gridDim.x, &c0, &c1);
    if (c0 >= c1) return;
    // the first module ids are loaded before the event search, so that the
    // two latencies overlap
    const uint64_t mine = (uint64_t)threadIdx.x * kPerThread;
    uint4 cur = load_packed(L, c0 + mine, c1), next = load_packed(L, c0 + kChunk + mine, c1);
    const ChunkInfo ci = chunk_info<>(L, c0, c1, s_ev, s_off);
    const uint32_t M = L.g.M, warp = threadIdx.x >> 5;
    const bool sub = ci.use_sh && ci.nkeys <= kSubKeys;
    const uint32_t nbins = sub ? ci.nkeys * kHistWarps : ci.nkeys;
    for (uint32_t i = threadIdx.x; i < nbins; i += kHistThreads) sh[i] = 0;
    __syncthreads();
    uint32_t *bins = sub ? sh + warp * ci.nkeys : sh;
    const bool off_sh = ci.el - ci.ef + 1 < kChunkEvents;
    uint32_t es = ci.ef; // event of the step's first digi
    for (uint64_t s0 = c0; s0 < c1; s0 += kChunk) {
        const uint64_t k0 = s0 + mine;
        const uint32_t a[4] = {cur.x, cur.y, cur.z, cur.w};
        cur = next;
        next = load_packed(L, k0 + 2 * kChunk, c1);
        if (k0 >= c1) continue; // (no barriers below)
        if (off_sh)
            while (es < ci.el && s_off[es + 1 - ci.ef] <= s0) ++es;
        const bool one = ci.use_sh && off_sh && (es == ci.el || s_off[es + 1 - ci.ef] >= min(c1, s0 + kChunk));
        const uint32_t top = __vmaxu2(__vmaxu2(a[0], a[1]), __vmaxu2(a[2], a[3]));
        // all present, valid and of the step's event: most groups
        if (one && k0 + kPerThread <= c1 && max(top & 0xFFFFu, top >> 16) < M) {
            uint32_t *eb = bins + (es - ci.ef) * M;
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) atomicAdd(eb + (j & 1 ? a[j / 2] >> 16 : a[j / 2] & 0xFFFFu), 1u);
            continue;
        }
        uint32_t e_of[kPerThread];
        digi_events(L, s_off, ci.ef, ci.el, k0, e_of);
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            const uint32_t m = j & 1 ? a[j / 2] >> 16 : a[j / 2] & 0xFFFFu;
            if (k0 + j >= c1) continue;
            if (m >= M) {
                atomicOr(&L.ws.event_err[e_of[j]], kErrBadDigi);
                continue;
            }
            const uint64_t key = (uint64_t)e_of[j] * M + m;
            if (ci.use_sh)
                atomicAdd(&bins[key - ci.keybase], 1u);
            else
                atomicAdd(&L.ws.count2[key], 1u);
        }
    }
    __syncthreads();
    // With few keys (long runs per key) the flush's atomic returns this
    // block's offset inside each key's bucket, and the scatter kernel (over
    // the same ranges) places its digis from there; with many keys the
    // counts go to count2 and the scatter hands out positions step by step,
    // so that blocks running at the same time fill neighbouring positions.
    uint32_t *boffs = L.ws.blk_off + (size_t)blockIdx.x * kHistCap;
    for (uint32_t i = threadIdx.x; i < ci.nkeys; i += kHistThreads) {
        if (sub) {
            uint32_t v = 0;
            for (uint32_t w = 0; w < kHistWarps; ++w) v += sh[w * ci.nkeys + i];
            boffs[i] = v ? atomicAdd(&L.ws.count[ci.keybase + i], v) : 0u;
        } else if (sh[i]) {
            atomicAdd(&L.ws.count2[ci.keybase + i], sh[i]);
        }
    }
}

// ---------------------------------------------------------------- scan

// Per item, count[] holds the digis of histogram blocks with few keys
// (their runs are reserved, by offset, in blk_off) and count2[] those of
// blocks with many keys (placed step by step by the scatter); the scan sets
// boff = the item's bucket start, cursor = the start of the step-by-step
// part (after every reserved run) and count = the item's total.  Items of
// more than cc.large_digis digis are listed for the clustering kernel.
__global__ void __launch_bounds__(256) scan_kernel(const Launch L)
{
    __shared__ uint32_t tmp[256 / 32 + 1];
    pdl_wait();
    pdl_trigger();
    if (L.ws.ctl[1] & kErrBadOffsets) return;
    const uint32_t e = blockIdx.x, M = L.g.M;
    const uint64_t kb = (uint64_t)e * M;
    const uint32_t per = (M + 255) / 256;
    const uint32_t m0 = min(M, threadIdx.x * per), m1 = min(M, m0 + per);
    uint32_t local = 0;
    for (uint32_t m = m0; m < m1; ++m) local += L.ws.count[kb + m] + L.ws.count2[kb + m];
    uint32_t total;
    uint32_t run = block_exclusive_scan<256>(local, tmp, &total) + (uint32_t)L.offsets[e];
    for (uint32_t m = m0; m < m1; ++m) {
        const uint32_t c1 = L.ws.count[kb + m], n = c1 + L.ws.count2[kb + m];
        if (n > L.cc.large_digis) L.ws.large[atomicAdd(&L.ws.ctl[5], 1u)] = (uint32_t)(kb + m);
        L.ws.boff[kb + m] = run;
        L.ws.cursor[kb + m] = run + c1;
        L.ws.count[kb + m] = n;
        run += n;
    }
}

// Digis a thread of the scatter kernel holds where a range has few keys, the
// step of a block there, and the kernel's shared memory (bytes): the staged
// digis with their keys and three words a key, or (many keys) a count and a
// base a key and the next step's digis.
constexpr int kScatPer = 2 * kPerThread;
constexpr uint32_t kScatStep = kHistThreads * kScatPer;
constexpr size_t kScatSort = (size_t)kScatStep * (8 + 2) + 3 * 4 * (kSubKeys + 32);
constexpr size_t kScatDirect = (size_t)kHistCap * 8 + kChunk * (2 + 4);
constexpr size_t kScatterSmem = kScatSort > kScatDirect ? kScatSort : kScatDirect;
static_assert(kSubKeys + 32 <= (uint32_t)kHistThreads && kSubKeys < kChunkEvents, "a key a thread, every offset kept");

// A thread's modules (~0: absent) and words of the step at s0.
__device__ __forceinline__ void load_scatter(const Launch &L, uint64_t s0, uint64_t c1, uint32_t (&m)[kScatPer],
                                             uint32_t (&w)[kScatPer])
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint64_t k0 = s0 + ((uint64_t)h * kHistThreads + threadIdx.x) * kPerThread;
        uint32_t m8[kPerThread], w8[kPerThread];
        load_modules(L, k0, c1, m8);
        load_words(L, k0, c1, w8);
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            m[h * kPerThread + j] = m8[j];
            w[h * kPerThread + j] = w8[j];
        }
    }
}

// The scatter of a block's range [c0, c1) with at most kSubKeys keys: every
// step of kScatStep digis is ranked by key with one shared-memory atomic a
// digi, sorted by key in shared memory, and each key's run is written with
// consecutive threads from the block's offset inside the bucket (reserved by
// the histogram's flush), so no step needs a global atomic.  Bound by
// shared-memory wavefronts (76% of the LSU pipe: rank, place and read back
// each digi, the last two with the bank conflicts of a random order).  Against
// steps of half the size with a histogram a warp and the event looked up for
// every digi: 27.7M digis on 64 modules 153 -> 127 us.  Leaving the keys out
// of the stage, a warp finding the runs of its share, was 124 us there but
// 35 us instead of 30 for 5.8M digis in 48 events.  km and w: the
// first step's modules (then key | rank << 16; 0xFFFF: none) and words, two
// groups of kPerThread a thread.
__device__ __forceinline__ void scatter_few(const Launch &L, uint32_t *sh, const ChunkInfo &ci, const uint64_t *s_off,
                                            uint32_t *s_scan, uint32_t (&km)[kScatPer], uint32_t (&w)[kScatPer])
{
    const uint32_t tid = threadIdx.x, M = L.g.M, nkeys = ci.nkeys;
    uint2 *stage = reinterpret_cast<uint2 *>(sh);                     // [kScatStep] sorted by key
    uint16_t *skey = reinterpret_cast<uint16_t *>(stage + kScatStep); // [kScatStep]
    uint32_t *cnt = reinterpret_cast<uint32_t *>(skey + kScatStep);   // [kSubKeys + 32] digis of a key (and of none)
    uint32_t *lk = cnt + kSubKeys + 32;                               // their start in the stage
    uint32_t *to = lk + kSubKeys + 32;                                // from the stage to the buckets
    uint32_t kg = 0; // thread t: where the next digis of key t go
    if (tid < nkeys) kg = L.ws.boff[ci.keybase + tid] + L.ws.blk_off[(size_t)blockIdx.x * kHistCap + tid];
    if (tid < kSubKeys + 32) cnt[tid] = 0;
    __syncthreads();
    uint32_t es = ci.ef; // event of the step's first digi
    for (uint64_t s0 = ci.c0; s0 < ci.c1; s0 += kScatStep) {
        while (es < ci.el && s_off[es + 1 - ci.ef] <= s0) ++es;
        const bool one = es == ci.el || s_off[es + 1 - ci.ef] >= min(ci.c1, s0 + kScatStep);
        const bool both = s0 + kScatStep / 2 < ci.c1; // the second groups hold digis
        const uint32_t ekey = (es - ci.ef) * M;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h && !both) continue;
            uint32_t *x = km + h * kPerThread, rank[kPerThread];
            uint32_t e_of[kPerThread];
            if (!one) digi_events(L, s_off, ci.ef, ci.el, s0 + ((uint64_t)h * kHistThreads + tid) * kPerThread, e_of);
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) // (an absent digi's module is ~0)
                x[j] = x[j] < M ? (one ? ekey : (e_of[j] - ci.ef) * M) + x[j] : 0xFFFFu;
            // (no branches, so that the atomics' latencies overlap)
#pragma unroll
            for (int j = 0; j < kPerThread; ++j)
                rank[j] = atomicAdd(&cnt[x[j] == 0xFFFFu ? kSubKeys + (tid & 31) : x[j]], 1u);
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) x[j] |= x[j] == 0xFFFFu ? 0u : rank[j] << 16;
        }
        __syncthreads();
        const uint32_t tot = tid < nkeys ? cnt[tid] : 0u;
        uint32_t total;
        const uint32_t start = block_exclusive_scan<kHistThreads>(tot, s_scan, &total);
        if (tid < kSubKeys + 32) {
            lk[tid] = start;
            to[tid] = kg - start;
            cnt[tid] = 0;
            kg += tot;
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t k0 = s0 + ((uint64_t)h * kHistThreads + tid) * kPerThread;
            if (h && !both) continue;
            const uint32_t *x = km + h * kPerThread;
            uint32_t e_of[kPerThread];
            if (!one) digi_events(L, s_off, ci.ef, ci.el, k0, e_of);
            const uint32_t i0 = (uint32_t)(k0 - s_off[es - ci.ef]);
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) {
                const uint32_t key = x[j] & 0xFFFFu;
                if (key == 0xFFFFu) continue;
                const uint32_t p = lk[key] + (x[j] >> 16);
                stage[p] = make_uint2(w[h * kPerThread + j],
                                      one ? i0 + j : (uint32_t)(k0 + j - s_off[e_of[j] - ci.ef]));
                skey[p] = (uint16_t)key;
            }
        }
        __syncthreads();
        if (s0 + kScatStep < ci.c1) load_scatter(L, s0 + kScatStep, ci.c1, km, w); // (in flight while this step is written out)
#pragma unroll 4
        for (uint32_t p = tid; p < total; p += kHistThreads) L.ws.bucket[to[skey[p]] + p] = stage[p];
    }
}

// Scatter, persistent, over the histogram kernel's ranges: block b walks its
// range (one event search a block).  With few keys scatter_few.  With many
// keys, in steps of kChunk digis (the next step's words and module ids are
// loaded while the current step is written out, cp.async), one global atomic
// per key and step hands out the positions (after the reserved runs), and each
// digi goes straight to its place; a range with more keys than a shared
// histogram holds takes one atomic per digi.
__global__ void __launch_bounds__(kHistThreads, 2) scatter_kernel(const __grid_constant__ Launch L)
{
    extern __shared__ __align__(16) uint32_t sh[];
    pdl_wait();
    pdl_trigger();
    uint32_t *cnt = sh;             // digis of each key
    uint32_t *bas = sh + kHistCap;  // and its base
    __shared__ uint32_t s_ev[2];
    __shared__ uint64_t s_off[kChunkEvents + 1];
    __shared__ uint32_t s_scan[kHistThreads / 32 + 1];
    // next step's module ids and words (16-byte aligned for cp.async)
    uint16_t *pf_m = reinterpret_cast<uint16_t *>(bas + kHistCap);
    uint32_t *pf_w = reinterpret_cast<uint32_t *>(pf_m + kChunk);
    if (L.ws.ctl[1] & kErrBadOffsets) return;
    uint64_t c0, c1;
    block_range(L.N, blockIdx.x, gridDim.x, &c0, &c1);
    if (c0 >= c1) return;
    // the first digis are loaded before the event search, so that the two
    // latencies overlap
    uint32_t m0[kScatPer], w0[kScatPer];
    load_scatter(L, c0, c1, m0, w0);
    const ChunkInfo ci = chunk_info<>(L, c0, c1, s_ev, s_off);
    const uint32_t M = L.g.M;
    if (ci.use_sh && ci.nkeys <= kSubKeys) { // (uniform)
        __syncthreads();                     // s_off
        scatter_few(L, sh, ci, s_off, s_scan, m0, w0);
        return;
    }
    uint64_t k0 = c0 + (uint64_t)threadIdx.x * kPerThread;
    uint32_t m[kPerThread], e_of[kPerThread], w[kPerThread], rank[kPerThread];
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) m[j] = m0[j], w[j] = w0[j];
    const bool off_sh = ci.el - ci.ef + 1 < kChunkEvents;
    auto event_start = [&](uint32_t e) -> uint64_t { return off_sh ? s_off[e - ci.ef] : L.offsets[e]; };
    for (uint64_t s0 = c0;; s0 += kChunk, k0 += kChunk) {
        for (uint32_t i = threadIdx.x; i < ci.nkeys; i += kHistThreads) cnt[i] = 0;
        __syncthreads();
        const bool more = s0 + kChunk < c1; // another step follows
        const bool pf = more && prefetch_digis(L, k0 + kChunk, c1, pf_m, pf_w);
        digi_events(L, s_off, ci.ef, ci.el, k0, e_of);
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            const bool ok = k0 + j < ci.c1 && m[j] < M;
            if (!ok) {
                m[j] = 0xFFFFFFFFu;
                continue;
            }
            const uint64_t key = (uint64_t)e_of[j] * M + m[j];
            rank[j] = ci.use_sh ? atomicAdd(&cnt[key - ci.keybase], 1u) : atomicAdd(&L.ws.cursor[key], 1u);
        }
        __syncthreads();
        // (four atomics a thread in flight: 1.48M digis on 1,856 modules 22.5 -> 20.5 us)
        for (uint32_t i = threadIdx.x; i < ci.nkeys; i += 4 * kHistThreads) {
            uint32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = i + u * kHistThreads < ci.nkeys ? cnt[i + u * kHistThreads] : 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (v[u]) v[u] = atomicAdd(&L.ws.cursor[ci.keybase + i + u * kHistThreads], v[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * kHistThreads < ci.nkeys) bas[i + u * kHistThreads] = v[u];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            if (m[j] == 0xFFFFFFFFu) continue;
            const uint64_t key = (uint64_t)e_of[j] * M + m[j];
            const uint32_t p = ci.use_sh ? bas[key - ci.keybase] + rank[j] : rank[j];
            L.ws.bucket[p] = make_uint2(w[j], (uint32_t)(k0 + j - event_start(e_of[j])));
        }
        __syncthreads();
        if (!more) break;
        if (pf) {
            take_prefetched(pf_m, pf_w, m, w);
        } else {
            load_modules(L, k0 + kChunk, c1, m);
            load_words(L, k0 + kChunk, c1, w);
        }
    }
}

// Scatter for many modules (more than kSubKeys, so that every histogram block
// counted into count2), persistent: a block sorts kWideStep digis at a time by
// key in shared memory, takes each key's positions with one global atomic and
// writes each key's run with consecutive threads.  Against scatter_kernel's
// step of 4,096 digis, whose digis land nearly alone (2.2 a key for 1,856
// modules), a run is 8.8 digis: a third of the sectors and a quarter of the
// atomics (29.4M digis in 8 events: 281 -> 183 us; 171 us with the digis'
// events looked up only in steps over several).  Bound by shared-memory
// wavefronts (rank, placing and reading back each digi; half of their peak,
// one block an SM) and by L2 writes; a thread's 32 digi words and keys spill in
// part (64 registers a thread: 180 bytes of stores, 156 of loads).  A step over
// more keys than the tables hold takes one atomic a digi, as scatter_kernel
// does.
constexpr int kWideThreads = 1024;
constexpr int kWidePer = 2 * kPerThread;                // digis a thread holds
constexpr uint32_t kWideStep = kWideThreads * kWidePer; // digis a block sorts at a time
constexpr size_t kWideSmem = (size_t)kWideStep * (8 + 2) + 4 * (3 * (size_t)kHistCap + 32);

__global__ void __launch_bounds__(kWideThreads, 1) scatter_wide_kernel(const __grid_constant__ Launch L)
{
    extern __shared__ __align__(16) uint32_t sh[];
    __shared__ uint32_t tmp[kWideThreads / 32 + 1];
    __shared__ uint32_t s_ev[2];
    __shared__ uint64_t s_off[kChunkEvents + 1];
    pdl_wait();
    pdl_trigger();
    if (L.ws.ctl[1] & kErrBadOffsets) return;
    const uint32_t tid = threadIdx.x, M = L.g.M;
    uint2 *stage = reinterpret_cast<uint2 *>(sh);                     // [kWideStep] sorted by key
    uint16_t *skey = reinterpret_cast<uint16_t *>(stage + kWideStep); // [kWideStep]
    uint32_t *cnt = reinterpret_cast<uint32_t *>(skey + kWideStep);   // [kHistCap + 32] digis of a key (and of none)
    uint32_t *lk = cnt + kHistCap + 32;                               // [kHistCap] their start in the stage
    uint32_t *to = lk + kHistCap;                                     // [kHistCap] from the stage to the buckets
    static_assert(kHistCap <= 4 * kWideThreads, "four keys a thread");
    // all event offsets in shared memory when they fit, else a step's
    const bool all_off = L.E < kChunkEvents;
    if (all_off)
        for (uint32_t i = tid; i <= L.E; i += kWideThreads) s_off[i] = L.offsets[i];
    // km: key, then key | rank << 16 (0xFFFF: none); the thread's digis are two
    // groups of kPerThread
    uint32_t km[kWidePer], w[kWidePer];
    auto load_step = [&](uint64_t s0) {
        const uint64_t c1 = min(L.N, s0 + kWideStep);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t k0 = s0 + ((uint64_t)h * kWideThreads + tid) * kPerThread;
            uint32_t m8[kPerThread], w8[kPerThread];
            load_modules(L, k0, c1, m8);
            load_words(L, k0, c1, w8);
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) {
                km[h * kPerThread + j] = m8[j];
                w[h * kPerThread + j] = w8[j];
            }
        }
    };
    const uint64_t first = (uint64_t)blockIdx.x * kWideStep, stride = (uint64_t)gridDim.x * kWideStep;
    if (first < L.N) load_step(first);
    __syncthreads();
    for (uint64_t s0 = first; s0 < L.N; s0 += stride) {
        const uint64_t c1 = min(L.N, s0 + kWideStep);
        for (uint32_t i = tid; i < (uint32_t)kHistCap; i += kWideThreads) cnt[i] = 0;
        ChunkInfo ci;
        if (all_off) {
            if (tid < 32) {
                const uint32_t ef = find_event_warp(s_off, 0, L.E - 1, s0);
                const uint32_t el = find_event_warp(s_off, ef, L.E - 1, c1 - 1);
                if (tid == 0) {
                    s_ev[0] = ef;
                    s_ev[1] = el;
                }
            }
            __syncthreads();
            ci.ef = s_ev[0];
            ci.el = s_ev[1];
            ci.use_sh = (uint64_t)(ci.el - ci.ef + 1) * M <= (uint64_t)kHistCap;
            ci.keybase = (uint64_t)ci.ef * M;
        } else {
            ci = chunk_info<kWideThreads>(L, s0, c1, s_ev, s_off);
            __syncthreads();
        }
        const uint64_t *off = all_off ? s_off + ci.ef : s_off; // of event ef on
        if (!ci.use_sh) { // (uniform)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint64_t k0 = s0 + ((uint64_t)h * kWideThreads + tid) * kPerThread;
                uint32_t e_of[kPerThread];
                digi_events(L, off, ci.ef, ci.el, k0, e_of);
#pragma unroll
                for (int j = 0; j < kPerThread; ++j) {
                    const uint32_t m = km[h * kPerThread + j];
                    if (k0 + j >= c1 || m >= M) continue;
                    const uint32_t p = atomicAdd(&L.ws.cursor[(uint64_t)e_of[j] * M + m], 1u);
                    L.ws.bucket[p] = make_uint2(w[h * kPerThread + j], (uint32_t)(k0 + j - L.offsets[e_of[j]]));
                }
            }
            if (s0 + stride < L.N) load_step(s0 + stride);
            __syncthreads();
            continue;
        }
        // whether the step lies in one event, which then no digi looks for
        const bool one = ci.ef == ci.el;
        // rank of each digi among its key's (no branches, so that the atomics'
        // latencies overlap)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t *x = km + h * kPerThread, rank[kPerThread];
            if (!one) {
                uint32_t e_of[kPerThread];
                digi_events(L, off, ci.ef, ci.el, s0 + ((uint64_t)h * kWideThreads + tid) * kPerThread, e_of);
#pragma unroll
                for (int j = 0; j < kPerThread; ++j) x[j] = x[j] < M ? (e_of[j] - ci.ef) * M + x[j] : 0xFFFFu;
            }
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) { // (an absent digi's module is ~0)
                x[j] = x[j] < (one ? M : 0xFFFFu) ? x[j] : 0xFFFFu;
                rank[j] = atomicAdd(&cnt[x[j] == 0xFFFFu ? (uint32_t)kHistCap + (tid & 31) : x[j]], 1u);
            }
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) x[j] |= x[j] == 0xFFFFu ? 0u : rank[j] << 16;
        }
        __syncthreads();
        uint32_t total;
        {
            const uint32_t k = 4 * tid;
            const uint4 c = *reinterpret_cast<const uint4 *>(cnt + k);
            // (the atomics' latency overlaps the scan)
            const uint32_t cs[4] = {c.x, c.y, c.z, c.w};
            uint32_t g[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) g[i] = cs[i] ? atomicAdd(&L.ws.cursor[ci.keybase + k + i], cs[i]) : 0u;
            const uint32_t l0 = block_exclusive_scan<kWideThreads>(c.x + c.y + c.z + c.w, tmp, &total);
            const uint32_t l1 = l0 + c.x, l2 = l1 + c.y, l3 = l2 + c.z;
            *reinterpret_cast<uint4 *>(lk + k) = make_uint4(l0, l1, l2, l3);
            *reinterpret_cast<uint4 *>(to + k) = make_uint4(g[0] - l0, g[1] - l1, g[2] - l2, g[3] - l3);
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t k0 = s0 + ((uint64_t)h * kWideThreads + tid) * kPerThread;
            const uint32_t *x = km + h * kPerThread;
            uint32_t e_of[kPerThread];
            if (!one) digi_events(L, off, ci.ef, ci.el, k0, e_of);
            const bool off_sh = all_off || ci.el - ci.ef + 1 < kChunkEvents;
            const uint32_t i0 = (uint32_t)(k0 - off[0]);
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) {
                const uint32_t key = x[j] & 0xFFFFu;
                if (key == 0xFFFFu) continue;
                const uint32_t p = lk[key] + (x[j] >> 16);
                uint32_t index = i0 + j;
                if (!one) index = (uint32_t)(k0 + j - (off_sh ? off[e_of[j] - ci.ef] : L.offsets[e_of[j]]));
                stage[p] = make_uint2(w[h * kPerThread + j], index);
                skey[p] = (uint16_t)key;
            }
        }
        __syncthreads();
        if (s0 + stride < L.N) load_step(s0 + stride); // (in flight while this step is written out)
#pragma unroll 4
        for (uint32_t p = tid; p < total; p += kWideThreads) L.ws.bucket[to[skey[p]] + p] = stage[p];
        __syncthreads();
    }
}

// ---------------------------------------------------------------- bucketing of small launches

// bucket_kernel: histogram, scan and scatter in one, for launches of few
// digis: a thread-block cluster an event, each of its blocks a contiguous
// slice of the event.  Every block counts its slice by module in shared
// memory; after a cluster barrier each reads the others' counts (distributed
// shared memory, four modules a load) and so knows, for every module, the
// bucket's start and its own offset inside it; then it sorts its digis by
// module in shared memory and writes each module's run with consecutive
// threads.  A slice is at most kBucketStep digis, a step a block.  Where no
// event has more than kBucketDigis (the host knows the largest) a cluster has
// an event.  Else (L.bucket_parts) a larger event is split evenly among
// several, and each counts the others' parts as well, before its own and after
// it, so that no cluster waits for another (17 us where no event is split, 21
// with two parts, 25 with four; one cluster in two and four steps took 30 and
// 49).  With one event the kernel also clears the launch's control words, so
// that nothing precedes it.  Bound by launch and global-memory latency: one
// launch in place of a memset and three kernels.
constexpr int kBucketThreads = 1024;
constexpr int kBucketCluster = 8;                             // portable cluster size
constexpr int kBucketPer = 2 * kPerThread;                    // digis a thread holds
constexpr uint32_t kBucketStep = kBucketThreads * kBucketPer; // digis a block sorts

// Lines of the small launches (bucket_fits, finish_fits).
constexpr uint64_t kSmallDigis = 1u << 21;   // digis of a launch that finish_kernel ends
constexpr uint64_t kSmallHost = 1u << 19;    // the same with outputs in host memory, bucket_kernel not before it
constexpr uint64_t kBucketTotal = 1u << 20;  // digis of a launch of more events that bucket_kernel starts
constexpr uint32_t kBucketAtOnce = 15;       // its clusters that run at once (of 19: eight blocks of a GPC each)
constexpr uint32_t kBucketModules = 2048;    // modules (three or five words each in shared memory)
// largest event: a step a block, wherever the event starts (its groups of
// kPerThread digis are up to two more than its digis fill)
constexpr uint64_t kBucketDigis = kBucketCluster * (kBucketStep - kPerThread);
static_assert(kBucketDigis / kPerThread + 2 <= kBucketCluster * (kBucketStep / kPerThread), "a step a block");
constexpr uint32_t kFinishItems = 16384;     // (event, module) items every block scans

__host__ __device__ constexpr uint32_t bucket_keys(uint32_t M) { return (M + 3) & ~3u; }
__host__ __device__ constexpr size_t bucket_smem(uint32_t M, bool parts)
{
    return (size_t)kBucketStep * (8 + 2) + (size_t)bucket_keys(M) * (parts ? 5 : 3) * 4;
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// Four words at this block's shared address a, in block r of the cluster.
__device__ __forceinline__ uint4 lds_cluster4(uint32_t a, uint32_t r)
{
    uint4 v;
    asm volatile("{\n\t"
                 ".reg .u32 ra;\n\t"
                 "mapa.shared::cluster.u32 ra, %4, %5;\n\t"
                 "ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [ra];\n\t"
                 "}" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a), "r"(r) : "memory");
    return v;
}

template <bool kParts>
__global__ void __launch_bounds__(kBucketThreads, 1) bucket_kernel(const __grid_constant__ Launch L)
{
    extern __shared__ __align__(16) uint32_t sh[];
    __shared__ uint32_t tmp[2][kBucketThreads / 32 + 1];
    __shared__ uint32_t s_bad, s_none[32];
    pdl_trigger();
    const uint32_t tid = threadIdx.x, M = L.g.M, MK = bucket_keys(M), rank = cluster_rank();
    uint32_t e = blockIdx.x / kBucketCluster, part = 0, parts = 1; // the cluster's event, and which part of it
    if constexpr (kParts) {
        __shared__ uint32_t s_place[3];
        if (tid < 32) { // (at most 32 events; offsets that do not fit are found below, by the first event they spoil)
            const uint64_t a = tid < L.E ? L.offsets[tid] : 0, b = tid < L.E ? L.offsets[tid + 1] : 0;
            const bool fit = a < b && b <= L.N;
            const uint32_t n = tid >= L.E ? 0u : fit ? (uint32_t)((b - a + kBucketDigis - 1) / kBucketDigis) : 1u;
            uint32_t incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, o);
                if ((int)tid >= o) incl += y;
            }
            const uint32_t past = __ballot_sync(kFull, incl > e), at = past ? __ffs(past) - 1 : 0u;
            const uint32_t first = __shfl_sync(kFull, incl - n, at), of = __shfl_sync(kFull, n, at);
            if (tid == 0) {
                s_place[0] = past ? at : ~0u;
                s_place[1] = e - first;
                s_place[2] = of;
            }
        }
        __syncthreads();
        if (s_place[0] == ~0u) return; // (the whole cluster: every event has its clusters already)
        e = s_place[0];
        part = s_place[1];
        parts = s_place[2];
    }
    uint2 *stage = reinterpret_cast<uint2 *>(sh);                       // [kBucketStep] sorted by module
    uint16_t *skey = reinterpret_cast<uint16_t *>(stage + kBucketStep); // [kBucketStep]
    uint32_t *hist = reinterpret_cast<uint32_t *>(skey + kBucketStep);  // [MK] digis of the slice
    uint32_t *lk = hist + MK;                                           // [MK] their start in the stage
    uint32_t *gb = lk + MK;                                             // [MK] their first bucket position
    uint32_t *rest = gb + MK; // [2 * MK] (with parts) digis of the parts before this one, and of those after
    for (uint32_t k = tid; k < MK; k += kBucketThreads) hist[k] = 0;
    if (kParts && parts > 1)
        for (uint32_t k = tid; k < 2 * MK; k += kBucketThreads) rest[k] = 0;
    if (tid == 0) s_bad = 0;
    const uint64_t o0 = L.offsets[e], o1 = L.offsets[e + 1];
    const bool bad_offsets = o0 > o1 || o1 > L.N || (e == 0 && o0 != 0) || (e == L.E - 1 && o1 != L.N);
    if (L.E == 1 && rank == 0) { // otherwise cleared before the launch
        if (tid < 16) L.ws.ctl[tid] = tid == 1 && bad_offsets ? kErrBadOffsets : 0u;
        if (tid == 16) L.ws.event_err[0] = 0;
    }
    if (bad_offsets) { // uniform over the cluster
        if (L.E > 1 && rank == 0 && tid == 0) atomicOr(&L.ws.ctl[1], kErrBadOffsets);
        return;
    }
    // the slice [c0, c1), cut at multiples of kPerThread digis of the launch
    // (so that every thread's groups of digis are 16-byte aligned)
    const uint64_t g0 = o0 / kPerThread, ng = (o1 + kPerThread - 1) / kPerThread - g0;
    const uint32_t slices = kParts ? parts * kBucketCluster : kBucketCluster;
    auto cut = [&](uint32_t p) { return (g0 + ng * (p * kBucketCluster + rank) / slices) * kPerThread; };
    auto end = [&](uint32_t p) { return (g0 + ng * (p * kBucketCluster + rank + 1) / slices) * kPerThread; };
    const uint64_t a0 = cut(part), c0 = max(o0, a0), c1 = min(o1, end(part));
    // whether the second group of a thread's digis holds any: an event of at
    // most half a step a block does without it (30,000 digis: 30.9 -> 25.4 us)
    const bool both = c1 > a0 + kBucketStep / 2;
    // a thread's digis: group h at a0 + (h * threads + tid) * kPerThread;
    // km: module, then (counted) module | rank << 16; 0xFFFF: none
    uint32_t km[kBucketPer], w[kBucketPer];
    auto first = [&](int h) { return a0 + ((uint64_t)h * kBucketThreads + tid) * kPerThread; };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint64_t k0 = first(h);
        uint32_t m8[kPerThread] = {}, w8[kPerThread] = {};
        if (h == 0 || both) {
            load_modules(L, k0, c1, m8);
            load_words(L, k0, c1, w8);
        }
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            const bool in = k0 + j >= c0 && k0 + j < c1;
            km[h * kPerThread + j] = in ? m8[j] : 0xFFFFFFFFu;
            w[h * kPerThread + j] = w8[j];
        }
    }
    __syncthreads();
    bool bad = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) { // (no branches: the latencies overlap; 60,000 digis: 32.9 -> 30.9 us)
        if (h && !both) {
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) km[kPerThread + j] = 0xFFFFu;
            continue;
        }
        uint32_t r[kPerThread];
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            const uint32_t k = km[h * kPerThread + j];
            r[j] = atomicAdd(k < M ? hist + k : s_none + (tid & 31), 1u);
        }
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            uint32_t &k = km[h * kPerThread + j];
            bad |= k >= M && k != 0xFFFFFFFFu;
            k = k < M ? k | (r[j] << 16) : 0xFFFFu;
        }
    }
    if (bad) s_bad = 1;
    for (uint32_t p = 0; kParts && p < parts; ++p) { // this block's slice of the event's other parts
        if (p == part) continue;
        const uint64_t b0 = cut(p), b1 = min(o1, end(p));
        uint32_t *counts = p < part ? rest : rest + MK;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t k0 = b0 + ((uint64_t)h * kBucketThreads + tid) * kPerThread;
            uint32_t m8[kPerThread];
            load_modules(L, k0, b1, m8);
#pragma unroll
            for (int j = 0; j < kPerThread; ++j)
                if (k0 + j >= o0 && k0 + j < b1 && m8[j] < M) atomicAdd(counts + m8[j], 1u);
        }
    }
    cluster_arrive();
    cluster_wait();
    if (tid == 0 && s_bad) atomicOr(&L.ws.event_err[e], kErrBadDigi);
    // every module's bucket, and this block's offset inside it: four modules a thread
    static_assert(kBucketModules <= 4 * kBucketThreads, "four modules a thread");
    uint32_t total; // digis in the stage
    {
        const uint32_t k = 4 * tid;
        uint4 t = make_uint4(0, 0, 0, 0), before = t, own = t;
        if (k < MK) {
            const uint32_t ha = (uint32_t)__cvta_generic_to_shared(hist + k);
            uint4 v[kBucketCluster];
#pragma unroll
            for (uint32_t r = 0; r < kBucketCluster; ++r) v[r] = lds_cluster4(ha, r);
#pragma unroll
            for (uint32_t r = 0; r < kBucketCluster; ++r) {
                t.x += v[r].x, t.y += v[r].y, t.z += v[r].z, t.w += v[r].w;
                if (r < rank) before.x += v[r].x, before.y += v[r].y, before.z += v[r].z, before.w += v[r].w;
                if (r == rank) own = v[r];
            }
            if (kParts && parts > 1) {
                const uint32_t ra = (uint32_t)__cvta_generic_to_shared(rest + k);
#pragma unroll
                for (uint32_t r = 0; r < kBucketCluster; ++r) {
                    const uint4 b = lds_cluster4(ra, r), a = lds_cluster4(ra + 4 * MK, r);
                    before.x += b.x, before.y += b.y, before.z += b.z, before.w += b.w;
                    t.x += a.x + b.x, t.y += a.y + b.y, t.z += a.z + b.z, t.w += a.w + b.w;
                }
            }
        }
        cluster_arrive(); // the others' counts are read
        uint32_t unused;
        uint32_t run = block_exclusive_scan<kBucketThreads>(t.x + t.y + t.z + t.w, tmp[0], &unused) + (uint32_t)o0;
        const uint32_t mine = block_exclusive_scan<kBucketThreads>(own.x + own.y + own.z + own.w, tmp[1], &total);
        if (k < MK) {
            const uint4 b = make_uint4(run, run + t.x, run + t.x + t.y, run + t.x + t.y + t.z);
            *reinterpret_cast<uint4 *>(gb + k) =
                make_uint4(b.x + before.x, b.y + before.y, b.z + before.z, b.w + before.w);
            *reinterpret_cast<uint4 *>(lk + k) =
                make_uint4(mine, mine + own.x, mine + own.x + own.y, mine + own.x + own.y + own.z);
            if (rank == 0 && part == 0) {
                const uint32_t bs[4] = {b.x, b.y, b.z, b.w}, ts[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                for (uint32_t i = 0; i < 4; ++i) {
                    if (k + i >= M) break;
                    const uint64_t item = (uint64_t)e * M + k + i;
                    L.ws.count[item] = ts[i];
                    L.ws.boff[item] = bs[i];
                    if (ts[i] > L.cc.large_digis) L.ws.large[atomicAdd(&L.ws.ctl[5], 1u)] = (uint32_t)item;
                }
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kBucketPer; ++j) {
        const uint32_t key = km[j] & 0xFFFFu;
        if (key == 0xFFFFu) continue;
        const uint32_t p = lk[key] + (km[j] >> 16);
        stage[p] = make_uint2(w[j], (uint32_t)(first(j / kPerThread) + j % kPerThread - o0));
        skey[p] = (uint16_t)key;
    }
    __syncthreads();
    for (uint32_t p = tid; p < total; p += kBucketThreads) {
        const uint32_t key = skey[p];
        L.ws.bucket[gb[key] + (p - lk[key])] = stage[p];
    }
    cluster_wait(); // the others have read this block's counts
}

// ---------------------------------------------------------------- clustering

// Moments accumulate in 32 bits: sum(q * col) and sum(q * (row - root row))
// cannot overflow while Q <= INT32_MAX / 512 (row < 256, col < 512).  Items
// with a heavier cluster recompute them in 64 bits.
constexpr int32_t kQSafe32 = 0x7FFFFFFF / 512;
constexpr uint32_t kNoSlot = 0xFFFFFFFFu;

// Barrier of the `threads` threads of one group (named barrier `id` >= 1;
// barrier 0 is the block's __syncthreads).  The compiler's own builtin, not
// inline assembly: like __syncthreads it is convergent, so the compiler
// never duplicates it into paths that a warp's threads take apart.
__device__ __forceinline__ void group_sync(uint32_t id, uint32_t threads)
{
    __syncwarp();
    __barrier_sync_count(id, threads);
}

// Centroid coordinate sum / Q from an exact, non-negative moment: one float
// division when both are exact in float (the correctly rounded quotient),
// else integer quotient plus the remainder fraction, so the float result is
// within a few ulps whatever the magnitude.  The integer quotient (below 512:
// a row or a column) comes from a float estimate and the remainder's sign.
__device__ __forceinline__ float centroid_abs(uint32_t sum, uint32_t Q)
{
    uint32_t qt = 0, rem = sum;
    if (sum >= 16777216u || Q >= 16777216u) {
        qt = (uint32_t)__fdividef((float)sum, (float)Q);
        rem = sum - qt * Q;
        if ((int32_t)rem < 0) {
            --qt;
            rem += Q;
        } else if (rem >= Q) {
            ++qt;
            rem -= Q;
        }
    }
    return (float)qt + (float)rem / (float)Q;
}
__device__ __forceinline__ float centroid_abs(long long sum, int32_t Q)
{
    if (sum < 0x80000000LL) return centroid_abs((uint32_t)sum, (uint32_t)Q);
    const long long qt = sum / Q;
    return (float)qt + (float)(sum - qt * Q) / (float)Q;
}

// Static shared memory of one group of threads that clusters items on its
// own (GT threads: its own named barrier, its own tickets).
struct GroupShared {
    uint32_t ticket;
    uint32_t flag;                 // run tier: an invalid digi; packed tier: bit i: the pack's item i is faulty
    uint32_t heavy, pixels, extras;
    uint32_t bucket_end;           // end of the ticket's buckets
    uint32_t pack_end;             // packed tier: end of the planned pack (an item of the ticket); run tier: scratch slot
    uint32_t tmp[32];              // scans; packed tier: kept clusters of each item
    uint32_t n[kGroup], b[kGroup]; // digis and bucket start of the ticket's items
    ItemRec rec[kGroup];
    uint16_t pack[kGroup + 1];     // packed tier: first packed digi of each item, and the total
};
static_assert(kWholeBytes + sizeof(GroupShared) * kRunGroups1 + kRunThreads1 / 32 * 128 <= 227 * 1024,
              "the largest tile beside a block's static memory");

template <int GT, bool kWhole>
__device__ __forceinline__ void gsync(uint32_t bar)
{
    if constexpr (kWhole)
        __syncthreads();
    else
        group_sync(bar, GT);
}

// Exclusive scan of one value per thread over the group, with one barrier:
// every thread's accesses before the call are visible to the group after it.
template <int GT, bool kWhole>
__device__ __forceinline__ uint32_t group_exclusive_scan(uint32_t v, uint32_t *tmp, uint32_t gt, uint32_t bar,
                                                         uint32_t *total)
{
    constexpr int kWarps = GT / 32;
    const uint32_t lane = gt & 31, warp = gt >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, o);
        if ((int)lane >= o) x += y;
    }
    if (lane == 31) tmp[warp] = x;
    gsync<GT, kWhole>(bar);
    const uint32_t wt = lane < kWarps ? tmp[lane] : 0u;
    uint32_t ws = wt;
#pragma unroll
    for (int o = 1; o < kWarps; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, ws, o);
        if ((int)lane >= o) ws += y;
    }
    *total = __shfl_sync(kFull, ws, kWarps - 1);
    return __shfl_sync(kFull, ws - wt, warp) + x - v;
}

// Shared memory by 32-bit address, with the byte offset as an immediate: the
// run tier's records are five words, and with one address a record all its
// fields cost no further address arithmetic.
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
template <int kOff = 0>
__device__ __forceinline__ uint32_t lds(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(kOff) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
template <int kOff = 0>
__device__ __forceinline__ void sts(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u32 [%0+%1], %2;" ::"r"(a), "n"(kOff), "r"(v) : "memory");
}
template <int kOff = 0>
__device__ __forceinline__ void reds_add(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0+%1], %2;" ::"r"(a), "n"(kOff), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ uint32_t atoms_or(uint32_t a, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.shared.or.b32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void reds_or(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atoms_min(uint32_t a, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.shared.min.u32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(v) : "memory");
    return old;
}

// ---- run tier
//
// One item by a group of GT threads on a survivor bitmap whose rows start at
// word boundaries (W = ceil(C / 32) words a row).  The unit of the union-find
// and of the sums is the run: a maximal stretch of surviving pixels inside
// one bitmap word.  Runs are numbered in word order, which is row-major
// order, so the smallest run of a cluster holds its smallest linear index
// (the id), and the runs of the row above that touch a run are consecutive.
// Phases, one group barrier between them:
//   1 the item's words; both bitmaps cleared
//   2 a bit per digi, in one of two bitmaps (survivors, the others); a digi
//     whose pixel is taken is found by counting: the pixels set in either must
//     be as many as the digis
//   3 runs per word by a scan over the words; run records initialised (they
//     lie over the bitmap of the dropped digis, free from here on)
//   4 every survivor adds its ADC and ADC * bit to its run, both in one word
//     (at most 32 pixels of 255: 13 and 17 bits); a run's first pixel stores
//     the run's position
//   5 a run works its charge and sum q * col out from these (its pixels'
//     calibration and columns are its own), and links itself, by a plain store, under the first run above that
//     it touches (or the run that ends the word to its left); runs with
//     further contacts (one in ten or so) go to a list
//   6 the listed runs are united with those, by find and link
//   7 every run finds its root and adds its sums to it
//   8 the position of the root into every run (the label of its digis);
//     kept roots counted
//   9 labels of the digis; kept roots staged in run (= id) order
//
// What bounds it: instruction issue and the latency of shared memory; an item
// is a chain of ten barriers, so several groups a block work on items of
// their own, every phase issues its loads two digis or two runs at a time,
// and the frequent conditions are predicates, not branches.  Runs, not
// pixels, are the nodes because there are 0.6 of them a digi in blob-like
// data (0.5 to 0.8): against a node and four atomics a pixel (the tier this
// replaced) a pixel needs no rank and two atomics, and a run looks at one word
// above it instead of eight pixels.  27.7M digis in 16,384 items: 24 -> 14
// warp instructions a digi, 934 -> 514 us; 29.4M digis in 14,848 items with
// 13,000-digi ones among them: 1,374 -> 570 us (its records are 20 bytes, so
// these fit a block's shared memory now).  Of 146 us for 7.0M digis (57% of
// the issue slots and 60% of the LSU pipe in use): labels and root positions
// 31, links and unions 26, sums over runs 13, staging 13, pixel sums 11, the
// bits 8, first runs and records 6, their scan 3, clearing 2, tickets and packs
// the rest.
//
// Run records:
//   word 0  union-find parent
//   word 1  row | col << 8 of the first pixel (the digi word's layout), its
//           length << 17, and in the packed tier its item << 23; from phase 8
//           on the root's position and item, and a flag
//   word 2  the sum of phase 4; then the ADC sum and << 20 the pixels, of the
//           run, then (roots) of the cluster: Q = gain * ADC - ped * pixels
//   word 3  sum q * col, the same way
//   word 4  the list of phase 5; then (roots) sum q * (row - root's row);
//           with compact labels at last the ordinal
// Items of up to kNarrowDigis digis, whose sums fit word 2, in shared memory
// (kNarrow).  Larger ones keep the charge in word 2 and the pixels below the
// parent in word 0, or with records in global scratch (kGlobal) in a word of
// their own.
constexpr int kRunDigis = 8; // digis a thread holds at once
constexpr uint32_t kRunShift = 18, kRunPixels = (1u << kRunShift) - 1u; // kWide: parent << 18 | pixels
constexpr uint32_t kAdcBits = 20, kAdcMask = (1u << kAdcBits) - 1u;       // kNarrow: ADC sum | pixels << 20
constexpr uint32_t kNarrowDigis = 4095;
static_assert(kNarrowDigis * 255u <= kAdcMask && kNarrowDigis < 1u << (32 - kAdcBits), "word 2 of kNarrow");
enum RunKind { kNarrow, kWide, kGlobal };
constexpr uint32_t kRunKept = 1u << 31, kRunDropped = 1u << 30, kRunPos = 0x1FFFFu;
constexpr uint32_t kRunItem = 15u << 23; // packed tier: the run's item

template <RunKind kKind>
struct Runs { // kNarrow and kWide: shared memory
    uint32_t base;
    using At = uint32_t;
    __device__ __forceinline__ At at(uint32_t i) const { return base + i * (uint32_t)kRunBytes; }
    template <int f>
    __device__ __forceinline__ static uint32_t ld(At a) { return lds<4 * f>(a); }
    template <int f>
    __device__ __forceinline__ static void st(At a, uint32_t v) { sts<4 * f>(a, v); }
    template <int f>
    __device__ __forceinline__ static void red(At a, uint32_t v) { reds_add<4 * f>(a, v); }
    __device__ __forceinline__ uint32_t parent(uint32_t i) const
    {
        return kKind == kWide ? ld<0>(at(i)) >> kRunShift : ld<0>(at(i));
    }
    __device__ __forceinline__ void set_parent(uint32_t i, uint32_t p) const
    {
        st<0>(at(i), kKind == kWide ? p << kRunShift : p);
    }
    __device__ __forceinline__ uint32_t min_parent(uint32_t i, uint32_t p) const
    {
        return kKind == kWide ? atoms_min(at(i), p << kRunShift) >> kRunShift : atoms_min(at(i), p);
    }
    // the packed sum v into the pixel's run, if in != 0; the run's position,
    // if head != 0 (predicated: no branch among the lanes)
    __device__ __forceinline__ static void add_pixel(At a, uint32_t v, uint32_t in, uint32_t head, uint32_t pos)
    {
        asm volatile("{\n\t"
                     ".reg .pred p, h;\n\t"
                     "setp.ne.u32 p, %2, 0;\n\t"
                     "setp.ne.u32 h, %3, 0;\n\t"
                     "@p red.shared.add.u32 [%0+8], %1;\n\t"
                     "@h st.shared.u32 [%0+4], %4;\n\t"
                     "}" ::"r"(a), "r"(v), "r"(in), "r"(head), "r"(pos) : "memory");
    }
    // a run's ADC sum and length, or its charge, into word 2
    __device__ __forceinline__ static void set_sum(At a, uint32_t adc, uint32_t len, uint32_t q)
    {
        st<2>(a, kKind == kWide ? q : adc | (len << kAdcBits));
    }
    __device__ __forceinline__ static uint32_t charge(uint32_t word2, int2 cal)
    {
        return kKind == kWide ? word2 : (uint32_t)cal.x * (word2 & kAdcMask) - (uint32_t)cal.y * (word2 >> kAdcBits);
    }
    // pixels of a run into its root's (its own if it is one)
    __device__ __forceinline__ static void add_pixels(At a, uint32_t v)
    {
        if (kKind == kWide) red<0>(a, v);
    }
    __device__ __forceinline__ static uint32_t pixels(At a)
    {
        return kKind == kWide ? ld<0>(a) & kRunPixels : ld<2>(a) >> kAdcBits;
    }
    __device__ __forceinline__ static void set_ordinal(At a, uint32_t v) { st<4>(a, v); }
    __device__ __forceinline__ static uint32_t ordinal(At a) { return ld<4>(a); }
    __device__ __forceinline__ static void init(At a, uint32_t i)
    {
        st<0>(a, kKind == kWide ? i << kRunShift : i);
        st<2>(a, 0);
        st<4>(a, 0);
    }
};
template <>
struct Runs<kGlobal> {
    uint32_t *base;
    using At = uint32_t *;
    __device__ __forceinline__ At at(uint32_t i) const { return base + (size_t)i * (kBigRunBytes / 4); }
    template <int f>
    __device__ __forceinline__ static uint32_t ld(At a) { return *(volatile uint32_t *)(a + f); }
    template <int f>
    __device__ __forceinline__ static void st(At a, uint32_t v) { *(volatile uint32_t *)(a + f) = v; }
    template <int f>
    __device__ __forceinline__ static void red(At a, uint32_t v) { atomicAdd(a + f, v); }
    __device__ __forceinline__ uint32_t parent(uint32_t i) const { return ld<0>(at(i)); }
    __device__ __forceinline__ void set_parent(uint32_t i, uint32_t p) const { st<0>(at(i), p); }
    __device__ __forceinline__ uint32_t min_parent(uint32_t i, uint32_t p) const { return atomicMin(at(i), p); }
    __device__ __forceinline__ static void add_pixel(At a, uint32_t v, uint32_t in, uint32_t head, uint32_t pos)
    {
        if (in) {
            atomicAdd(a + 2, v);
            if (head) st<1>(a, pos);
        }
    }
    __device__ __forceinline__ static void set_sum(At a, uint32_t, uint32_t, uint32_t q) { st<2>(a, q); }
    __device__ __forceinline__ static uint32_t charge(uint32_t word2, int2) { return word2; }
    __device__ __forceinline__ static void add_pixels(At a, uint32_t v) { atomicAdd(a + 5, v); }
    __device__ __forceinline__ static uint32_t pixels(At a) { return ld<5>(a); }
    __device__ __forceinline__ static void set_ordinal(At a, uint32_t v) { st<4>(a, v); }
    __device__ __forceinline__ static uint32_t ordinal(At a) { return ld<4>(a); }
    __device__ __forceinline__ static void init(At a, uint32_t i)
    {
        st<0>(a, i);
        st<2>(a, 0);
        st<4>(a, 0);
        st<5>(a, 0);
    }
};

// Find with path halving (each visited run is re-pointed to its
// grandparent).  Parents only ever point to a smaller run of the same tree,
// so a plain store that races with a link elsewhere leaves a valid ancestor
// behind; a link that loses such a race is retried by its union.
template <class A>
__device__ __forceinline__ uint32_t run_find(const A &a, uint32_t x)
{
    uint32_t y = a.parent(x);
    while (y != x) {
        const uint32_t z = a.parent(y);
        if (z != y) a.set_parent(x, z);
        x = y;
        y = z;
    }
    return x;
}

// Lock-free union of the trees of x and y by one thread: the larger root is
// linked under the smaller with an atomic minimum; a link that finds its
// root already linked elsewhere retries from the new parent.
template <class A>
__device__ __forceinline__ void run_union(const A &a, uint32_t x, uint32_t y)
{
    for (;;) {
        x = run_find(a, x);
        y = run_find(a, y);
        if (x == y) return;
        const uint32_t hi = max(x, y), lo = min(x, y), old = a.min_parent(hi, lo);
        if (old == hi) return;
        x = old;
        y = lo;
    }
}

// What a run sees of the bitmap: its word, the word above, the words beside
// both (up_left and left are only used past a row's first word, up_right
// before its last), the first run of the word above (or, if that word is
// empty, of the next one) and of the word after it.
struct RunView {
    uint32_t word, left, up, up_left, up_right, pre, next;
};
// Runs that touch run i (position p) before it: [*k, *end) of the row above,
// and *left, the run that ends the word to its left (kNoSlot: none).
// Returns its length.
__device__ __forceinline__ uint32_t run_contacts(const RunView &v, uint32_t W, uint32_t i, uint32_t p, uint32_t *k,
                                                 uint32_t *end, uint32_t *left)
{
    const uint32_t cw = (p >> 13) & 0xFu, b = (p >> 8) & 31u;
    const uint32_t len = (uint32_t)__clz(__brev(~(v.word >> b))); // 32 for a full word
    const bool above = (p & 0xFFu) != 0, left_edge = b == 0 && cw != 0, right_edge = b + len == 32 && cw + 1 < W;
    const uint32_t u = above ? v.up : 0u, hu = u & ~(u << 1);
    const uint32_t mask = (kFull >> (32 - len)) << b, t = u & (mask | (mask << 1) | (mask >> 1));
    uint32_t k0 = 0, e0 = 0;
    if (t) {
        k0 = v.pre + __popc(hu & (t ^ (t - 1))) - 1u;      // heads up to t's lowest bit
        e0 = v.pre + __popc(hu & (kFull >> __clz(t)));     // and up to its highest
    }
    if (left_edge && above && (v.up_left >> 31)) { // the run that ends the word before
        if (!e0) e0 = v.pre;
        k0 = v.pre - 1u;
    }
    if (right_edge && above && (v.up_right & 1u)) { // the run that starts the word after
        if (!e0) k0 = v.next;
        e0 = v.next + 1u;
    }
    *k = k0;
    *end = e0;
    *left = left_edge && (v.left >> 31) ? i - 1u : kNoSlot;
    return len;
}

// The item's digis, kBatch at a time so that their loads overlap: f(k, j, x)
// for the thread's digis from j on with words x[kBatch] (kNoDigi for those past
// the last), held in w from w[k] on with kSingle (all of them loaded by
// load_digis), else loaded here.
constexpr int kBatch = 2; // (4: more slots past a thread's last digi; 27.7M digis 530 us, 2: 519, 1: 526)
constexpr uint32_t kNoDigi = 0xFFFFFFFFu; // an invalid word (row 255, column 511)
template <int GT>
__device__ __forceinline__ void load_digis(uint32_t (&w)[kRunDigis], const uint2 *digis, uint32_t mine)
{
#pragma unroll
    for (int k = 0; k < kRunDigis; ++k) w[k] = (uint32_t)k < mine ? __ldg(&digis[k * GT].x) : kNoDigi;
}
template <int GT, bool kSingle, class F>
__device__ __forceinline__ void each_batch(uint32_t (&w)[kRunDigis], const uint2 *digis, uint32_t mine, F &&f)
{
    // digis: the thread's first, GT from one to the next, mine of them
    if constexpr (kSingle) {
#pragma unroll
        for (int k = 0; k < kRunDigis; k += kBatch) {
            if ((uint32_t)k < mine) {
                uint32_t x[kBatch];
#pragma unroll
                for (int u = 0; u < kBatch; ++u) x[u] = w[k + u];
                f(k, (uint32_t)k, x);
            }
        }
    } else {
#pragma unroll 1
        for (uint32_t base = 0; base < mine; base += kBatch) {
            uint32_t x[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) x[u] = base + u < mine ? __ldg(&digis[(size_t)(base + u) * GT].x) : kNoDigi;
            f(0, base, x);
        }
    }
}

// Packed sum of a surviving digi with word x: ADC, and ADC * bit << kSumShift.
constexpr uint32_t kSumShift = 13, kSumMask = (1u << kSumShift) - 1u;
__device__ __forceinline__ uint32_t pixel_sum(uint32_t x)
{
    const uint32_t adc = (x >> 17) & 0xFFu;
    return adc * (1u | (((x >> 8) & 31u) << kSumShift));
}

// Phases 5 and 6 for the runs of a; view(p) is what the run at position p
// sees (its loads independent of each other: two runs a thread at a time),
// calib(p) its module's gain (x) and pedestal (y).
template <int GT, bool kWhole, class A, class V, class B>
__device__ __forceinline__ void link_runs(const A &a, const V &view, const B &calib, uint32_t W, uint32_t nruns,
                                          GroupShared &gs, uint32_t gt, uint32_t bar)
{
    for (uint32_t i0 = gt; i0 < nruns; i0 += 2 * GT) {
        uint32_t i[2] = {i0, i0 + GT}, p[2], sum[2];
        RunView v[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const typename A::At r = a.at(i[u] < nruns ? i[u] : i0);
            p[u] = A::template ld<1>(r);
            sum[u] = A::template ld<2>(r);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) v[u] = view(p[u]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (i[u] >= nruns) break;
            uint32_t k, end, left;
            const uint32_t len = run_contacts(v[u], W, i[u], p[u], &k, &end, &left);
            const typename A::At r = a.at(i[u]);
            A::template st<1>(r, p[u] | (len << 17));
            // q = gain * ADC - ped over the run's pixels, columns c0 ..
            const int2 cal = calib(p[u]);
            const uint32_t c0 = (p[u] >> 8) & 0x1FFu, adc = sum[u] & kSumMask, base = c0 & ~31u;
            A::set_sum(r, adc, len, cal.x * adc - cal.y * len);
            A::template st<3>(r, cal.x * ((sum[u] >> kSumShift) + base * adc) -
                                     cal.y * (len * c0 + ((len * (len - 1u)) >> 1)));
            if (k < end)
                a.set_parent(i[u], k);
            else if (left != kNoSlot)
                a.set_parent(i[u], left);
            if (end > k + 1 || (k < end && left != kNoSlot))
                A::template st<4>(a.at(atomicAdd(&gs.extras, 1u)), i[u]);
        }
    }
    gsync<GT, kWhole>(bar);
    for (uint32_t e = gt, ne = gs.extras; e < ne; e += GT) {
        const typename A::At re = a.at(e);
        const uint32_t i = A::template ld<4>(re);
        A::template st<4>(re, 0);
        const uint32_t p = A::template ld<1>(a.at(i));
        uint32_t k, end, left;
        run_contacts(view(p), W, i, p, &k, &end, &left);
        for (++k;; ++k) { // the first contact is linked already
            uint32_t y = k;
            if (k >= end) {
                if (left == kNoSlot) break;
                y = left;
                left = kNoSlot;
            }
            run_union(a, i, y);
        }
    }
}

// Phase 7: only roots receive sums, so a run's own are still its own; two
// runs a thread at a time.
template <int GT, class A, class B>
__device__ __forceinline__ void sum_runs(const A &a, const B &calib, uint32_t nruns, uint32_t gt)
{
    for (uint32_t i0 = gt; i0 < nruns; i0 += 2 * GT) {
        const uint32_t i1 = i0 + GT < nruns ? i0 + GT : i0;
        uint32_t x0 = i0, x1 = i1, y0 = a.parent(i0), y1 = a.parent(i1);
        while (y0 != x0 || y1 != x1) {
            x0 = y0;
            x1 = y1;
            y0 = a.parent(x0);
            y1 = a.parent(x1);
        }
        const uint32_t i[2] = {i0, i1}, x[2] = {x0, x1};
        uint32_t p[2], q[2], mc[2], px[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const typename A::At r = a.at(i[u]);
            p[u] = A::template ld<1>(r);
            q[u] = A::template ld<2>(r);
            mc[u] = A::template ld<3>(r);
            px[u] = A::template ld<1>(a.at(x[u]));
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (u == 1 && i1 == i0) break;
            const typename A::At rx = a.at(x[u]);
            if (x[u] != i[u]) {
                a.set_parent(i[u], x[u]);
                A::template red<2>(rx, q[u]);
                A::template red<3>(rx, mc[u]);
                A::template red<4>(rx, A::charge(q[u], calib(p[u])) * ((p[u] & 0xFFu) - (px[u] & 0xFFu)));
            }
            A::add_pixels(rx, (p[u] >> 17) & 63u);
        }
    }
}

// The 32-run chunks [c0, c1) of a warp of the group (phases 8 and 9).
template <int GT>
__device__ __forceinline__ void warp_chunks(uint32_t nruns, uint32_t warp, uint32_t *c0, uint32_t *c1)
{
    const uint32_t chunks = (nruns + 31) >> 5, cpw = (chunks + GT / 32 - 1) / (GT / 32);
    *c0 = min(chunks, warp * cpw);
    *c1 = min(chunks, *c0 + cpw);
}

// Phase 8: the root's position (and item) into every run, with kRunKept on a
// kept root and kRunDropped on the runs of a cluster below threshold; gs.heavy
// set if a cluster's moments may have overflowed 32 bits; also(run, root's
// position, kept) for every run.  With
// kItems the kept roots of each item are counted in gs.tmp[16 ..].  One
// barrier; returns the kept roots of all runs, and in *ord those before the
// warp's chunks.  Roots of the items in `faulty` (bits; kItems) are not kept.
template <int GT, bool kWhole, bool kItems, class A, class B, class T>
__device__ __forceinline__ uint32_t mark_runs(const A &a, const B &calib, const T &also, uint32_t nruns, int32_t cthr,
                                              uint32_t faulty, GroupShared &gs, uint32_t gt, uint32_t bar,
                                              uint32_t *ord)
{
    constexpr int kWarps = GT / 32;
    const uint32_t lane = gt & 31, warp = gt >> 5;
    uint32_t c0, c1, wrun = 0;
    warp_chunks<GT>(nruns, warp, &c0, &c1);
    for (uint32_t ch = c0; ch < c1; ++ch) {
        const uint32_t i = (ch << 5) + lane;
        bool lead = false;
        if (i < nruns) {
            const uint32_t x = a.parent(i);
            const typename A::At rx = a.at(x);
            const uint32_t px = A::template ld<1>(rx);
            const int32_t Q = (int32_t)A::charge(A::template ld<2>(rx), calib(px));
            const bool kept = Q >= cthr && !(kItems && (faulty >> ((px & kRunItem) >> 23)) & 1u);
            lead = kept && x == i;
            if (Q > kQSafe32) gs.heavy = 1;
            also(a.at(i), px, kept);
            A::template st<1>(a.at(i), (px & (kItems ? kRunPos | kRunItem : kRunPos)) |
                                           (lead ? kRunKept : kept ? 0u : kRunDropped));
            if (kItems && lead) atomicAdd(&gs.tmp[16 + ((px & kRunItem) >> 23)], 1u);
        }
        wrun += __popc(__ballot_sync(kFull, lead));
    }
    if (lane == 0) gs.tmp[warp] = wrun;
    gsync<GT, kWhole>(bar);
    const uint32_t wt = lane < kWarps ? gs.tmp[lane] : 0u;
    uint32_t ws = wt;
#pragma unroll
    for (int o = 1; o < kWarps; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, ws, o);
        if ((int)lane >= o) ws += y;
    }
    *ord = __shfl_sync(kFull, ws - wt, warp);
    return __shfl_sync(kFull, ws, kWarps - 1);
}

// Phase 9: put(run, ordinal) for every kept root, in run order, gathered 32
// at a time so that every lane stages a cluster.
template <int GT, class A, class P>
__device__ __forceinline__ void stage_runs(const A &a, uint32_t nruns, uint32_t ord, uint16_t *wlist, uint32_t gt,
                                           const P &put)
{
    const uint32_t lane = gt & 31;
    uint32_t c0, c1, cnt = 0;
    warp_chunks<GT>(nruns, gt >> 5, &c0, &c1);
    for (uint32_t ch = c0;; ++ch) {
        const bool last = ch >= c1;
        if (!last) {
            const uint32_t i = (ch << 5) + lane;
            const bool kept = i < nruns && (A::template ld<1>(a.at(i)) & kRunKept);
            const uint32_t bal = __ballot_sync(kFull, kept);
            if (kept) wlist[cnt + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)i;
            cnt += __popc(bal);
            __syncwarp();
        }
        if (cnt >= 32 || (last && cnt > 0)) {
            if (lane < cnt) put((uint32_t)wlist[lane], ord + lane);
            if (last) break;
            __syncwarp();
            const uint32_t v = wlist[32 + lane];
            __syncwarp();
            wlist[lane] = (uint16_t)v;
            __syncwarp();
            cnt -= 32;
            ord += 32;
        } else if (last) {
            break;
        }
    }
}

// The sums of root i as a staged cluster at position `at`.
template <class A>
__device__ __forceinline__ void stage_root(const Launch &L, const A &a, uint32_t i, uint64_t at, int2 cal, bool heavy,
                                           const unsigned long long *exact)
{
    const typename A::At r = a.at(i);
    const uint32_t p = A::template ld<1>(r);
    const int32_t Q = (int32_t)A::charge(A::template ld<2>(r), cal), np = (int32_t)A::pixels(r);
    float x, y;
    if (heavy) {
        x = centroid_abs((long long)exact[2 * (size_t)i], Q);
        y = centroid_abs((long long)exact[2 * (size_t)i + 1], Q);
    } else {
        x = centroid_abs(A::template ld<4>(r) + (p & 0xFFu) * (uint32_t)Q, (uint32_t)Q);
        y = centroid_abs(A::template ld<3>(r), (uint32_t)Q);
    }
    L.ws.staging.put(at, (int32_t)((p & 0xFFu) * L.g.C + ((p >> 8) & 0x1FFu)), Q, np, x, y);
}

template <int GT, bool kWhole, RunKind kKind, bool kSingle>
__device__ __forceinline__ uint32_t run_clusters(const Launch &L, const ItemCtx &it, uint32_t sb, uint32_t rp,
                                                 const Runs<kKind> a, unsigned long long *exact, uint32_t nruns,
                                                 uint32_t (&w)[kRunDigis], GroupShared &gs, uint16_t *wlist,
                                                 uint32_t gt, uint32_t bar)
{
    using A = Runs<kKind>;
    const uint32_t C = L.g.C, W = (C + 31) >> 5;
    const uint32_t n = it.n;
    const uint32_t mine = n > gt ? (n - gt - 1) / GT + 1 : 0u;
    const uint2 *digis = L.ws.bucket + it.b + gt;
    const int32_t gain = it.gain, ped = it.ped;
    // runs of a batch of digis, kNoSlot for those below threshold and past the last
    auto runs_of = [&](const uint32_t (&x)[kBatch], uint32_t (&run)[kBatch], uint32_t (&in)[kBatch], uint32_t (&head)[kBatch]) {
        uint32_t word[kBatch], pre[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const uint32_t wi = x[u] == kNoDigi ? 0u : (x[u] & 0xFFu) * W + ((x[u] >> 13) & 0xFu);
            word[u] = lds(sb + 4 * wi);
            pre[u] = lds_u16(rp + 2 * wi);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const uint32_t b = x[u] == kNoDigi ? 0u : 1u << ((x[u] >> 8) & 31u), h = word[u] & ~(word[u] << 1);
            in[u] = word[u] & b;
            head[u] = h & b;
            run[u] = in[u] ? pre[u] + __popc(h & (b | (b - 1u))) - 1u : kNoSlot;
        }
    };

    // 3 (rest)
    for (uint32_t i = gt; i < nruns; i += GT) A::init(a.at(i), i);
    gsync<GT, kWhole>(bar);

    // 4
    each_batch<GT, kSingle>(w, digis, mine, [&](int k, uint32_t, const uint32_t (&x)[kBatch]) {
        uint32_t run[kBatch], in[kBatch], head[kBatch];
        runs_of(x, run, in, head);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            A::add_pixel(a.at(in[u] ? run[u] : 0u), pixel_sum(x[u]), in[u], head[u], x[u] & kRunPos);
            if constexpr (kSingle) w[k + u] = run[u];
        }
    });
    gsync<GT, kWhole>(bar);

    // 5, 6
    auto view = [&](uint32_t p) {
        const uint32_t r = p & 0xFFu, cw = (p >> 13) & 0xFu, wi = r * W + cw, wu = r ? wi - W : wi;
        const uint32_t own = sb + 4 * wi, u = sb + 4 * wu, ra = rp + 2 * wu, back = cw ? 4u : 0u;
        RunView v;
        v.word = lds(own);
        v.up = lds(u);
        v.pre = lds_u16(ra);
        v.left = lds(own - back);
        v.up_left = lds(u - back);
        v.up_right = lds<4>(u); // (past the last word lies the table of first runs)
        v.next = lds_u16(ra + 2);
        return v;
    };
    auto calib = [&](uint32_t) { return make_int2(gain, ped); };
    link_runs<GT, kWhole>(a, view, calib, W, nruns, gs, gt, bar);
    gsync<GT, kWhole>(bar);

    // 7
    sum_runs<GT>(a, calib, nruns, gt);
    uint32_t iv[kSingle ? kRunDigis : 1] = {}; // in-event indices for the labels
    auto index_of = [&](int k, uint32_t j) {
        if constexpr (kSingle)
            return iv[k];
        else
            return __ldg(&digis[(size_t)j * GT].y);
    };
    if constexpr (kSingle) {
        if (it.label_e || it.label16_e) {
#pragma unroll
            for (int k = 0; k < kRunDigis; ++k)
                if ((uint32_t)k < mine) iv[k] = __ldg(&digis[k * GT].y);
        }
    }
    gsync<GT, kWhole>(bar);
    // 8
    uint32_t ord;
    // (kNarrow: the label itself into word 0, whose parent is used up, so that
    // a digi's label is one load)
    const bool label0 = kKind == kNarrow && it.label_e;
    auto label_run = [&](typename A::At r, uint32_t px, bool kept) {
        if (label0) A::template st<0>(r, kept ? (px & 0xFFu) * C + ((px >> 8) & 0x1FFu) : (uint32_t)-2);
    };
    const uint32_t K = mark_runs<GT, kWhole, false>(a, calib, label_run, nruns, L.g.cluster_thr, 0u, gs, gt, bar, &ord);
    const bool heavy = gs.heavy != 0;
    if (heavy) { // both moments of every root again, in 64 bits
        for (uint32_t i = gt; i < nruns; i += GT) {
            exact[2 * (size_t)i] = 0;
            exact[2 * (size_t)i + 1] = 0;
        }
        gsync<GT, kWhole>(bar);
        for (uint32_t j = 0; j < mine; ++j) {
            const uint32_t digi = __ldg(&digis[(size_t)j * GT].x);
            uint32_t x[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) x[u] = u ? kNoDigi : digi;
            uint32_t run[kBatch], in[kBatch], head[kBatch];
            runs_of(x, run, in, head);
            if (!in[0]) continue;
            uint32_t root;
            if (label0) { // the run of the label's pixel
                const uint32_t id = A::template ld<0>(a.at(run[0]));
                if ((int32_t)id < 0) continue;
                x[0] = id / C;
                x[0] |= (id - x[0] * C) << 8;
                runs_of(x, run, in, head);
                root = run[0];
            } else {
                root = a.parent(run[0]);
            }
            const size_t y = root;
            const long long q = (long long)((int32_t)((digi >> 17) & 0xFFu) * gain - ped);
            atomicAdd(&exact[2 * y], (unsigned long long)(q * (long long)(digi & 0xFFu)));
            atomicAdd(&exact[2 * y + 1], (unsigned long long)(q * (long long)((digi >> 8) & 0x1FFu)));
        }
        gsync<GT, kWhole>(bar);
    }

    // 9: labels (the stores drain behind the staging)
    if (it.label_e) {
        each_batch<GT, kSingle>(w, digis, mine, [&](int k, uint32_t j, const uint32_t (&x)[kBatch]) {
            uint32_t run[kBatch], in[kBatch], head[kBatch], at[kBatch], p[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) at[u] = j + u < mine ? index_of(k + u, j + u) : 0u;
            if constexpr (kSingle) {
#pragma unroll
                for (int u = 0; u < kBatch; ++u) run[u] = x[u];
            } else {
                runs_of(x, run, in, head);
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const typename A::At r = a.at(run[u] == kNoSlot ? 0u : run[u]);
                p[u] = kKind == kNarrow ? A::template ld<0>(r) : A::template ld<1>(r);
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                int32_t lab = (int32_t)p[u];
                if (kKind != kNarrow)
                    lab = p[u] & kRunDropped ? -2 : (int32_t)((p[u] & 0xFFu) * C + ((p[u] >> 8) & 0x1FFu));
                if (j + u < mine) it.label_e[at[u]] = run[u] == kNoSlot ? -1 : lab;
            }
        });
    }
    stage_runs<GT>(a, nruns, ord, wlist, gt, [&](uint32_t i, uint32_t o) {
        stage_root(L, a, i, it.b + o, make_int2(gain, ped), heavy, exact);
        if (it.label16_e) A::set_ordinal(a.at(i), o); // read back by the compact labels
    });
    if (it.label16_e) { // compact labels, once every kept root has its ordinal
        gsync<GT, kWhole>(bar);
        each_batch<GT, kSingle>(w, digis, mine, [&](int k, uint32_t j, const uint32_t (&x)[kBatch]) {
            uint32_t run[kBatch], in[kBatch], head[kBatch];
            if constexpr (kSingle) {
#pragma unroll
                for (int u = 0; u < kBatch; ++u) run[u] = x[u];
            } else {
                runs_of(x, run, in, head);
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                if (j + u >= mine) break;
                uint16_t v = kLab16Below;
                if (run[u] != kNoSlot) {
                    const typename A::At rx = a.at(a.parent(run[u]));
                    v = A::template ld<1>(rx) & kRunKept ? (uint16_t)A::ordinal(rx) : kLab16Dropped;
                }
                it.label16_e[index_of(k + u, j + u)] = v;
            }
        });
    }
    return K;
}

// The run tier on run records in global scratch: items with more runs than
// the shared memory holds (out of line: rare, and its registers are its own).
template <int GT, bool kWhole>
__device__ __noinline__ uint32_t run_clusters_big(const Launch &L, const ItemCtx it, uint32_t sb, uint32_t rp,
                                                  unsigned char *base, uint32_t nruns, GroupShared &gs,
                                                  uint16_t *wlist, uint32_t gt, uint32_t bar)
{
    Runs<kGlobal> a;
    a.base = reinterpret_cast<uint32_t *>(base + (size_t)16 * nruns); // after the 64-bit moments
    uint32_t w[kRunDigis];
    return run_clusters<GT, kWhole, kGlobal, false>(L, it, sb, rp, a, reinterpret_cast<unsigned long long *>(base), nruns,
                                                 w, gs, wlist, gt, bar);
}

// One item of the run tier (phases 1-3, then run_clusters): `mem` is the
// shared address of the group's slice with room for `cap` runs, `exact` its
// slice of the 64-bit moments, `part` of `parts` its part of the block's slab
// of global scratch.  kKind kNarrow: the item has at most kNarrowDigis digis;
// kSingle: at most kRunDigis * GT, which stay in registers.  Returns the number of kept clusters (uniform
// over the group).  An item with an invalid or a duplicated digi flags its
// event and keeps none.
template <int GT, bool kWhole, RunKind kKind, bool kSingle>
__device__ __forceinline__ uint32_t run_item(const Launch &L, const ItemCtx &it, uint32_t mem, uint32_t cap,
                                             unsigned long long *exact, uint32_t part, uint32_t parts,
                                             GroupShared &gs, uint16_t *wlist, uint32_t gt, uint32_t bar)
{
    const uint32_t R = L.g.R, C = L.g.C, W = (C + 31) >> 5, nw4 = run_words(R, C);
    const int32_t thr = L.g.pixel_thr;
    const uint32_t n = it.n, mine = n > gt ? (n - gt - 1) / GT + 1 : 0u;
    const uint2 *digis = L.ws.bucket + it.b + gt;
    const int32_t gain = it.gain, ped = it.ped;
    const uint32_t sb = mem, rp = sb + 4 * nw4;
    const uint32_t ab = mem + (uint32_t)run_fixed_bytes(R, C); // the bitmap of the dropped digis; then the run records

    // 1
    uint32_t w[kRunDigis];
    if constexpr (kSingle) load_digis<GT>(w, digis, mine);
    for (uint32_t i = gt; i < nw4 / 4; i += GT) {
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(sb + 16 * i), "r"(0) : "memory");
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(ab + 16 * i), "r"(0) : "memory");
    }
    if (gt == 0) {
        gs.flag = 0;
        gs.heavy = 0;
        gs.pixels = 0;
        gs.extras = 0;
    }
    gsync<GT, kWhole>(bar);

    // 2
    uint32_t valid = 0;
    each_batch<GT, kSingle>(w, digis, mine, [&](int, uint32_t, const uint32_t (&x)[kBatch]) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u) { // (words past the last digi are invalid, and OR in nothing)
            const uint32_t r = x[u] & 0xFFu, c = (x[u] >> 8) & 0x1FFu, adc = x[u] >> 17;
            const bool ok = r < R && c < C && adc - 1u < 255u; // ADC not 0, bits 25-31 clear
            const uint32_t o = ok ? 4 * (r * W + (c >> 5)) : 0u, bit = ok ? 1u << (c & 31) : 0u;
            reds_or(((int32_t)adc * gain - ped >= thr ? sb : ab) + o, bit);
            valid += ok ? 1u : 0u;
        }
    });
    if (__any_sync(kFull, valid != mine) && (gt & 31) == 0) gs.flag = 1;
    gsync<GT, kWhole>(bar);

    // 3: runs of a word, counted over contiguous groups of four words a thread
    const uint32_t per = ((nw4 / 4 + GT - 1) / GT) * 4;
    const uint32_t w0 = min(nw4, gt * per), w1 = min(nw4, w0 + per);
    auto four = [](uint32_t addr) {
        uint4 v;
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "r"(addr)
                     : "memory");
        return v;
    };
    uint32_t local = 0, pixels = 0;
    for (uint32_t i = w0; i < w1; i += 4) {
        const uint4 s = four(sb + 4 * i), d = four(ab + 4 * i);
        local += __popc(s.x & ~(s.x << 1)) + __popc(s.y & ~(s.y << 1)) + __popc(s.z & ~(s.z << 1)) +
                 __popc(s.w & ~(s.w << 1));
        pixels += __popc(s.x | d.x) + __popc(s.y | d.y) + __popc(s.z | d.z) + __popc(s.w | d.w);
    }
    pixels = __reduce_add_sync(kFull, pixels);
    if ((gt & 31) == 0 && pixels) atomicAdd(&gs.pixels, pixels);
    uint32_t nruns;
    uint32_t run = group_exclusive_scan<GT, kWhole>(local, gs.tmp, gt, bar, &nruns);
    if (gs.flag || gs.pixels != n) { // (uniform: both are settled by the scan's barrier)
        if (gt == 0) atomicOr(it.err_e, gs.flag ? kErrBadDigi : kErrDup);
        gsync<GT, kWhole>(bar);
        return 0;
    }
    for (uint32_t i = w0; i < w1; i += 4) {
        const uint4 s = four(sb + 4 * i);
        const uint32_t p0 = run, p1 = p0 + __popc(s.x & ~(s.x << 1)), p2 = p1 + __popc(s.y & ~(s.y << 1)),
                       p3 = p2 + __popc(s.z & ~(s.z << 1));
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(rp + 2 * i), "r"(p0 | (p1 << 16)), "r"(p2 | (p3 << 16))
                     : "memory");
        run = p3 + __popc(s.w & ~(s.w << 1));
    }
    uint32_t K;
    if (nruns <= cap) {
        Runs<kKind> a;
        a.base = ab;
        K = run_clusters<GT, kWhole, kKind, kSingle>(L, it, sb, rp, a, exact, nruns, w, gs, wlist, gt, bar);
    } else {
        uint64_t first, room;
        if (L.ws.big_arena) { // a slot a run, bump-allocated
            if (gt == 0) gs.pack_end = atomicAdd(&L.ws.ctl[2], nruns);
            gsync<GT, kWhole>(bar);
            first = gs.pack_end;
            room = first < L.ws.big_slots ? L.ws.big_slots - first : 0;
        } else { // the group's part of the block's slab
            room = L.ws.big_slots / parts;
            first = (uint64_t)blockIdx.x * L.ws.big_slots + part * room;
        }
        if (nruns <= room) {
            K = run_clusters_big<GT, kWhole>(L, it, sb, rp, L.ws.big + first * kBigSlotBytes, nruns, gs, wlist, gt,
                                             bar);
        } else {
            if (gt == 0) atomicOr(&L.ws.ctl[1], kErrCapacity);
            K = 0;
        }
    }
    gsync<GT, kWhole>(bar); // the slice is free for the next item
    return K;
}

// ---- packed tier
//
// The small items of a ticket together: up to four digis a thread (at most
// 1,023) of up to 16 items by a group of GT threads, through the run tier's
// phases on a sparse bitmap.
// Of each item's bitmap words only the touched ones are stored, in (item,
// row, word) order: a bit per word of the module says which are (16 bits a
// row, so that a word's neighbours in its row lie in the same field), and the
// set bits before a word are its place.  So the runs are numbered in (item,
// row-major) order as in the run tier, with no hashing and nothing to probe,
// and the kept roots come out item by item in id order.  Phases, one group
// barrier between them:
//   a the digis' items and words; tables cleared
//   b a bit per touched word
//   c touched words before each field, by a scan
//   d a bit per digi, among the survivors or the dropped (set already, or in
//     both: a duplicate)
//   e runs before each touched word, by a scan; run records initialised
//   f charge and position into the runs, then 5 to 9 of the run tier
// An item with an invalid or a duplicated digi flags its event, keeps no
// cluster and gets no labels, as in the other tiers (its digis pass through
// the phases all the same: their sums mean nothing, but stay in its own runs).
// What bounds it: the latency of the phases, which all items of a ticket
// share; the work is the digis', not the modules'.  29,696 items of 32 digis:
// 343 us with a warp an item -> 57 us.
constexpr int kPackPer = 4; // digis a thread holds

// One warp (lane = its lane): the pack that starts at item i0 of the ticket,
// as many of the next items of at most pmax digis as pcap holds (larger ones
// are passed over).  Writes gs.pack (first packed digi of each item from i0
// on, the total from the pack's end on) and returns the end.
__device__ __forceinline__ uint32_t plan_pack(GroupShared &gs, uint32_t i0, uint32_t pmax, uint32_t pcap,
                                              uint32_t lane, uint32_t n_lane)
{
    const uint32_t pn = n_lane <= pmax ? n_lane : 0u;
    uint32_t incl = pn;
#pragma unroll
    for (int o = 1; o < kGroup; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if ((int)lane >= o) incl += y;
    }
    const uint32_t fits = __ballot_sync(kFull, lane < (uint32_t)kGroup - i0 && incl <= pcap);
    const uint32_t cnt = __ffs(~fits) - 1; // leading items that fit (kGroup < 32, so ~fits != 0)
    const uint32_t total = __shfl_sync(kFull, incl, cnt ? cnt - 1 : 0);
    if (lane <= (uint32_t)kGroup) gs.pack[lane] = (uint16_t)(lane < cnt ? incl - pn : total);
    return i0 + cnt;
}

template <int GT, bool kWhole>
__device__ __forceinline__ void pack_items(const Launch &L, uint32_t mem, unsigned long long *exact, uint32_t i0,
                                           uint32_t items, uint32_t total, GroupShared &gs, uint16_t *wlist,
                                           uint32_t gt, uint32_t bar)
{
    using A = Runs<kNarrow>;
    const uint32_t R = L.g.R, C = L.g.C, W = (C + 31) >> 5, RH = (R + 1) >> 1, pcap = L.cc.pack_digis;
    const int32_t thr = L.g.pixel_thr;
    // fields: RH words of two rows an item; and the touched words before each
    const uint32_t nf = items * RH, fields = mem, before = fields + 4 * kGroup * RH;
    const uint32_t drop = (before + 2 * kGroup * RH + 15) & ~15u, surv = drop + 4 * (pcap + 1);
    const uint32_t rpre = surv + 4 * (pcap + 1);
    A a;
    a.base = (rpre + 2 * (pcap + 2) + 3) & ~3u;

    // a
    uint32_t w[kPackPer], idx[kPackPer], li[kPackPer], at[kPackPer];
#pragma unroll
    for (int k = 0; k < kPackPer; ++k) {
        const uint32_t t = gt + k * GT;
        w[k] = kNoDigi;
        idx[k] = li[k] = at[k] = 0;
        if (t < total) {
            uint32_t i = 0; // the last item whose first digi is at or before t
#pragma unroll
            for (uint32_t step = kGroup / 2; step; step >>= 1)
                if (gs.pack[i + step] <= t) i += step;
            const uint2 d = __ldg(L.ws.bucket + gs.b[i0 + i] + (t - gs.pack[i]));
            li[k] = i;
            w[k] = d.x;
            idx[k] = d.y;
        }
    }
    for (uint32_t i = gt; i < nf; i += GT) sts(fields + 4 * i, 0);
    for (uint32_t i = gt; i <= total; i += GT) {
        sts(drop + 4 * i, 0);
        sts(surv + 4 * i, 0);
    }
    if (gt < (uint32_t)kGroup) gs.tmp[16 + gt] = 0;
    if (gt == 0) {
        gs.heavy = 0;
        gs.extras = 0;
        gs.flag = 0;
    }
    gsync<GT, kWhole>(bar);
    // (phase f is the last to flag)
    auto flag = [&](uint32_t i, uint32_t err) {
        atomicOr(L.ws.event_err + gs.rec[i0 + i].e, err);
        atomicOr(&gs.flag, 1u << i);
    };

    // b
#pragma unroll
    for (int k = 0; k < kPackPer; ++k) {
        if (gt + k * GT >= total) break;
        const uint32_t r = w[k] & 0xFFu, c = (w[k] >> 8) & 0x1FFu, adc = w[k] >> 17;
        if (r >= R || c >= C || adc - 1u >= 255u) { // ADC 0, or any of the bits 25-31
            flag(li[k], kErrBadDigi);
            w[k] = kNoDigi;
        } else {
            reds_or(fields + 4 * (li[k] * RH + (r >> 1)), 1u << (((r & 1u) << 4) + (c >> 5)));
        }
    }
    gsync<GT, kWhole>(bar);

    // c
    uint32_t touched;
    {
        const uint32_t per = (nf + GT - 1) / GT, f0 = min(nf, gt * per), f1 = min(nf, f0 + per);
        uint32_t local = 0;
        for (uint32_t i = f0; i < f1; ++i) local += __popc(lds(fields + 4 * i));
        uint32_t run = group_exclusive_scan<GT, kWhole>(local, gs.tmp, gt, bar, &touched);
        for (uint32_t i = f0; i < f1; ++i) {
            sts_u16(before + 2 * i, run);
            run += __popc(lds(fields + 4 * i));
        }
    }
    gsync<GT, kWhole>(bar);
    // place of word cw of row r of item i (of the next touched one if it is
    // not), and whether it and the words beside it in the row are touched
    // (bits 1, 0 and 2 of *near)
    auto place = [&](uint32_t i, uint32_t r, uint32_t cw, uint32_t *near) {
        const uint32_t f = i * RH + (r >> 1), field = lds(fields + 4 * f), sh = ((r & 1u) << 4) + cw;
        const uint32_t row = ((field >> ((r & 1u) << 4)) & 0xFFFFu) << 1; // bit cw + 1: word cw
        *near = (row >> cw) & 7u;
        return lds_u16(before + 2 * f) + __popc(field & ((1u << sh) - 1u));
    };

    // d
    uint32_t dropped = 0; // bit k: digi k is below threshold
#pragma unroll
    for (int k = 0; k < kPackPer; ++k) {
        if (gt + k * GT >= total) break;
        if (w[k] == kNoDigi) continue;
        const ItemRec &rec = gs.rec[i0 + li[k]];
        const uint32_t r = w[k] & 0xFFu, c = (w[k] >> 8) & 0x1FFu, bit = 1u << (c & 31);
        uint32_t near;
        at[k] = place(li[k], r, c >> 5, &near);
        const bool keep = (int32_t)((w[k] >> 17) & 0xFFu) * rec.gain - rec.ped >= thr;
        if (atoms_or((keep ? surv : drop) + 4 * at[k], bit) & bit) flag(li[k], kErrDup);
        dropped |= keep ? 0u : 1u << k;
    }
    gsync<GT, kWhole>(bar);

    // e
    uint32_t nruns;
    {
        const uint32_t per = (touched + GT - 1) / GT, f0 = min(touched, gt * per), f1 = min(touched, f0 + per);
        uint32_t local = 0;
        for (uint32_t i = f0; i < f1; ++i) {
            const uint32_t x = lds(surv + 4 * i);
            local += __popc(x & ~(x << 1));
        }
        uint32_t run = group_exclusive_scan<GT, kWhole>(local, gs.tmp, gt, bar, &nruns);
        for (uint32_t i = f0; i < f1; ++i) {
            const uint32_t x = lds(surv + 4 * i);
            sts_u16(rpre + 2 * i, run);
            run += __popc(x & ~(x << 1));
        }
        if (gt == 0) sts_u16(rpre + 2 * touched, nruns);
        for (uint32_t i = gt; i < nruns; i += GT) A::init(a.at(i), i);
    }
    gsync<GT, kWhole>(bar);

    // f
#pragma unroll
    for (int k = 0; k < kPackPer; ++k) {
        if (gt + k * GT >= total) break;
        const uint32_t x = w[k];
        w[k] = kNoSlot;
        if (x == kNoDigi) continue;
        const uint32_t word = lds(surv + 4 * at[k]), b = 1u << ((x >> 8) & 31u), h = word & ~(word << 1);
        if ((dropped >> k) & 1u) { // (a survivor at its pixel is a duplicate too)
            if (word & b) flag(li[k], kErrDup);
            continue;
        }
        const uint32_t run = lds_u16(rpre + 2 * at[k]) + __popc(h & (b | (b - 1u))) - 1u;
        A::add_pixel(a.at(run), pixel_sum(x), 1u, h & b, (x & kRunPos) | (li[k] << 23));
        w[k] = run;
    }
    gsync<GT, kWhole>(bar);
    auto view = [&](uint32_t p) {
        const uint32_t r = p & 0xFFu, cw = (p >> 13) & 0xFu, i = (p & kRunItem) >> 23;
        uint32_t near, above;
        const uint32_t own = surv + 4 * place(i, r, cw, &near);
        const uint32_t up = place(i, r ? r - 1u : 0u, cw, &above), here = (above >> 1) & 1u;
        RunView v;
        v.word = lds(own);
        v.left = near & 1u ? lds<-4>(own) : 0u;
        v.up = here ? lds(surv + 4 * up) : 0u;
        v.up_left = above & 1u ? lds<-4>(surv + 4 * up) : 0u;
        v.up_right = above & 4u ? lds(surv + 4 * (up + here)) : 0u;
        v.pre = lds_u16(rpre + 2 * up);
        v.next = lds_u16(rpre + 2 * (up + here));
        return v;
    };
    auto calib = [&](uint32_t p) {
        const ItemRec &rec = gs.rec[i0 + ((p & kRunItem) >> 23)];
        return make_int2(rec.gain, rec.ped);
    };
    link_runs<GT, kWhole>(a, view, calib, W, nruns, gs, gt, bar);
    gsync<GT, kWhole>(bar);
    sum_runs<GT>(a, calib, nruns, gt);
    gsync<GT, kWhole>(bar);
    uint32_t ord;
    mark_runs<GT, kWhole, true>(a, calib, [](A::At, uint32_t, bool) {}, nruns, L.g.cluster_thr, gs.flag, gs, gt, bar,
                                &ord);
    const bool heavy = gs.heavy != 0;
    const uint32_t faulty = gs.flag;
    if (heavy) { // both moments again, in 64 bits
        for (uint32_t i = gt; i < 2 * nruns; i += GT) exact[i] = 0;
        gsync<GT, kWhole>(bar);
#pragma unroll
        for (int k = 0; k < kPackPer; ++k) {
            if (gt + k * GT >= total || w[k] == kNoSlot) continue;
            const ItemRec &rec = gs.rec[i0 + li[k]];
            const uint32_t x = __ldg(&L.ws.bucket[gs.b[i0 + li[k]] + (gt + k * GT - gs.pack[li[k]])].x);
            const uint32_t y = a.parent(w[k]);
            const long long q = (long long)((int32_t)((x >> 17) & 0xFFu) * rec.gain - rec.ped);
            atomicAdd(&exact[2 * y], (unsigned long long)(q * (long long)(x & 0xFFu)));
            atomicAdd(&exact[2 * y + 1], (unsigned long long)(q * (long long)((x >> 8) & 0x1FFu)));
        }
        gsync<GT, kWhole>(bar);
    }
    // each item's kept clusters, and those of the items before it
    const uint32_t lane = gt & 31, kept = lane < (uint32_t)kGroup ? gs.tmp[16 + lane] : 0u;
    uint32_t first = kept;
#pragma unroll
    for (int o = 1; o < kGroup; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, first, o);
        if ((int)lane >= o) first += y;
    }
    first -= kept;
    if (gt < (uint32_t)kGroup && gs.pack[gt + 1] > gs.pack[gt]) {
        L.ws.cursor[gs.ticket * L.cc.ticket_items + i0 + gt] = kept;
        gs.rec[i0 + gt].e = first; // (a packed item's event is not needed any more)
    }
    if (L.out.label) {
#pragma unroll
        for (int k = 0; k < kPackPer; ++k) {
            if (gt + k * GT >= total) break;
            if ((faulty >> li[k]) & 1u) continue;
            int32_t lab = -1;
            if (w[k] != kNoSlot) {
                const uint32_t p = A::ld<1>(a.at(w[k]));
                lab = p & kRunDropped ? -2 : (int32_t)((p & 0xFFu) * C + ((p >> 8) & 0x1FFu));
            }
            L.out.label[gs.rec[i0 + li[k]].label_off + idx[k]] = lab;
        }
    }
    gsync<GT, kWhole>(bar);
    stage_runs<GT>(a, nruns, ord, wlist, gt, [&](uint32_t i, uint32_t o) {
        const uint32_t item = (A::ld<1>(a.at(i)) & kRunItem) >> 23;
        const ItemRec &rec = gs.rec[i0 + item];
        const uint32_t k = o - rec.e;
        stage_root(L, a, i, gs.b[i0 + item] + k, make_int2(rec.gain, rec.ped), heavy, exact);
        if (L.out.label16) A::set_ordinal(a.at(i), k); // read back by the compact labels
    });
    if (L.out.label16) {
        gsync<GT, kWhole>(bar);
#pragma unroll
        for (int k = 0; k < kPackPer; ++k) {
            if (gt + k * GT >= total) break;
            if ((faulty >> li[k]) & 1u) continue;
            uint16_t v = kLab16Below;
            if (w[k] != kNoSlot) {
                const A::At rx = a.at(a.parent(w[k]));
                v = A::ld<1>(rx) & kRunKept ? (uint16_t)A::ordinal(rx) : kLab16Dropped;
            }
            L.out.label16[gs.rec[i0 + li[k]].label_off + idx[k]] = v;
        }
    }
    gsync<GT, kWhole>(bar); // the slice and the plan are free
}

// ---------------------------------------------------------------- hash label store

// Home slot of a key in a table of H slots (multiplicative hashing: the high
// bits of key times the 32-bit golden ratio, scaled to [0, H)).
__device__ __forceinline__ uint32_t hash_home(uint32_t key, uint32_t H) { return __umulhi(key * 0x9E3779B1u, H); }

// Find on packed keys with path halving (the index of a key is its low
// bits); parents only ever decrease, as in run_find.
template <uint32_t kIdx>
__device__ __forceinline__ uint32_t key_find(uint32_t *par, uint32_t x)
{
    volatile uint32_t *p = par;
    uint32_t y = p[x & kIdx];
    while (y != x) {
        const uint32_t z = p[y & kIdx];
        if (z != y) p[x & kIdx] = z;
        x = y;
        y = z;
    }
    return x;
}

// Lock-free union of the trees of packed keys a and b (the root with the
// larger key is linked under the smaller with atomicMin; a lost race retries
// from the new parent), as run_union on runs.
template <uint32_t kIdx>
__device__ __forceinline__ void key_union(uint32_t *par, uint32_t a, uint32_t b)
{
    for (;;) {
        a = key_find<kIdx>(par, a);
        b = key_find<kIdx>(par, b);
        if (a == b) return;
        if (a < b) {
            const uint32_t t = a;
            a = b;
            b = t;
        }
        const uint32_t old = atomicMin(&par[a & kIdx], b);
        if (old == a) return;
        a = old;
    }
}

// The hash store (tuning label_store = kStoreHash) clusters an item with a
// group of item_threads threads, one of the block's kCCThreads / item_threads
// groups, each with its own slice of shared memory and its own named
// barrier, so that several items of a ticket run side by side.  Pixel
// lookup goes through an open-addressing table keyed by linear pixel index
// (2n slots for n digis, linear probing) instead of module-sized bitmaps, so
// the memory an item needs follows its digi count.  Digi j of the item (in
// bucket order) owns entry j of the accumulator and parent arrays; the
// union-find links packed keys (lin << kHashIdxBits | j) with atomicMin, so
// the root of every cluster is its pixel of smallest linear index (the
// cluster id) with no sort.  Ids are put in order at the end: kept roots are
// counted per row, the row counts scanned, and each root ranked by column
// among the kept roots of its own row.
struct HashMem {
    int2 *m;           // [cap] root: sum q*row, sum q*col (32-bit, as in the run tier)
    int32_t *q;        // [cap] root: charge
    uint32_t *np;      // [cap] root: pixel count; then its ordinal (compact labels)
    uint32_t *par;     // [cap] packed parent key; then a kept root's row base
    uint32_t *rowcnt;  // [256] kept roots per row
    uint32_t *table;   // [2 cap] (lin + 1) << 13 | surviving << 12 | j, 0 empty; then the row lists
    unsigned long long *exact; // [2 cap] (global) 64-bit moments of an item with a heavy cluster
};

__device__ __forceinline__ HashMem hash_mem(unsigned char *dsm, size_t smem, uint32_t groups, uint32_t gid,
                                            uint32_t cap, unsigned long long *exact)
{
    const size_t slice = (smem / groups) & ~(size_t)15;
    HashMem h;
    h.m = reinterpret_cast<int2 *>(dsm + slice * gid);
    h.q = reinterpret_cast<int32_t *>(h.m + cap);
    h.np = reinterpret_cast<uint32_t *>(h.q + cap);
    h.par = h.np + cap;
    h.rowcnt = h.par + cap;
    h.table = h.rowcnt + 256;
    h.exact = exact + (size_t)2 * cap * gid;
    return h;
}

// Table entry of pixel `lin` if it is there and survives the pixel
// threshold, else 0.  The table holds at most H / 2 entries, so a probe
// always ends at an empty slot.
__device__ __forceinline__ uint32_t hash_survivor(const uint32_t *table, uint32_t H, uint32_t lin)
{
    uint32_t s = hash_home(lin, H);
    for (uint32_t i = 0; i < H; ++i) {
        const uint32_t e = table[s];
        if (e == 0) return 0u;
        if ((e >> 13) == lin + 1) return (e >> 12) & 1u ? e : 0u;
        s = s + 1 == H ? 0u : s + 1;
    }
    return 0u;
}

// Packed union-find key of a table entry.
__device__ __forceinline__ uint32_t hash_key(uint32_t e)
{
    return (((e >> 13) - 1u) << kHashIdxBits) | (e & ((1u << kHashIdxBits) - 1u));
}

// One item of at most hash_capacity digis clustered by the calling group
// (gt = thread index in the group, GT = its size, bar = its barrier id);
// gflag and gheavy are the group's shared flag words (zero on entry, left
// zero).  Thread gt holds digis gt, gt + GT, ... in registers throughout.
// Phases, one group barrier each:
//   0 table and row counters emptied (the words load meanwhile)
//   1 every valid digi into the table (a pixel already there is a
//     duplicate); parent and accumulators of the survivors
//   2 unions with the surviving neighbours before the pixel in row-major
//     order: left L and up U; without U, upper-left UL (unless L, which
//     reaches UL through its own U) and upper-right UR.  With U, UL and UR
//     are U's own left and right neighbours, so every 8-adjacency is
//     covered with at most two unions a pixel.
//   3 roots, and charge, size and moments per root (32-bit shared atomics;
//     a cluster heavier than kQSafe32 sends the item through the exact
//     64-bit pass, as in the run tier)
//   4 labels; kept roots counted per row
//   5 row bases by a scan of the row counts (each warp scans all 256, eight
//     a lane); every kept root's column into its row's list
//   6 ordinal = row base + kept roots of the row with a smaller column;
//     staging; (compact labels) the ordinals read back per digi
// Returns the number of kept clusters (uniform over the group).
template <int kD>
__device__ uint32_t hash_item(const Launch &L, const ItemCtx &it, const HashMem &h, uint32_t gt, uint32_t GT,
                              uint32_t bar, uint32_t *gflag, uint32_t *gheavy)
{
    constexpr uint32_t kIdx = (1u << kHashIdxBits) - 1u;
    const uint32_t R = L.g.R, C = L.g.C;
    const int32_t thr = L.g.pixel_thr, cthr = L.g.cluster_thr;
    const uint32_t n = it.n, lane = threadIdx.x & 31, H = 2 * n;
    const uint2 *digis = L.ws.bucket + it.b;
    const int32_t gain = it.gain, ped = it.ped;

    // 0
    for (uint32_t i = gt; i < H; i += GT) h.table[i] = 0;
    for (uint32_t i = gt; i < 256; i += GT) h.rowcnt[i] = 0;
    uint32_t w[kD], rt[kD];
#pragma unroll
    for (int k = 0; k < kD; ++k) {
        const uint32_t j = gt + k * GT;
        w[k] = j < n ? __ldg(&digis[j].x) : 0u;
    }
    group_sync(bar, GT);

    // 1
    uint32_t err = 0;
#pragma unroll
    for (int k = 0; k < kD; ++k) {
        rt[k] = kNoSlot;
        const uint32_t j = gt + k * GT;
        if (j >= n) continue;
        const uint32_t x = w[k], r = x & 0xFFu, c = (x >> 8) & 0x1FFu, adc = (x >> 17) & 0xFFu;
        if (r >= R || c >= C || adc == 0 || (x >> 25) != 0) {
            err |= kErrBadDigi;
            continue;
        }
        const uint32_t lin = r * C + c;
        const bool surv = (int32_t)adc * gain - ped >= thr;
        const uint32_t e = ((lin + 1) << 13) | ((uint32_t)surv << 12) | j;
        uint32_t s = hash_home(lin, H), i = 0;
        for (; i < H; ++i) {
            const uint32_t old = atomicCAS(&h.table[s], 0u, e);
            if (old == 0) break;
            if ((old >> 13) == lin + 1) {
                err |= kErrDup;
                break;
            }
            s = s + 1 == H ? 0u : s + 1;
        }
        if (i == H) err |= kErrCapacity; // not reached: at most n entries in 2n slots
        if (surv) {
            const uint32_t key = (lin << kHashIdxBits) | j;
            h.par[j] = key;
            h.q[j] = 0;
            h.np[j] = 0;
            h.m[j] = make_int2(0, 0);
            rt[k] = key;
        }
    }
    err = __reduce_or_sync(kFull, err);
    if (err && lane == 0) atomicOr(gflag, err);
    group_sync(bar, GT);
    const uint32_t flag = *(volatile uint32_t *)gflag;
    if (flag) {
        group_sync(bar, GT); // every thread of the group has read the flag
        if (gt == 0) {
            if (flag & (kErrBadDigi | kErrDup)) atomicOr(it.err_e, flag & (kErrBadDigi | kErrDup));
            if (flag & kErrCapacity) atomicOr(&L.ws.ctl[1], kErrCapacity);
            *gflag = 0;
        }
        return 0;
    }

    // 2
#pragma unroll
    for (int k = 0; k < kD; ++k) {
        if (rt[k] == kNoSlot) continue;
        const uint32_t x = w[k], r = x & 0xFFu, c = (x >> 8) & 0x1FFu, lin = r * C + c;
        const uint32_t eL = c > 0 ? hash_survivor(h.table, H, lin - 1) : 0u;
        uint32_t e1 = eL, e2 = 0;
        if (r > 0) {
            const uint32_t eU = hash_survivor(h.table, H, lin - C);
            if (eU) {
                e2 = eU;
            } else {
                if (!eL && c > 0) e1 = hash_survivor(h.table, H, lin - C - 1);
                if (c + 1 < C) e2 = hash_survivor(h.table, H, lin - C + 1);
            }
        }
        if (e1) key_union<kIdx>(h.par, rt[k], hash_key(e1));
        if (e2) key_union<kIdx>(h.par, rt[k], hash_key(e2));
    }
    group_sync(bar, GT);

    // 3
    bool heavy_here = false;
#pragma unroll
    for (int k = 0; k < kD; ++k) {
        if (rt[k] == kNoSlot) continue;
        const uint32_t root = key_find<kIdx>(h.par, rt[k]), y = root & kIdx;
        const uint32_t x = w[k];
        const int32_t q = (int32_t)((x >> 17) & 0xFFu) * gain - ped;
        const int32_t old = atomicAdd(&h.q[y], q);
        if (old + q > kQSafe32) heavy_here = true;
        atomicAdd(&h.np[y], 1u);
        atomicAdd(&h.m[y].x, q * (int32_t)(x & 0xFFu));
        atomicAdd(&h.m[y].y, q * (int32_t)((x >> 8) & 0x1FFu));
        rt[k] = root;
    }
    if (heavy_here) *gheavy = 1;
    group_sync(bar, GT);
    const bool heavy = *(volatile uint32_t *)gheavy != 0;
    if (heavy) {
        for (uint32_t i = gt; i < 2 * n; i += GT) h.exact[i] = 0;
        group_sync(bar, GT);
#pragma unroll
        for (int k = 0; k < kD; ++k) {
            if (rt[k] == kNoSlot) continue;
            const uint32_t x = w[k], y = rt[k] & kIdx;
            const long long q = (long long)((int32_t)((x >> 17) & 0xFFu) * gain - ped);
            atomicAdd(&h.exact[2 * y], (unsigned long long)(q * (long long)(x & 0xFFu)));
            atomicAdd(&h.exact[2 * y + 1], (unsigned long long)(q * (long long)((x >> 8) & 0x1FFu)));
        }
        group_sync(bar, GT);
    }

    // 4
    uint32_t kr = 0; // bit k: digi k of this thread is a kept root
#pragma unroll
    for (int k = 0; k < kD; ++k) {
        const uint32_t j = gt + k * GT;
        if (j >= n) continue;
        int32_t lab = -1;
        if (rt[k] != kNoSlot) {
            const bool kept = h.q[rt[k] & kIdx] >= cthr;
            lab = kept ? (int32_t)(rt[k] >> kHashIdxBits) : -2;
            const uint32_t x = w[k], r = x & 0xFFu;
            if (kept && rt[k] == (((r * C + ((x >> 8) & 0x1FFu)) << kHashIdxBits) | j)) {
                h.par[j] = atomicAdd(&h.rowcnt[r], 1u); // arrival in the row
                kr |= 1u << k;
            }
        }
        if (it.label_e) it.label_e[__ldg(&digis[j].y)] = lab;
    }
    group_sync(bar, GT);
    if (gt == 0) *gheavy = 0; // read by every thread before the barrier above

    // 5
    uint32_t K, base8;
    {
        uint32_t s8 = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) s8 += h.rowcnt[lane * 8 + i];
        uint32_t incl = s8;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, o);
            if ((int)lane >= o) incl += y;
        }
        K = __shfl_sync(kFull, incl, 31);
        base8 = incl - s8; // kept roots in the rows before this lane's eight
    }
#pragma unroll
    for (int k = 0; k < kD; ++k) {
        if ((uint32_t)k * GT >= n) break; // uniform over the warp
        const uint32_t r = w[k] & 0xFFu;
        uint32_t pre = __shfl_sync(kFull, base8, r >> 3);
        if ((kr >> k) & 1u) {
            const uint32_t j = gt + k * GT;
            for (uint32_t i = r & ~7u; i < r; ++i) pre += h.rowcnt[i];
            h.table[pre + h.par[j]] = (w[k] >> 8) & 0x1FFu;
            h.par[j] = pre;
        }
    }
    group_sync(bar, GT);

    // 6
#pragma unroll
    for (int k = 0; k < kD; ++k) {
        if (!((kr >> k) & 1u)) continue;
        const uint32_t j = gt + k * GT, x = w[k], r = x & 0xFFu, c = (x >> 8) & 0x1FFu;
        const uint32_t pre = h.par[j], end = pre + h.rowcnt[r];
        uint32_t ord = pre;
        for (uint32_t i = pre; i < end; ++i) ord += h.table[i] < c ? 1u : 0u;
        const int32_t Q = h.q[j];
        long long mr, mc;
        if (heavy) {
            mr = (long long)h.exact[2 * j];
            mc = (long long)h.exact[2 * j + 1];
        } else {
            const int2 mm = h.m[j];
            mr = mm.x;
            mc = mm.y;
        }
        L.ws.staging.put(it.b + ord, (int32_t)(rt[k] >> kHashIdxBits), Q, (int32_t)h.np[j], centroid_abs(mr, Q),
                         centroid_abs(mc, Q));
        if (it.label16_e) h.np[j] = ord; // read back by the compact labels
    }
    if (it.label16_e) {
        group_sync(bar, GT);
#pragma unroll
        for (int k = 0; k < kD; ++k) {
            const uint32_t j = gt + k * GT;
            if (j >= n) continue;
            uint16_t v = kLab16Below;
            if (rt[k] != kNoSlot) {
                const uint32_t y = rt[k] & kIdx;
                v = h.q[y] >= cthr ? (uint16_t)h.np[y] : kLab16Dropped;
            }
            it.label16_e[__ldg(&digis[j].y)] = v;
        }
    }
    group_sync(bar, GT); // the slice is free for the group's next item
    return K;
}

// Ordered output across tickets.  chain[g] holds ticket g's aggregate (the
// number of clusters it staged, flag bit 62), published by its owner as soon
// as it is staged, without waiting; chain[ngroups + g] receives its inclusive
// prefix (flag bit 63).  The prefix spreads by a cooperative frontier:
// ctl[3] = F means tickets below F carry their inclusive prefix.  Any warp may
// push F forward: it reads the aggregates of the 32 tickets from F on, scans
// the run of consecutive published ones on top of the inclusive prefix of
// F - 1, publishes those prefixes and raises F.  Racing warps compute and
// write identical values.
__device__ void advance_frontier(unsigned long long *chain, uint32_t *frontier, uint64_t ngroups)
{
    const unsigned long long kFlagInc = 1ull << 63, kMask = (1ull << 62) - 1;
    const uint32_t lane = threadIdx.x & 31;
    unsigned long long *inc = chain + ngroups;
    for (int rounds = 0; rounds < 64; ++rounds) {
        uint32_t F = 0;
        if (lane == 0) F = *(volatile uint32_t *)frontier;
        F = __shfl_sync(kFull, F, 0);
        if (F >= ngroups) return;
        unsigned long long prev = 0;
        if (F > 0) {
            const unsigned long long pv = ld_acquire(&inc[F - 1]);
            if (!(pv & kFlagInc)) return; // the prefix below F is not visible yet
            prev = pv & kMask;
        }
        const uint64_t j = (uint64_t)F + lane;
        const unsigned long long a = j < ngroups ? ld_acquire(&chain[j]) : 0ull;
        const uint32_t avail = __ballot_sync(kFull, (a >> 62) != 0);
        const uint32_t u = (~avail) ? (uint32_t)(__ffs(~avail) - 1) : 32u; // leading run of published tickets
        if (u == 0) return;
        unsigned long long x = lane < u ? (a & kMask) : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, x, o);
            if ((int)lane >= o) x += y;
        }
        if (lane < u) st_release(&inc[j], kFlagInc | (prev + x));
        __syncwarp();
        __threadfence();
        if (lane == 0) atomicMax(frontier, F + u);
        if (u < 32) return;
    }
}

// Resolve ticket g (one full warp): its exclusive prefix once the frontier
// has passed it.  Non-blocking mode returns false if it has not; blocking
// mode keeps pushing the frontier, for at most kSpinLimit iterations and
// kWaitNs of wall time, then reports kErrTimeout (and every later blocking
// wait of the launch gives up at once).  Every aggregate is published
// without waiting, so a blocking wait only expires if one never is.
__device__ bool chain_resolve(unsigned long long *chain, uint32_t *frontier, uint64_t ngroups, uint64_t g,
                              unsigned long long agg, bool blocking, unsigned long long *excl_out,
                              uint32_t *launch_err)
{
    const unsigned long long kFlagInc = 1ull << 63, kMask = (1ull << 62) - 1;
    const uint32_t lane = threadIdx.x & 31;
    const unsigned long long *inc = chain + ngroups;
    unsigned long long t0 = 0;
    for (uint32_t spins = 0;; ++spins) {
        unsigned long long v = 0;
        uint32_t failed = 0;
        if (lane == 0) {
            v = ld_acquire(&inc[g]);
            failed = *(volatile uint32_t *)launch_err & kErrTimeout;
        }
        v = __shfl_sync(kFull, v, 0);
        failed = __shfl_sync(kFull, failed, 0);
        if (blocking && failed && !(v & kFlagInc)) {
            *excl_out = 0;
            return true;
        }
        if (!(v & kFlagInc)) {
            advance_frontier(chain, frontier, ngroups);
            if (lane == 0) v = ld_acquire(&inc[g]);
            v = __shfl_sync(kFull, v, 0);
        }
        if (v & kFlagInc) {
            *excl_out = (v & kMask) - agg;
            return true;
        }
        if (!blocking) return false;
        unsigned long long now = 0;
        if (lane == 0) now = global_ns();
        now = __shfl_sync(kFull, now, 0);
        if (spins == 0) t0 = now;
        if (spins > kSpinLimit || now - t0 > kWaitNs) {
            if (lane == 0) atomicOr(launch_err, kErrTimeout);
            *excl_out = 0;
            return true;
        }
        __nanosleep(64);
    }
}

// ---------------------------------------------------------------- clustering kernels

// What lane gt of a group's first warp loads of ticket g: its item's record
// (calibration and event start: inputs, so these can be read before the
// previous kernel is done) and then its count and bucket start.  Lanes past
// the ticket read its first item and drop it.
struct TicketLane {
    ItemRec rec;
    uint32_t count, b;
};
__device__ __forceinline__ uint32_t ticket_item(const Launch &L, uint32_t g, uint32_t lane, bool *ok)
{
    const uint32_t item = g * L.cc.ticket_items + lane;
    *ok = lane < L.cc.ticket_items && item < L.cc.items;
    return *ok ? item : g * L.cc.ticket_items;
}
__device__ __forceinline__ void load_record(const Launch &L, uint32_t g, uint32_t lane, TicketLane *t)
{
    bool ok;
    const uint32_t at = ticket_item(L, g, lane, &ok), e = L.E == 1 ? 0u : at / L.g.M, m = at - e * L.g.M;
    t->rec.e = e;
    t->rec.gain = L.g.gain[m];
    t->rec.ped = L.g.ped[m];
    t->rec.label_off = (uint32_t)L.offsets[e];
}
__device__ __forceinline__ void load_counts(const Launch &L, uint32_t g, uint32_t lane, TicketLane *t)
{
    bool ok;
    const uint32_t at = ticket_item(L, g, lane, &ok);
    t->count = L.ws.count[at];
    t->b = L.ws.boff[at];
}

// Ticket g of a group: its items' counts, bucket starts and records, and the
// plan of its first pack; false when the tickets are out.  first: t is
// loaded, and g is the group's own first ticket (dealt over the blocks before
// the groups of one); else the next one comes from a counter.
template <int GT, bool kWhole>
__device__ __forceinline__ bool take_ticket(const Launch &L, GroupShared &gs, uint32_t gt, uint32_t bar, bool first,
                                            uint32_t g, TicketLane &t)
{
    const uint32_t G = L.cc.ticket_items;
    if (gt < 32) { // one warp takes the ticket and loads its items
        if (!first) {
            if (gt == 0) g = L.cc.workers + atomicAdd(&L.ws.ctl[0], 1u);
            g = __shfl_sync(kFull, g, 0);
            if (g < L.cc.tickets) { // (every load before the first store, so that their latencies overlap)
                load_record(L, g, gt, &t);
                load_counts(L, g, gt, &t);
            }
        }
        if (g < L.cc.tickets) {
            bool ok;
            const uint32_t item = ticket_item(L, g, gt, &ok), n = ok ? t.count : 0u;
            if (gt < (uint32_t)kGroup) {
                gs.n[gt] = n;
                gs.b[gt] = t.b;
                gs.rec[gt] = t.rec;
                if (ok) {
                    if (n == 0) L.ws.cursor[item] = 0;
                    if (gt == G - 1 || item == L.cc.items - 1) gs.bucket_end = t.b + n;
                }
            }
            const uint32_t end = min(plan_pack(gs, 0, L.cc.pack_item, L.cc.pack_digis, gt, n), G);
            if (gt == 0) gs.pack_end = end;
        }
        if (gt == 0) gs.ticket = g;
    }
    gsync<GT, kWhole>(bar);
    return gs.ticket < L.cc.tickets;
}

// Pull the ticket's buckets (words and digi indices, contiguous over its
// items) into L2, one 128-byte line per thread, so that the items after the
// first do not wait on DRAM.
template <int GT>
__device__ __forceinline__ void prefetch_ticket(const Launch &L, const GroupShared &gs, uint32_t gt)
{
    const uint32_t b0 = gs.b[0], digis = gs.bucket_end - b0;
    for (uint32_t at = 16 * gt; at < digis; at += 16 * GT)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(L.ws.bucket + b0 + at));
}

// All packs of a ticket (the first is planned by take_ticket).
template <int GT, bool kWhole>
__device__ __forceinline__ void pack_ticket(const Launch &L, uint32_t mem, unsigned long long *exact,
                                            GroupShared &gs, uint16_t *wlist, uint32_t gt, uint32_t bar)
{
    for (uint32_t i0 = 0;;) {
        const uint32_t total = gs.pack[kGroup], end = gs.pack_end;
        if (total) pack_items<GT, kWhole>(L, mem, exact, i0, end - i0, total, gs, wlist, gt, bar);
        i0 = end;
        if (i0 >= L.cc.ticket_items) break;
        gsync<GT, kWhole>(bar); // the last pack's plan is read
        if (gt < 32) {
            const uint32_t e = min(plan_pack(gs, i0, L.cc.pack_item, L.cc.pack_digis, gt,
                                             i0 + gt < (uint32_t)kGroup ? gs.n[i0 + gt] : 0u),
                                   L.cc.ticket_items);
            if (gt == 0) gs.pack_end = e;
        }
        gsync<GT, kWhole>(bar);
    }
}

// The clustering kernel, persistent: kGroups groups of kThreads / kGroups
// threads a block, each with its own slice of the block's shared memory, its
// own named barrier and its own tickets of consecutive items, so that one
// group's barriers and loads overlap the others' work.  Items of at most
// cc.pack_item digis go through the packed tier, a ticket's worth at a time,
// the others through the run tier one by one.  (A module's bitmap costs its
// clearing and scan whatever it holds, a pack's list of touched words costs
// each digi: the line is pack_max.)  Items of more than
// cc.large_digis digis (scan_kernel lists them; with cc.own a block looks at
// its own item), whose runs would not fit a slice or which are few, come first:
// the whole block takes them one at a time, on all of its
// shared memory, held in registers up to kRunDigis a thread (items of 4,500
// digis: 24.9 -> 22.2 us a million digis, of 8,000: 20.7 -> 19.3; four items
// of 2,500 at once: 17.2, which is why the groups have the rest).  64 registers
// a thread, which 1,024 threads an SM leave, spill a little outside the inner
// loops (80 to 90 bytes of stores and 52 of loads a thread).
template <int kThreads, int kGroups, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks) cc_kernel(const __grid_constant__ Launch L)
{
    constexpr int GT = kThreads / kGroups;
    constexpr bool kWhole = kGroups == 1;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ GroupShared s_gs[kGroups];
    __shared__ uint16_t s_wlist[kThreads / 32][64];
    const uint32_t tid = threadIdx.x, gid = tid / GT, gt = tid - gid * GT, bar = 1 + gid;
    // the group's first ticket: its records before the previous kernel is done
    // (the launch's first kernel is an ordinary launch, so that the call's
    // inputs are in place when this one starts)
    const uint32_t ticket0 = gid * gridDim.x + blockIdx.x;
    TicketLane lane_of;
    if (gt < 32 && ticket0 < L.cc.tickets) load_record(L, ticket0, gt, &lane_of);
    pdl_wait();
    pdl_trigger();
    const uint32_t launch_err = L.ws.ctl[1], nlarge = kWhole ? 0u : L.ws.ctl[5];
    if (gt < 32 && ticket0 < L.cc.tickets) load_counts(L, ticket0, gt, &lane_of);
    if (launch_err & kErrBadOffsets) return;

    uint16_t *wlist = s_wlist[tid >> 5];
    unsigned long long *exact = L.ws.exact + (size_t)blockIdx.x * 2 * L.cc.exact_slots;
    uint32_t *kcount = L.ws.cursor; // each item's count of kept clusters

    if constexpr (!kWhole) {
        if (nlarge) {
            GroupShared &gs = s_gs[0];
            bool come = true;
            // where several blocks share an SM and the list is short, only the
            // first of each SM comes for it: two at work on one SM take 1.6 times
            // as long (ten items of 13,000 digis 210 -> 130 us)
            if constexpr (kMinBlocks > 1) {
                if (!L.cc.own && nlarge <= (uint32_t)L.sm_count) {
                    if (tid == 0) {
                        const uint32_t sm = sm_id() & 255u, bit = 1u << (sm & 31u);
                        gs.flag = atomicOr(&L.ws.ctl[8 + (sm >> 5)], bit) & bit;
                    }
                    __syncthreads();
                    come = gs.flag == 0;
                }
            }
            while (come) {
                if (tid == 0) {
                    uint32_t t, item = blockIdx.x;
                    if (L.cc.own) {
                        t = item < L.cc.items && L.ws.count[item] > L.cc.large_digis ? 0u : nlarge;
                    } else {
                        t = atomicAdd(&L.ws.ctl[7], 1u);
                        if (t < nlarge) item = L.ws.large[t];
                    }
                    gs.ticket = t;
                    if (t < nlarge) {
                        gs.pack_end = item;
                        gs.n[0] = L.ws.count[item];
                        gs.b[0] = L.ws.boff[item];
                        gs.rec[0] = make_rec(L, item);
                    }
                }
                __syncthreads();
                if (gs.ticket >= nlarge) break;
                const ItemCtx it = make_item(L, gs.rec[0], gs.b[0], gs.n[0]);
                const uint32_t item = gs.pack_end;
                const uint32_t K =
                    it.n <= (uint32_t)(kRunDigis * kThreads)
                        ? run_item<kThreads, true, kWide, true>(L, it, smem_addr(dsm), L.cc.whole_runs, exact, 0, 1, gs,
                                                                wlist, tid, 0)
                        : run_item<kThreads, true, kWide, false>(L, it, smem_addr(dsm), L.cc.whole_runs, exact, 0, 1,
                                                                 gs, wlist, tid, 0);
                if (tid == 0) kcount[item] = K;
                if (L.cc.own) break;
                __syncthreads();
            }
        }
        __syncthreads();
    }

    const uint32_t mem = smem_addr(dsm) + L.cc.slice * gid;
    exact += (size_t)2 * L.cc.runs * gid;
    GroupShared &gs = s_gs[gid];
    for (bool first = true; take_ticket<GT, kWhole>(L, gs, gt, bar, first, ticket0, lane_of); first = false) {
        prefetch_ticket<GT>(L, gs, gt);
        pack_ticket<GT, kWhole>(L, mem, exact, gs, wlist, gt, bar);
        for (uint32_t i = 0; i < L.cc.ticket_items; ++i) {
            const uint32_t n = gs.n[i];
            if (n <= L.cc.pack_item || (!kWhole && n > L.cc.large_digis)) continue;
            const ItemCtx it = make_item(L, gs.rec[i], gs.b[i], n);
            constexpr RunKind kMulti = kWhole ? kWide : kNarrow; // (of groups: at most cc.large_digis digis)
            static_assert(kRunDigis * GT <= kNarrowDigis, "items held in registers");
            const uint32_t K = n <= (uint32_t)(kRunDigis * GT)
                                   ? run_item<GT, kWhole, kNarrow, true>(L, it, mem, L.cc.runs, exact, gid, kGroups,
                                                                gs, wlist, gt, bar)
                                   : run_item<GT, kWhole, kMulti, false>(L, it, mem, L.cc.runs, exact, gid, kGroups,
                                                                 gs, wlist, gt, bar);
            if (gt == 0) kcount[gs.ticket * L.cc.ticket_items + i] = K;
        }
        gsync<GT, kWhole>(bar); // the ticket's record is free
    }
}

// The clustering kernel with the hash label store (tuning label_store =
// kStoreHash): one ticket a block at a time; items of more than warp_max digis
// and within the store's capacity go to groups of item_threads threads,
// smaller ones through the packed tier and larger ones through the run tier,
// both by the whole block.
template <int kMinBlocks>
__global__ void __launch_bounds__(kCCThreads, kMinBlocks) cc_hash_kernel(const __grid_constant__ Launch L)
{
    constexpr int GT0 = kCCThreads;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ GroupShared gs;
    __shared__ uint32_t s_gflag[kCCThreads / 128], s_gheavy[kCCThreads / 128];
    pdl_wait();
    pdl_trigger();
    if (L.ws.ctl[1] & kErrBadOffsets) return;

    const uint32_t T = L.tune.tile_slots, tid = threadIdx.x;
    constexpr int kD = cc_digis_per_thread(kMinBlocks);
    const size_t smem = L.cc.slice;
    // the run tier's warp lists, at the end of the dynamic shared memory
    uint16_t *wlist = reinterpret_cast<uint16_t *>(dsm + (smem & ~(size_t)1) - kHashListBytes) + 64 * (tid >> 5);
    unsigned long long *exact = L.ws.exact + (size_t)blockIdx.x * 2 * L.cc.exact_slots;
    const uint32_t GT = L.tune.item_threads, hgroups = (uint32_t)kCCThreads / GT;
    const uint32_t hash_max = hash_capacity(smem, T, GT, (uint32_t)kD);
    const uint32_t gid = tid / GT, gtid = tid - gid * GT;
    const HashMem hm = hash_mem(dsm, smem, hgroups, gid, hash_max, exact);
    if (tid < (uint32_t)(kCCThreads / 128)) {
        s_gflag[tid] = 0;
        s_gheavy[tid] = 0;
    }
    uint32_t *kcount = L.ws.cursor;
    TicketLane lane_of;
    if (tid < 32 && blockIdx.x < L.cc.tickets) {
        load_record(L, blockIdx.x, tid, &lane_of);
        load_counts(L, blockIdx.x, tid, &lane_of);
    }
    for (bool first = true; take_ticket<GT0, true>(L, gs, tid, 0, first, blockIdx.x, lane_of); first = false) {
        prefetch_ticket<GT0>(L, gs, tid);
        pack_ticket<GT0, true>(L, smem_addr(dsm), exact, gs, wlist, tid, 0);
        const uint32_t item0 = gs.ticket * L.cc.ticket_items;
        // the items above the packed tier and within the store's capacity,
        // dealt round-robin to the block's groups
        uint32_t nh = 0;
        for (uint32_t i = 0; i < L.cc.ticket_items; ++i) {
            const uint32_t n = gs.n[i];
            if (n <= L.cc.pack_item || n > hash_max) continue;
            if (nh++ % hgroups != gid) continue;
            const ItemCtx it = make_item(L, gs.rec[i], gs.b[i], n);
            const uint32_t K = hash_item<kD>(L, it, hm, gtid, GT, 1 + gid, &s_gflag[gid], &s_gheavy[gid]);
            if (gtid == 0) kcount[item0 + i] = K;
        }
        __syncthreads();
        for (uint32_t i = 0; i < L.cc.ticket_items; ++i) {
            const uint32_t n = gs.n[i];
            if (n <= L.cc.pack_item || n <= hash_max) continue;
            const ItemCtx it = make_item(L, gs.rec[i], gs.b[i], n);
            const uint32_t K = run_item<GT0, true, kWide, false>(L, it, smem_addr(dsm), L.cc.runs, exact, 0, 1, gs,
                                                          wlist, tid, 0);
            if (tid == 0) kcount[item0 + i] = K;
        }
        __syncthreads(); // the ticket's record is free
    }
}


// Ordered output, in two kernels.
//
// offsets_kernel: block c takes chunk c of kOffItems consecutive items (in
// the order blocks start, so the chunks below it are running or done), scans
// the items' kept-cluster counts (cursor[], from cc_kernel), publishes the
// chunk's total in chain[c] and resolves its exclusive prefix with the
// cooperative frontier (a bounded wait; few, large chunks keep the frontier
// short); it writes every item's first output position to count[] (free
// since cc_kernel read it), the cluster offsets of the events that start in
// the chunk, and the capacity check.
constexpr int kOffThreads = 1024;
constexpr uint32_t kOffItems = kOffThreads;

__global__ void __launch_bounds__(kOffThreads) offsets_kernel(const Launch L)
{
    __shared__ uint32_t s_tmp[kOffThreads / 32 + 1];
    __shared__ uint32_t s_chunk;
    pdl_wait();
    pdl_trigger();
    __shared__ unsigned long long s_prefix;
    const uint32_t tid = threadIdx.x, M = L.g.M;
    const uint64_t EM = (uint64_t)L.E * M;
    const uint64_t nchunks = (EM + kOffItems - 1) / kOffItems;
    if (L.ws.ctl[1] & kErrBadOffsets) return;
    if (tid == 0) s_chunk = atomicAdd(&L.ws.ctl[4], 1u);
    __syncthreads();
    const uint64_t c = s_chunk;
    if (c >= nchunks) return;
    const uint64_t item = c * kOffItems + tid;
    const bool in = item < EM;
    const uint32_t k = in ? L.ws.cursor[item] : 0u;
    uint32_t total;
    const uint32_t ex = block_exclusive_scan<kOffThreads>(k, s_tmp, &total);
    if (tid < 32) {
        // The chunk's total is all that other blocks read of it, so a relaxed
        // store suffices.  (The test hook kDebugWithholdTicket0 keeps chunk
        // 0's total back, so that the waits on it expire.)
        const unsigned long long kAgg = 1ull << 62;
        if (tid == 0 && (c != 0 || !(L.debug & kDebugWithholdTicket0))) st_relaxed(&L.ws.chain[c], kAgg | total);
        __syncwarp();
        unsigned long long P = 0;
        chain_resolve(L.ws.chain, &L.ws.ctl[3], nchunks, c, total, true, &P, &L.ws.ctl[1]);
        if (tid == 0) s_prefix = P;
    }
    __syncthreads();
    const unsigned long long P = s_prefix;
    if (in) {
        const unsigned long long o = P + ex;
        L.ws.count[item] = (uint32_t)o;
        uint32_t e, m;
        item_coords(item, M, &e, &m);
        if (m == 0) L.out.cluster_offsets[e] = o;
        // the output chunks whose first position falls in this item's range
        if (k > 0)
            for (unsigned long long q = (o + kOutChunk - 1) / kOutChunk; q * kOutChunk < o + k; ++q)
                L.ws.chunk_item[q] = (uint32_t)item;
    }
    if (tid == 0 && c == nchunks - 1) {
        L.out.cluster_offsets[L.E] = P + total;
        L.ws.ctl[6] = (uint32_t)(P + total);
    }
    if (tid == 0 && P + total > L.out.capacity) atomicOr(&L.ws.ctl[1], kErrCapacity);
}

// Output positions p0 .. p0 + 3 (those below T) of one thread: `it` is the
// item of p0, its clusters the positions [start, start + K); next(i, &start,
// &K) gives those of item i.
template <class F>
__device__ __forceinline__ void copy_positions(const Launch &L, uint32_t p0, uint32_t T, bool vec, uint32_t it,
                                               uint32_t start, uint32_t K, F &&next)
{
    const Staging sg = L.ws.staging;
    const uint32_t M = L.g.M;
    const uint32_t nv = min(4u, T - p0);
    uint32_t mo[4];
    int32_t id[4], q[4], np[4];
    float x[4], y[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        mo[j] = 0;
        id[j] = q[j] = np[j] = 0;
        x[j] = y[j] = 0.f;
        if ((uint32_t)j >= nv) continue;
        const uint32_t p = p0 + j;
        while (p - start >= K) { // on to the item holding p (count[it + 1] = start + K)
            ++it;
            next(it, &start, &K);
        }
        const uint64_t a = (uint64_t)L.ws.boff[it] + (p - start);
        uint32_t e, m;
        item_coords(it, M, &e, &m);
        mo[j] = m;
        id[j] = sg.id[a];
        q[j] = sg.charge[a];
        np[j] = sg.npix[a];
        x[j] = sg.x[a];
        y[j] = sg.y[a];
    }
    const ClusterCols host = {L.out.module, L.out.id, L.out.charge, L.out.npix, L.out.x, L.out.y};
    const bool in_head = p0 + nv <= L.out.head_n, past_head = p0 >= L.out.head_n;
    if (nv == 4 && (in_head || (past_head && vec))) {
        const ClusterCols &d = in_head ? L.out.head : host;
        *reinterpret_cast<uint4 *>(d.module + p0) = make_uint4(mo[0], mo[1], mo[2], mo[3]);
        *reinterpret_cast<int4 *>(d.id + p0) = make_int4(id[0], id[1], id[2], id[3]);
        *reinterpret_cast<int4 *>(d.charge + p0) = make_int4(q[0], q[1], q[2], q[3]);
        *reinterpret_cast<int4 *>(d.npix + p0) = make_int4(np[0], np[1], np[2], np[3]);
        *reinterpret_cast<float4 *>(d.x + p0) = make_float4(x[0], x[1], x[2], x[3]);
        *reinterpret_cast<float4 *>(d.y + p0) = make_float4(y[0], y[1], y[2], y[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if ((uint32_t)j >= nv) continue;
            const ClusterCols &d = p0 + j < L.out.head_n ? L.out.head : host;
            d.module[p0 + j] = mo[j];
            d.id[p0 + j] = id[j];
            d.charge[p0 + j] = q[j];
            d.npix[p0 + j] = np[j];
            d.x[p0 + j] = x[j];
            d.y[p0 + j] = y[j];
        }
    }
}

// 16-byte stores into the output columns are possible.
__device__ __forceinline__ bool columns_aligned(const Outputs &o)
{
    return ((reinterpret_cast<uintptr_t>(o.module) | reinterpret_cast<uintptr_t>(o.id) |
             reinterpret_cast<uintptr_t>(o.charge) | reinterpret_cast<uintptr_t>(o.npix) |
             reinterpret_cast<uintptr_t>(o.x) | reinterpret_cast<uintptr_t>(o.y)) & 15) == 0;
}

// Status code of an event with these error bits (its own and the launch's).
__device__ __forceinline__ int32_t event_status(uint32_t bits)
{
    if (bits & kErrBadOffsets) return 3; // HP_EINVAL
    if (bits & kErrTimeout) return 8;    // HP_ETIMEOUT
    if (bits & kErrCapacity) return 6;   // HP_ECAPACITY
    if (bits & kErrBadDigi) return 4;    // HP_EBADDIGI
    if (bits & kErrDup) return 5;        // HP_EDUP
    return 0;                            // HP_OK
}

// copy_kernel: the staged clusters (SoA, at each item's bucket start) to
// their ordered output positions, driven by the output: a warp takes a chunk
// of kOutChunk consecutive positions, four a lane, finds the item of its
// first position by a binary search between the items that hold the first
// positions of this chunk and the next (chunk_item[], from offsets_kernel),
// and walks on from there.  Every warp store is then a whole, aligned 512-byte
// run of one output array, which matters most when the outputs are mapped
// host memory written over the chip-to-chip link (partial lines cost there).
// The first E threads write the per-event status codes from the error bits.
constexpr int kCopyThreads = 256;

__global__ void __launch_bounds__(kCopyThreads) copy_kernel(const Launch L)
{
    pdl_wait();
    const uint32_t lane = threadIdx.x & 31, M = L.g.M;
    const uint64_t gt = (uint64_t)blockIdx.x * kCopyThreads + threadIdx.x;
    const bool bad_offsets = (L.ws.ctl[1] & kErrBadOffsets) != 0;
    if (bad_offsets && gt <= L.E) L.out.cluster_offsets[gt] = 0; // no clusters
    if (gt < L.E) {
        L.out.event_status[gt] = event_status(L.ws.event_err[gt] | L.ws.ctl[1]);
    }
    if (bad_offsets) return;
    const uint32_t total = L.ws.ctl[6];
    const uint32_t T = (uint32_t)min((unsigned long long)total, (unsigned long long)L.out.capacity);
    const uint32_t nchunks = (uint32_t)(((uint64_t)total + kOutChunk - 1) / kOutChunk);
    const uint32_t last_item = (uint32_t)((uint64_t)L.E * M - 1);
    const bool vec = columns_aligned(L.out);
    const uint64_t warps = (uint64_t)gridDim.x * (kCopyThreads / 32);
    for (uint64_t ch = gt >> 5; ch < nchunks; ch += warps) {
        const uint32_t p0 = (uint32_t)ch * kOutChunk + 4 * lane;
        if (p0 >= T) continue;
        // the item of p0: the last one in [lo, hi] whose range starts at or
        // before p0 (empty items share their start with the next item)
        uint32_t lo = L.ws.chunk_item[ch];
        uint32_t hi = ch + 1 < nchunks ? L.ws.chunk_item[ch + 1] : last_item;
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1) >> 1;
            if (L.ws.count[mid] <= p0) lo = mid;
            else hi = mid - 1;
        }
        uint32_t it = lo, start = L.ws.count[it], K = L.ws.cursor[it];
        copy_positions(L, p0, T, vec, it, start, K, [&](uint32_t i, uint32_t *start_, uint32_t *k_) {
            *start_ = L.ws.count[i];
            *k_ = L.ws.cursor[i];
        });
    }
    // with compact labels: every item's first cluster counted from its event's first
    if (L.out.item_first) {
        const uint64_t EM = (uint64_t)L.E * M;
        for (uint64_t item = gt; item < EM; item += (uint64_t)gridDim.x * kCopyThreads)
            L.out.item_first[item] = L.ws.count[item] - L.ws.count[item - item % M];
    }
}

// finish_kernel: offsets_kernel and copy_kernel in one, for launches of few
// items (finish_fits): every block scans all items' counts for itself (in
// shared memory, so no block waits for another), then copies its share of the
// output positions, one a thread (whole lines a warp, and one chain of loads a
// thread), finding its item by a binary search there.  Bound by launch latency
// and a handful of L2 round trips.
constexpr int kFinishThreads = 1024;

__global__ void __launch_bounds__(kFinishThreads) finish_kernel(const __grid_constant__ Launch L)
{
    extern __shared__ uint32_t offs[]; // [EM + 1] first output position of each item
    __shared__ uint32_t tmp[kFinishThreads / 32 + 1];
    pdl_wait();
    const uint32_t tid = threadIdx.x, M = L.g.M, EM = L.cc.items;
    const uint64_t gt = (uint64_t)blockIdx.x * kFinishThreads + tid;
    const uint32_t launch_bits = L.ws.ctl[1], err0 = gt < L.E ? L.ws.event_err[gt] : 0u;
    if (launch_bits & kErrBadOffsets) {
        for (uint64_t e = gt; e <= L.E; e += (uint64_t)gridDim.x * kFinishThreads) {
            L.out.cluster_offsets[e] = 0; // no clusters
            if (e < L.E) L.out.event_status[e] = event_status(launch_bits);
        }
        return;
    }
    for (uint32_t i = tid; i < EM; i += kFinishThreads) offs[i] = L.ws.cursor[i];
    __syncthreads();
    const uint32_t per = ((EM + kFinishThreads - 1) / kFinishThreads) | 1u; // odd: no bank conflicts
    const uint32_t i0 = min(EM, tid * per), i1 = min(EM, i0 + per);
    uint32_t sum = 0, total;
    for (uint32_t i = i0; i < i1; ++i) sum += offs[i];
    uint32_t run = block_exclusive_scan<kFinishThreads>(sum, tmp, &total);
    for (uint32_t i = i0; i < i1; ++i) {
        const uint32_t k = offs[i];
        offs[i] = run;
        run += k;
    }
    if (tid == 0) offs[EM] = total;
    __syncthreads();
    const uint32_t bits = launch_bits | (total > L.out.capacity ? kErrCapacity : 0u);
    for (uint64_t e = gt; e <= L.E; e += (uint64_t)gridDim.x * kFinishThreads) {
        L.out.cluster_offsets[e] = offs[e * M];
        if (e < L.E) L.out.event_status[e] = event_status((e == gt ? err0 : L.ws.event_err[e]) | bits);
    }
    const uint32_t T = (uint32_t)min((unsigned long long)total, (unsigned long long)L.out.capacity);
    const Staging sg = L.ws.staging;
    const ClusterCols host = {L.out.module, L.out.id, L.out.charge, L.out.npix, L.out.x, L.out.y};
    for (uint64_t at = gt; at < T; at += (uint64_t)gridDim.x * kFinishThreads) {
        const uint32_t p = (uint32_t)at;
        uint32_t lo = 0, hi = EM - 1; // the last item that starts at or before p
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1) >> 1;
            if (offs[mid] <= p) lo = mid;
            else hi = mid - 1;
        }
        const uint64_t a = (uint64_t)L.ws.boff[lo] + (p - offs[lo]);
        const ClusterCols &d = p < L.out.head_n ? L.out.head : host;
        d.module[p] = L.E == 1 ? lo : lo % M;
        const int32_t id = sg.id[a], q = sg.charge[a], np = sg.npix[a];
        const float x = sg.x[a], y = sg.y[a];
        d.id[p] = id;
        d.charge[p] = q;
        d.npix[p] = np;
        d.x[p] = x;
        d.y[p] = y;
    }
    if (L.out.item_first)
        for (uint64_t item = gt; item < EM; item += (uint64_t)gridDim.x * kFinishThreads)
            L.out.item_first[item] = offs[item] - offs[item - item % M];
}

// Serving batches: block (x, e) copies a slice of request e's digis.
// Four digis a thread, read with one 16-byte (words) and one 8-byte
// (module ids) load where the source allows it: the sources are host memory
// read over the chip-to-chip link, where wide loads carry more per request.
__global__ void __launch_bounds__(256) gather_kernel(const GatherEntry *table, uint32_t *words, uint16_t *modules)
{
    const GatherEntry g = table[blockIdx.y];
    const bool wv = (reinterpret_cast<uintptr_t>(g.words) & 15) == 0;
    const bool mv = (reinterpret_cast<uintptr_t>(g.modules) & 7) == 0;
    const uint64_t n4 = g.n / 4, stride = (uint64_t)gridDim.x * blockDim.x;
    uint32_t *dw = words + g.off;
    uint16_t *dm = modules + g.off;
    for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += stride) {
        uint32_t w[4];
        uint16_t m[4];
        if (wv) {
            const uint4 v = reinterpret_cast<const uint4 *>(g.words)[q];
            w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = g.words[4 * q + j];
        }
        if (mv) {
            const ushort4 v = reinterpret_cast<const ushort4 *>(g.modules)[q];
            m[0] = v.x, m[1] = v.y, m[2] = v.z, m[3] = v.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) m[j] = g.modules[4 * q + j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            dw[4 * q + j] = w[j];
            dm[4 * q + j] = m[j];
        }
    }
    for (uint64_t i = 4 * n4 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += stride) {
        dw[i] = g.words[i];
        dm[i] = g.modules[i];
    }
}

} // namespace

cudaError_t launch_gather(const GatherEntry *table, uint32_t n_requests, uint64_t max_n, uint32_t *words,
                          uint16_t *modules, cudaStream_t stream)
{
    if (n_requests == 0 || max_n == 0) return cudaSuccess;
    const uint64_t bx = std::min<uint64_t>(32, (max_n + 4095) / 4096);
    gather_kernel<<<dim3((unsigned)bx, n_requests), 256, 0, stream>>>(table, words, modules);
    return cudaGetLastError();
}

size_t carve_workspace(void *base, uint32_t E, uint32_t M, uint64_t N, uint32_t R, uint32_t C, int cc_grid,
                       const Tuning &tune, Workspace *ws, int sm_count)
{
    size_t off = 0;
    auto take = [&](size_t bytes) -> unsigned char * {
        off = (off + 255) & ~(size_t)255;
        const size_t o = off;
        off += bytes;
        return base ? static_cast<unsigned char *>(base) + o : nullptr;
    };
    const uint64_t EM = (uint64_t)E * M;
    const uint64_t nchunks = (EM + kOffItems - 1) / kOffItems;
    Workspace w{};
    w.ctl = reinterpret_cast<uint32_t *>(take(64));
    w.event_err = reinterpret_cast<uint32_t *>(take(4ull * E));
    w.count = reinterpret_cast<uint32_t *>(take(4ull * EM));
    w.count2 = reinterpret_cast<uint32_t *>(take(4ull * EM));
    w.chain = reinterpret_cast<unsigned long long *>(take(16ull * nchunks)); // aggregates, then inclusive prefixes
    off = (off + 255) & ~(size_t)255;
    w.zero_bytes = off;
    w.boff = reinterpret_cast<uint32_t *>(take(4ull * EM));
    w.blk_off = reinterpret_cast<uint32_t *>(take(4ull * kHistCap * bucket_grid(N, sm_count)));
    w.cursor = reinterpret_cast<uint32_t *>(take(4ull * EM));
    w.bucket = reinterpret_cast<uint2 *>(take(8ull * N));
    w.chunk_item = reinterpret_cast<uint32_t *>(take(4ull * (N / kOutChunk + 2)));
    w.staging.id = reinterpret_cast<int32_t *>(take(4ull * N));
    w.staging.charge = reinterpret_cast<int32_t *>(take(4ull * N));
    w.staging.npix = reinterpret_cast<int32_t *>(take(4ull * N));
    w.staging.x = reinterpret_cast<float *>(take(4ull * N));
    w.staging.y = reinterpret_cast<float *>(take(4ull * N));
    w.large = reinterpret_cast<uint32_t *>(take(4ull * EM));
    const bool hash = tune.label_store == kStoreHash;
    const RunShape sh = run_shape(tune, EM, N, cc_grid);
    w.exact = reinterpret_cast<unsigned long long *>(
        take(16ull * (hash ? tune.tile_slots : run_exact_slots(R, C, tune.tile_slots, sh.groups)) *
             (cc_grid > 0 ? cc_grid : 1)));
    // a slab holds any item, and an item of each group at once (a group's
    // part holds the largest item it takes: see large_digis)
    const uint64_t any = std::min<uint64_t>((uint64_t)R * C, N);
    const uint64_t slab_slots =
        sh.groups > 1 ? std::max(any, sh.groups * std::min<uint64_t>(any, large_digis(R, C, tune.tile_slots, sh))) : any;
    const uint64_t slab_total = slab_slots * (uint64_t)(cc_grid > 0 ? cc_grid : 1);
    w.big_arena = N <= slab_total ? 1 : 0;
    w.big_slots = w.big_arena ? N : slab_slots;
    w.big = take(kBigSlotBytes * (w.big_arena ? N : slab_total));
    off = (off + 255) & ~(size_t)255;
    if (ws) *ws = w;
    return off;
}

namespace {

// Largest tile (a multiple of 256 slots, at most max_slots) with which
// `blocks` blocks of `kern` (`threads` threads, bytes(tile) of dynamic shared
// memory) stay resident on one SM; 0 if none does.  Also raises the kernel's
// dynamic shared memory limit to the most the device gives: the limit is the
// process's, not the context's, and a context for other modules must not lower
// it under one that lives (bytes() does not even grow with the module: slices
// fall back to 256 runs where larger ones would not fit).
template <class K, class F>
cudaError_t fit_tile(K kern, int device, int blocks, int threads, F bytes, uint32_t max_slots, uint32_t *tile)
{
    *tile = 0;
    int optin = 0;
    cudaError_t err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (err != cudaSuccess) return err;
    cudaFuncAttributes fa;
    err = cudaFuncGetAttributes(&fa, kern);
    if (err != cudaSuccess) return err;
    const size_t limit = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
    uint32_t t = max_slots;
    while (t >= 256 && bytes(t) > limit) t -= 256;
    if (t < 256) return cudaSuccess;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
    if (err != cudaSuccess) return err;
    for (; t >= 256; t -= 256) {
        int nb = 0;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, bytes(t));
        if (err != cudaSuccess) return err;
        if (nb >= blocks) {
            *tile = t;
            break;
        }
    }
    return cudaSuccess;
}

} // namespace

cudaError_t init_kernels(int device, uint32_t R, uint32_t C, uint32_t max_tile[4], uint32_t hash_tile[4])
{
    cudaError_t err = cudaSetDevice(device);
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScatterSmem);
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(scatter_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmem);
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(bucket_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)bucket_smem(kBucketModules, false));
    if (err == cudaSuccess)
        err = cudaFuncSetAttribute(bucket_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)bucket_smem(kBucketModules, true));
    if (err == cudaSuccess)
        err = cudaFuncSetAttribute(finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)((kFinishItems + 1) * 4));
    if (err != cudaSuccess) return err;
    max_tile[0] = hash_tile[0] = 0;
    auto run_bytes = [&](uint32_t groups) { return [=](uint32_t t) { return run_smem_bytes(R, C, t, groups); }; };
    auto hash_bytes = [&](uint32_t t) { return cc_smem_bytes(R, C, t); };
    err = fit_tile(cc_kernel<kRunThreads1, kRunGroups1, 1>, device, 1, kRunThreads1, run_bytes(kRunGroups1),
                   kMaxTileSlots, &max_tile[1]);
    if (err == cudaSuccess)
        err = fit_tile(cc_kernel<kRunThreads2, kRunGroups2, 2>, device, 2, kRunThreads2, run_bytes(kRunGroups2),
                       kSmemSlots, &max_tile[2]);
    uint32_t narrow = 0; // (the two-block kernel with more groups: the same tiles)
    if (err == cudaSuccess)
        err = fit_tile(cc_kernel<kRunThreads2n, kRunGroups2n, 2>, device, 2, kRunThreads2n, run_bytes(kRunGroups2n),
                       kSmemSlots, &narrow);
    max_tile[2] = std::min(max_tile[2], narrow);
    if (err == cudaSuccess)
        err = fit_tile(cc_kernel<kRunThreads3, kRunGroups3, 3>, device, 3, kRunThreads3, run_bytes(kRunGroups3),
                       kSmemSlots, &max_tile[3]);
    if (err == cudaSuccess)
        err = fit_tile(cc_hash_kernel<1>, device, 1, kCCThreads, hash_bytes, kMaxTileSlots, &hash_tile[1]);
    if (err == cudaSuccess)
        err = fit_tile(cc_hash_kernel<2>, device, 2, kCCThreads, hash_bytes, kSmemSlots, &hash_tile[2]);
    if (err == cudaSuccess)
        err = fit_tile(cc_hash_kernel<3>, device, 3, kCCThreads, hash_bytes, kSmemSlots, &hash_tile[3]);
    // one tile for both label stores, so that a setting's store can be changed alone
    for (int b = 1; b <= 3; ++b)
        if (hash_tile[b] && hash_tile[b] < max_tile[b]) max_tile[b] = hash_tile[b];
    return err;
}

const char *const kKernelNames[kNumKernels] = {"hist_kernel",   "scan_kernel",         "scatter_kernel", "cc_kernel",
                                                "offsets_kernel", "copy_kernel",         "bucket_kernel",
                                                "scatter_wide_kernel", "cc_hash_kernel", "finish_kernel"};

// Sizes of a launch's clustering kernel: its tickets, and what a group's
// slice of the shared memory (and the whole of it) holds.
static ClusterPlan cluster_plan(const Launch &L)
{
    const uint32_t R = L.g.R, C = L.g.C, T = L.tune.tile_slots;
    const bool hash = L.tune.label_store == kStoreHash;
    ClusterPlan p;
    p.items = (uint32_t)((uint64_t)L.E * L.g.M); // at most 2^31 (checked by the callers)
    const RunShape sh = run_shape(L.tune, p.items, L.N, L.cc_grid);
    const uint32_t groups = sh.groups;
    p.threads = sh.threads;
    p.workers = (uint32_t)L.cc_grid * groups;
    p.ticket_items = ticket_items(p.items, p.workers, L.tune.ticket_max, L.N);
    // small items: no more a ticket than fill the last round of tickets
    if (!large_items(L.N, p.items)) {
        const uint64_t per = (uint64_t)p.workers * p.ticket_items, rounds = (p.items + per - 1) / per;
        const uint64_t fill = (p.items + p.workers * rounds - 1) / (p.workers * rounds);
        p.ticket_items = (uint32_t)std::min<uint64_t>(p.ticket_items, std::max<uint64_t>(4, fill));
    }
    p.tickets = (p.items + p.ticket_items - 1) / p.ticket_items;
    p.smem = (uint32_t)(hash ? cc_smem_bytes(R, C, T) : run_smem_bytes(R, C, T, groups));
    p.slice = (p.smem / groups) & ~15u;
    p.whole_runs = run_capacity(p.smem, R, C);
    p.runs = run_capacity(p.slice, R, C);
    p.exact_slots = hash ? T : run_exact_slots(R, C, T, groups);
    if (hash) p.runs = std::min(run_capacity(p.slice - kHashListBytes, R, C), T);
    p.pack_digis = std::min(pack_capacity(hash ? p.slice - kHashListBytes : p.slice, R, p.runs),
                            (uint32_t)kPackPer * sh.threads / groups);
    p.pack_item = std::min(hash ? L.tune.warp_max : pack_max(L.tune.warp_max), p.pack_digis);
    p.large_digis = std::min(large_digis(R, C, T, sh), groups > 1 ? kNarrowDigis : 0xFFFFFFFFu);
    // With no more items than blocks a group's neighbours are idle, and larger
    // items take the whole block: with an item a ticket each block its own (with
    // a list, a block that clustered another's item came to its own item after
    // it: 128 items of 1,900-2,100 digis 51 us, 48 with a whole block for every
    // item, 37 so).  The line is five digis a thread of a group; 64 to 300 items,
    // a group / the whole block: of 1,200 digis 31-36 us either way, of 1,600
    // 34-41 / 32-36, of 1,800 38-47 / 33-37.  Else what a group holds in registers.
    p.own = groups > 1 && p.ticket_items == 1 && p.items <= (uint32_t)L.cc_grid;
    if (groups > 1 && p.items <= (uint32_t)L.cc_grid)
        p.large_digis = std::min(p.large_digis, (uint32_t)(p.own ? 5 : kRunDigis) * (sh.threads / groups));
    return p;
}

// Launch `kern` on `stream` as a programmatic dependent of the kernel before it.
template <typename K>
cudaError_t launch_dependent(K kern, unsigned grid, unsigned block, size_t smem, cudaStream_t stream, const Launch &L)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, L);
}

// Clusters that bucket_kernel needs besides one an event, where any of the
// events may hold most of the launch's digis.
static uint64_t bucket_parts(const Launch &L)
{
    return L.max_event || L.N <= kBucketDigis ? 0 : L.N / kBucketDigis;
}

// Whether the launch's digis are bucketed by bucket_kernel (one launch, a
// cluster an event) and its clusters ordered by finish_kernel, instead of by
// three kernels and two: small launches, whose time is that of the kernel
// boundaries (one event of 1,300 digis 36 -> 23 us, of 60,000 on 1,856 modules
// 49 -> 31 us).  The largest event decides, for an event is bucketed by eight
// blocks: in several steps it lost against the three kernels (events of 400,000
// and three times 30,000 digis: 84 us against 55; of 1.9M and fifteen times
// 2,000: 754 against 620).  Where the offsets are the device's, a launch of more
// than kBucketDigis gets as many clusters as its events can have parts, which
// costs even events 1 us and the others little or nothing (those of 400,000
// and 30,000: 61 us; of 250,000 and 10,000: 44 against 46; 9 even events of 0.3
// to 1M digis in all 13% less than with the three kernels).  8 events of
// 130,000 digis: 50 us against 56; 16, which take two rounds of clusters, of
// 60,000 2% less, of 130,000: 85 against 81.
static bool bucket_fits(const Launch &L)
{
    return L.N > 0 && L.N <= (L.E <= kBucketAtOnce ? kSmallDigis : kBucketTotal) && L.g.M <= kBucketModules &&
           (L.max_event ? L.max_event <= kBucketDigis : L.N / L.E <= kBucketDigis && L.E <= 32) &&
           (L.E + bucket_parts(L)) * kBucketCluster <= (uint64_t)L.sm_count;
}
// (With outputs in mapped host memory the copy keeps to 76 blocks of 1,216,
// and finish_kernel's one position a thread then takes longer than
// copy_kernel's four: latency of a host batch with the one / the other, 64
// events of 30,000 digis 289 / 273 us, in the mean over 32 and 64 events of
// 0.5 to 2M digis in all 3% more, below within 1%.  Where bucket_kernel starts
// the launch the pair is ahead by 2% up to kBucketTotal.)
static bool finish_fits(const Launch &L)
{
    const uint64_t most = !L.host_out ? kSmallDigis : bucket_fits(L) ? kBucketTotal : kSmallHost;
    return L.N <= most && L.cc.items <= kFinishItems && !L.debug;
}
static cudaError_t launch_bucket(const Launch &L, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((L.bucket_parts ? L.bucket_parts : L.E) * kBucketCluster);
    cfg.blockDim = dim3(kBucketThreads);
    cfg.dynamicSmemBytes = bucket_smem(L.g.M, L.bucket_parts != 0);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kBucketCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, L.bucket_parts ? bucket_kernel<true> : bucket_kernel<false>, L);
}

cudaError_t launch_reconstruct(const Launch &in, cudaStream_t stream, uint64_t *kernel_count, StageMarks *marks)
{
    NvtxRange range("hp_launch_reconstruct");
    Launch L = in;
    L.cc = cluster_plan(L);
    const bool finish = finish_fits(L), fused = finish && bucket_fits(L);
    L.bucket_parts = bucket_parts(L) ? L.E + (uint32_t)bucket_parts(L) : 0u;
    cudaError_t err = cudaSuccess;
    if (!fused)
        err = cudaMemsetAsync(L.ws.ctl, 0, L.ws.zero_bytes, stream);
    else if (L.E > 1) // (with one event the bucket kernel clears them)
        err = cudaMemsetAsync(L.ws.ctl, 0, (size_t)((unsigned char *)L.ws.count - (unsigned char *)L.ws.ctl), stream);
    if (err != cudaSuccess) return err;
    auto mark = [&](int i) {
        if (marks && err == cudaSuccess) err = cudaEventRecord(marks->ev[i], stream);
    };
    uint64_t nk = 0;
    auto ran = [&](int stage, Kernel k) {
        if (marks) marks->kernel[stage] = k;
        ++nk;
    };
    // persistent histogram and scatter over the same contiguous ranges
    const unsigned hist_grid = bucket_grid(L.N, L.sm_count), scat_grid = hist_grid; // the same ranges
    mark(0);
    if (fused) {
        mark(1);
        mark(2);
        if (err == cudaSuccess) err = launch_bucket(L, stream);
        ran(2, kBucket);
    }
    if (!fused && L.N > 0) {
        hist_kernel<<<hist_grid, kHistThreads, kHistCap * sizeof(uint32_t), stream>>>(L);
        ran(0, kHist);
    }
    if (!fused) {
        mark(1);
        if (err == cudaSuccess) err = launch_dependent(scan_kernel, L.E, 256, 0, stream, L);
        ran(1, kScan);
        mark(2);
    }
    if (!fused && L.N > 0) {
        const uint64_t steps = (L.N + kWideStep - 1) / kWideStep;
        // (the wide scatter wants a step a block, and steps over few events:
        // below, scatter_kernel's more and smaller blocks are faster)
        const bool wide = L.g.M > kSubKeys && steps >= (uint64_t)L.sm_count && L.N / L.E >= kWideStep;
        if (err == cudaSuccess) {
            if (wide)
                err = launch_dependent(scatter_wide_kernel, (unsigned)std::min<uint64_t>(steps, L.sm_count),
                                       kWideThreads, kWideSmem, stream, L);
            else
                err = launch_dependent(scatter_kernel, scat_grid, kHistThreads, kScatterSmem, stream, L);
        }
        ran(2, wide ? kScatterWide : kScatter);
    }
    mark(3);
    if (err == cudaSuccess) {
        const uint32_t b = L.tune.blocks_per_sm;
        if (L.tune.label_store == kStoreHash)
            err = launch_dependent(b >= 3 ? cc_hash_kernel<3> : b == 2 ? cc_hash_kernel<2> : cc_hash_kernel<1>,
                                   L.cc_grid, kCCThreads, L.cc.smem, stream, L);
        else if (b >= 3)
            err = launch_dependent(cc_kernel<kRunThreads3, kRunGroups3, 3>, L.cc_grid, kRunThreads3,
                                   L.cc.smem, stream, L);
        else if (b == 2 && L.cc.threads == (uint32_t)kRunThreads2n)
            err = launch_dependent(cc_kernel<kRunThreads2n, kRunGroups2n, 2>, L.cc_grid, kRunThreads2n,
                                   L.cc.smem, stream, L);
        else if (b == 2)
            err = launch_dependent(cc_kernel<kRunThreads2, kRunGroups2, 2>, L.cc_grid, kRunThreads2,
                                   L.cc.smem, stream, L);
        else
            err = launch_dependent(cc_kernel<kRunThreads1, kRunGroups1, 1>, L.cc_grid, kRunThreads1,
                                   L.cc.smem, stream, L);
    }
    ran(3, L.tune.label_store == kStoreHash ? kClusterHash : kCluster);
    mark(4);
    const uint64_t EM = (uint64_t)L.E * L.g.M;
    if (!finish) {
        if (err == cudaSuccess)
            err = launch_dependent(offsets_kernel, (unsigned)((EM + kOffItems - 1) / kOffItems), kOffThreads, 0, stream,
                                   L);
        ran(4, kOffsets);
    }
    mark(5);
    if (finish) { // a thread per expected cluster (one in eight digis; at most the copy's threads, looping)
        const uint64_t by_items = (L.N / 8 + kFinishThreads) / kFinishThreads;
        const uint64_t most = std::max<uint64_t>(1, (uint64_t)L.copy_grid * kCopyThreads / kFinishThreads);
        if (err == cudaSuccess)
            err = launch_dependent(finish_kernel, (unsigned)std::min(by_items, most), kFinishThreads,
                                   ((size_t)L.cc.items + 1) * 4, stream, L);
    } else { // a warp per output chunk (at most copy_grid blocks, looping), and a thread per event status and offset
        const uint64_t by_items = (L.N / kOutChunk + 1 + kCopyThreads / 32 - 1) / (kCopyThreads / 32);
        const uint64_t by_events = ((uint64_t)L.E + kCopyThreads) / kCopyThreads; // E + 1 offsets
        const uint64_t blocks =
            std::max<uint64_t>(1, std::max<uint64_t>(by_events, std::min<uint64_t>(by_items, (uint64_t)L.copy_grid)));
        if (err == cudaSuccess) err = launch_dependent(copy_kernel, (unsigned)blocks, kCopyThreads, 0, stream, L);
    }
    ran(5, finish ? kFinish : kCopy);
    mark(6);
    if (kernel_count) *kernel_count += nk;
    if (err != cudaSuccess) return err;
    return cudaGetLastError();
}

} // namespace hp
