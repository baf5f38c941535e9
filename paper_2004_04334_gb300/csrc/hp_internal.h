// Internal interface between the libhp host runtime and its sm_103a kernels.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stddef.h>
#include <stdint.h>

struct hp_ctx;

namespace hp {

// NVTX range around a host-side stage (visible to Nsight tools, e.g.
// `ncu --nvtx`; costs nothing measurable when no tool is attached).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// Error bits accumulated on the device (per event, and per launch).
constexpr uint32_t kErrBadDigi = 1u;
constexpr uint32_t kErrDup = 2u;
constexpr uint32_t kErrCapacity = 4u;
constexpr uint32_t kErrTimeout = 8u;
constexpr uint32_t kErrBadOffsets = 16u; // event offsets not 0 = o[0] <= o[1] <= ... <= o[E] = N (launch-wide)

// Tuning constants of the kernels.
constexpr int kChunk = 4096;         // digis per histogram / scatter block
constexpr int kHistThreads = 512;
constexpr int kHistCap = 4096;       // (event, module) bins a block can histogram in shared memory
constexpr int kCCThreads = 512;      // threads of a hash-store clustering block (the others: run_shape)
constexpr int kGroup = 16;           // most (event, module) items per work-queue ticket
constexpr int kWarpMax = 64;         // default of Tuning::warp_max
constexpr int kSmemSlots = 4096;     // runs of an item a block clusters in shared memory (default tile)
constexpr int kMaxTileSlots = 16384; // largest tile considered (one block per SM)

// Launch parameters of the clustering kernel, chosen per launch shape by the
// autotuner (defaults: the values above, two resident blocks per SM).
struct Tuning {
    uint32_t tile_slots = kSmemSlots; // runs in a block's shared memory; items with more use global scratch
    uint32_t blocks_per_sm = 2;       // 1 (four groups a block, largest tile), 2 (two or three groups) or 3 (one group)
    uint32_t ticket_max = kGroup;     // items per ticket before halving for small launches (<= kGroup)
    uint32_t warp_max = kWarpMax;     // 32 or 64: a twelfth of the packed tier's largest item (hash store: all of it)
    uint32_t label_store = 0;         // kStoreBitmap or kStoreHash: pixel lookup of the items above the packed tier
    uint32_t item_threads = kCCThreads; // threads clustering one item of the hash store: 128, 256 or 512
};

// Pixel lookup of the clustering items above the packed tier: module-sized
// bitmaps (a group of threads an item), or an open-addressing hash table keyed
// by linear pixel index, sized by the item's digi count (item_threads threads
// an item, several items of a block side by side).
constexpr uint32_t kStoreBitmap = 0;
constexpr uint32_t kStoreHash = 1;
// Digi index bits of the hash store's packed keys (items of at most 4096 digis).
constexpr uint32_t kHashIdxBits = 12;

// Digis a thread of the hash store holds in registers: fewer at three resident
// blocks per SM (40 registers).
__host__ __device__ constexpr int cc_digis_per_thread(int blocks_per_sm) { return blocks_per_sm >= 3 ? 5 : 8; }

// Largest item (digis) of the hash store: each of the block's
// kCCThreads / item_threads groups takes an equal 16-byte-aligned slice of
// the clustering kernel's dynamic shared memory (`smem` bytes) for 28 bytes
// a digi (accumulators, parent, two table slots) plus 256 row counters, and
// a slice of the block's 64-bit moment scratch (2 * tile_slots entries);
// each thread holds at most `per_thread` digis in registers.
__host__ __device__ inline uint32_t hash_capacity(size_t smem, uint32_t tile_slots, uint32_t item_threads,
                                                  uint32_t per_thread)
{
    const uint32_t groups = (uint32_t)kCCThreads / item_threads;
    const size_t slice = (smem / groups) & ~(size_t)15;
    size_t cap = slice > 1024 ? (slice - 1024) / 28 : 0;
    if (cap > tile_slots / groups) cap = tile_slots / groups;
    if (cap > (size_t)per_thread * item_threads) cap = (size_t)per_thread * item_threads;
    if (cap > (1u << kHashIdxBits)) cap = 1u << kHashIdxBits;
    return (uint32_t)cap;
}

// Whether a launch of N digis in EM items has items of 64 digis or more on
// average.
__host__ __device__ inline bool large_items(uint64_t N, uint64_t EM) { return N >= 64ull * EM; }

// Items per work-queue ticket of a launch of EM items on `grid` clustering
// groups: `gmax`, halved while a launch would have too few tickets per
// group.  Small items keep at least four a ticket, so that they share the
// packed tier's phases, and want two tickets a group; larger items go down to
// one a ticket and want four a group, so that a small launch's items spread
// over groups instead of queueing in one ticket.
__host__ __device__ inline uint32_t ticket_items(uint64_t EM, unsigned grid, uint32_t gmax, uint64_t N)
{
    const bool large = large_items(N, EM);
    const uint32_t least = large ? 1u : 4u;
    const uint64_t want = (large ? 4ull : 2ull) * grid;
    uint32_t g = gmax;
    while (g > least && (EM + g - 1) / g < want) g >>= 1;
    return g;
}

// Clusters parked between the clustering kernel and the ordered write, as
// structure-of-arrays indexed by bucket position: item i's k-th kept cluster
// (in id order) sits at boff[i] + k.
struct Staging {
    int32_t *id, *charge, *npix;
    float *x, *y;
    __device__ __forceinline__ void put(uint64_t at, int32_t id_, int32_t q, int32_t np_, float x_, float y_) const
    {
        id[at] = id_;
        charge[at] = q;
        npix[at] = np_;
        x[at] = x_;
        y[at] = y_;
    }
};

struct Geometry {
    uint32_t M, R, C;
    int32_t pixel_thr, cluster_thr;
    const int32_t *gain; // device [M]
    const int32_t *ped;  // device [M]
};

// The six per-cluster output columns.
struct ClusterCols {
    uint32_t *module;
    int32_t *id, *charge, *npix;
    float *x, *y;
};

struct Outputs {
    uint64_t capacity;
    uint32_t *module;
    int32_t *id, *charge, *npix;
    float *x, *y;
    uint64_t *cluster_offsets; // [E+1]
    int32_t *label;            // [N] or null
    int32_t *event_status;     // [E] written by copy_kernel
    // compact labels, instead of `label` (cc_kernel): each digi's cluster as
    // its rank among the kept clusters of its (event, module) item, 0xFFFF
    // below the pixel threshold, 0xFFFE in a cluster below the cluster
    // threshold; and (copy_kernel) each item's first cluster counted from its
    // event's first
    uint16_t *label16 = nullptr;    // [N] or null
    uint32_t *item_first = nullptr; // [E*M] (with label16)
    // Outputs in mapped host memory: positions below head_n go to these
    // device columns instead (16-byte aligned), which the launch then copies
    // to the host columns by DMA, so that the copy engine, not the SMs,
    // carries them over the host link; the positions from head_n on (the
    // launch cannot know the cluster count in advance) go straight to host.
    ClusterCols head{};
    uint32_t head_n = 0;
};

// Output positions a copy_kernel warp writes per step (four a lane).
constexpr uint32_t kOutChunk = 128;

// Scratch of one launch.  Before the first kernel hist_kernel the first
// `zero_bytes` bytes are zeroed (one memset): control words, per-event error
// bits, per-item counts and the chained-scan state.  Where bucket_kernel comes
// first the control words and error bits alone are, by a memset up to `count`
// or, for one event, by that kernel: it writes every count, and count2 and
// chain, which nothing reads then, hold what an earlier launch left.
struct Workspace {
    uint32_t *ctl;        // [16]: 0 item ticket, 1 launch error bits, 2 arena bump, 3 prefix frontier,
                          //       4 offsets chunk ticket, 5 large items and 7 their ticket,
                          //       6 clusters of the launch (offsets_kernel),
                          //       8-15 a bit per SM whose block came for large items (cc_kernel)
    uint32_t *event_err;  // [E]
    uint32_t *count;      // [E*M] digis of each item (reserved part, then the total: scan_kernel);
                          //       then each item's first output position (offsets_kernel)
    uint32_t *count2;     // [E*M] digis of histogram ranges with many keys (placed step by step)
    unsigned long long *chain; // [2 * n_chunks]: offsets_kernel chunk totals, then inclusive prefixes
    size_t zero_bytes;
    uint32_t *boff;       // [E*M] bucket start of each item
    uint32_t *blk_off;    // [bucket_grid * kHistCap] each histogram block's offset inside each key's bucket
    uint32_t *cursor;     // [E*M] scatter cursor of the step-by-step part; then each item's count of kept
                          //       clusters (cc_kernel)
    // [N] digi word and index within its event, item after item.  Pairs, so
    // that a digi that lands alone writes one sector instead of two: the
    // scatter of 29.4M digis over 1,856 modules an event 441 -> 281 us (171
    // since, sorted in wide steps), over 64 modules 170 -> 154 us (127 since).
    uint2 *bucket;
    Staging staging;      // [N] each array
    uint32_t *large;      // [E*M] items of more than cc.large_digis digis, ctl[5] of them (scan_kernel)
    uint32_t *chunk_item; // [N / kOutChunk + 2] item holding the first position of each output chunk
    unsigned long long *exact; // [cc_grid * 2 * run_exact_slots] 64-bit moments of heavy clusters
    unsigned char *big;   // scratch of items too large for shared memory
    uint64_t big_slots;   // slots per block (slab mode) or in total (arena mode)
    int big_arena;        // 1: bump-allocated arena, 0: one slab per block
};

// Sizes of the clustering kernel of one launch, worked out on the host.
struct ClusterPlan {
    uint32_t items, ticket_items, tickets; // (event, module) items, items a ticket, tickets
    uint32_t threads, workers;             // threads of a block; groups of all blocks
    uint32_t smem, slice;                  // dynamic shared memory of a block, and of each of its groups
    uint32_t runs, whole_runs;             // run records in a group's slice, and in the whole block's
    uint32_t exact_slots;                  // 64-bit moment slots of a block
    uint32_t pack_digis, pack_item;        // packed tier: digis of a pack, and of its largest item
    uint32_t large_digis;                  // items of more digis are clustered by a whole block,
    uint32_t own;                          // and every block clusters its own (an item a block), not those of a list
};

struct Launch {
    Geometry g;
    uint32_t E;
    uint64_t N;
    uint64_t max_event = 0;  // digis of the largest event, 0 where the host does not know
    bool host_out = false;   // the cluster columns are mapped host memory
    uint32_t bucket_parts = 0; // clusters of bucket_kernel where large events are split, else 0
    const uint64_t *offsets; // device [E+1]
    const uint32_t *words;   // device [N]
    const uint16_t *modules; // device [N]
    Outputs out;
    Workspace ws;
    int cc_grid;             // blocks of the clustering kernel
    ClusterPlan cc;          // sizes of the clustering kernel (cluster_plan)
    int copy_grid = 1216;    // most blocks of the output copy (8 an SM of a 152-SM GPU)
    int sm_count = 152;      // SMs of the device (grids of the persistent histogram and scatter)
    Tuning tune;
    uint32_t debug = 0;      // test hooks (kDebug*)
};

// Test hook: offsets_kernel never publishes chunk 0's cluster count,
// so the bounded waits of the ordered output expire and the launch reports
// HP_ETIMEOUT (the wait's limit is one second).
constexpr uint32_t kDebugWithholdTicket0 = 1u;

// Blocks of the persistent histogram and scatter kernels (the same
// contiguous digi ranges in both): two an SM, at least one kChunk a block.
__host__ __device__ inline unsigned bucket_grid(uint64_t N, int sm_count)
{
    const uint64_t chunks = (N + kChunk - 1) / kChunk;
    const uint64_t cap = 2ull * (uint64_t)(sm_count > 0 ? sm_count : 1);
    return (unsigned)(chunks < 1 ? 1 : (chunks < cap ? chunks : cap));
}

// Bytes of one global-tier slot: (Q, npix), two 64-bit and two 32-bit moments,
// parent, padded to 8-byte multiples so every slot range stays 8-byte aligned.
constexpr size_t kBigSlotBytes = 8 + 16 + 8 + 4 + 4;

// Dynamic shared memory of a clustering block of the hash label store: 20
// bytes a slot and three words per 32 pixels of a module.
__host__ __device__ inline size_t cc_smem_bytes(uint32_t R, uint32_t C, uint32_t tile_slots)
{
    const size_t nwords = ((size_t)R * C + 31) / 32;
    return (size_t)tile_slots * (8 + 8 + 4) + nwords * 4 * 3;
}

constexpr uint32_t kHashListBytes = (kCCThreads / 32) * 64 * 2; // of these, the run tier's warp lists

// The run tier of the clustering kernel.  A group of threads clusters an item
// in a slice of the block's shared memory: a survivor bitmap with rows of
// ceil(C / 32) words, the first run of every word (16 bits), and the records
// of the runs (20 bytes each), which lie over the bitmap of all digis.
constexpr size_t kRunBytes = 20;
constexpr size_t kBigRunBytes = 24; // a record in global scratch
__host__ __device__ inline uint32_t run_words(uint32_t R, uint32_t C) { return (R * ((C + 31) / 32) + 3) & ~3u; }
__host__ __device__ inline size_t run_fixed_bytes(uint32_t R, uint32_t C)
{
    const size_t nw = run_words(R, C);
    return nw * 4 + ((nw * 2 + 15) & ~(size_t)15);
}
// Runs that a slice of `bytes` holds.
__host__ __device__ inline uint32_t run_capacity(size_t bytes, uint32_t R, uint32_t C)
{
    const size_t fixed = run_fixed_bytes(R, C);
    return bytes > fixed ? (uint32_t)((bytes - fixed) / kRunBytes) : 0u;
}
// Dynamic shared memory of a block of `groups` groups whose whole holds
// tile_slots runs: at least slices of kSliceRuns runs where those leave two
// blocks an SM, of 256 where not, and of the bitmaps; at most what a lone
// block has besides its static memory (6,400 bytes for four groups), so that
// the largest tiles of small modules, which the hash store's limit allows,
// hold a few hundred runs less than they name.
constexpr size_t kSliceRuns = 1200, kSliceBytes = 112000, kWholeBytes = 225792;
__host__ __device__ inline size_t run_smem_bytes(uint32_t R, uint32_t C, uint32_t tile_slots, uint32_t groups)
{
    const size_t fixed = run_fixed_bytes(R, C), bits = (size_t)run_words(R, C) * 4;
    auto at_least = [&](size_t runs) { return fixed + (kRunBytes * runs > bits ? kRunBytes * runs : bits); };
    const size_t full = at_least(tile_slots), whole = full < kWholeBytes ? full : kWholeBytes;
    size_t parts = groups * ((at_least(kSliceRuns) + 15) & ~(size_t)15);
    if (parts > kSliceBytes) parts = groups * ((at_least(256) + 15) & ~(size_t)15);
    return whole > parts ? whole : parts;
}
// 64-bit moment slots of a block (its groups' slices hold no more runs together).
__host__ __device__ inline uint32_t run_exact_slots(uint32_t R, uint32_t C, uint32_t tile_slots, uint32_t groups)
{
    return run_capacity(run_smem_bytes(R, C, tile_slots, groups), R, C);
}
// Digis of a pack of the packed tier (two bitmap words, two counts and a run
// record each, beside kGroup items' tables of touched words) in a slice of
// `bytes` with moment scratch for `cap` runs; and the largest item it takes.
__host__ __device__ inline uint32_t pack_capacity(size_t bytes, uint32_t R, uint32_t cap)
{
    const size_t fixed = 6 * (size_t)kGroup * ((R + 1) / 2) + 64;
    const size_t fit = bytes > fixed ? (bytes - fixed) / (kRunBytes + 10) : 0;
    const uint32_t p = fit < 1023 ? (uint32_t)fit : 1023u;
    return p < cap ? p : cap;
}
// (384 or 768 digis: the best line for packs on sparse bitmaps; with hash
// tables in their place it lay at half of that)
__host__ __device__ inline uint32_t pack_max(uint32_t warp_max) { return 12 * warp_max; }

// Threads and groups of a clustering block for 1, 2 and 3 resident blocks per
// SM.  Two blocks an SM come as two groups of 256 threads each or as three of
// 160 (2n): an item is a chain of phases, and six groups an SM hide more of it
// than four, but a pack then holds 640 digis instead of 1,023 and a lone item
// has fewer threads.  Clustering kernel, 256 against 160 threads a group, in
// us: 16,384 items of 20 digis 39 / 31, of 80 73 / 55, of 150 88 / 91, of 300
// 164 / 161, of 500 238 / 258, of 781 347 / 270, of 1,000 357 / 317; 5,568
// items of 796 133 / 115; one event's 400 items of 796 20 / 24, its 64 of 469
// 14 / 20.
constexpr int kRunThreads1 = 1024, kRunGroups1 = 4;
constexpr int kRunThreads2 = 512, kRunGroups2 = 2;
constexpr int kRunThreads2n = 480, kRunGroups2n = 3;
constexpr int kRunThreads3 = 256, kRunGroups3 = 1;
struct RunShape {
    uint32_t threads, groups;
};
inline RunShape run_shape(const Tuning &t, uint64_t items, uint64_t N, int cc_grid)
{
    if (t.label_store == kStoreHash) return {(uint32_t)kCCThreads, 1u};
    if (t.blocks_per_sm >= 3) return {(uint32_t)kRunThreads3, (uint32_t)kRunGroups3};
    if (t.blocks_per_sm == 1) return {(uint32_t)kRunThreads1, (uint32_t)kRunGroups1};
    // three groups: more than one round of tickets, and items that leave most
    // of a pack, or of a group's registers, empty at 256 threads
    const unsigned workers = (unsigned)(cc_grid > 0 ? cc_grid : 1) * kRunGroups2;
    const bool rounds = items > (uint64_t)workers * ticket_items(items, workers, t.ticket_max, N);
    const bool size = N < 128 * items || N >= 640 * items;
    if (rounds && size) return {(uint32_t)kRunThreads2n, (uint32_t)kRunGroups2n};
    return {(uint32_t)kRunThreads2, (uint32_t)kRunGroups2};
}
// Digis above which an item is a whole block's: one and a half times the
// runs of a group's slice (0.6 runs a digi are usual; an item with more runs
// than the slice holds is finished in global scratch).
inline uint32_t large_digis(uint32_t R, uint32_t C, uint32_t tile_slots, RunShape sh)
{
    if (sh.groups == 1) return 0xFFFFFFFFu;
    return run_capacity((run_smem_bytes(R, C, tile_slots, sh.groups) / sh.groups) & ~(size_t)15, R, C) / 2 * 3;
}
// Lay out the workspace for (E, M, N) in `base` (nullptr: only compute size).
size_t carve_workspace(void *base, uint32_t E, uint32_t M, uint64_t N, uint32_t R, uint32_t C, int cc_grid,
                       const Tuning &tune, Workspace *ws, int sm_count);
// Configure kernel attributes once per device.  max_tile[b] receives the
// largest tile (slots) with which b clustering blocks stay resident per SM
// (0 if b blocks cannot be resident), for b = 1, 2 and 3 (at most
// kMaxTileSlots for one block, kSmemSlots otherwise); max_tile[0] unused.
// hash_tile[b] receives the same for the kernel's hash-store instance.
cudaError_t init_kernels(int device, uint32_t R, uint32_t C, uint32_t max_tile[4], uint32_t hash_tile[4]);
// The stages of one launch, in order, and the kernels that can run in them.
// Stage timers: ev[i] is recorded before stage i and ev[kNumStages] after the
// last one; kernel[i] is the kernel that ran in stage i (an index of
// kKernelNames), kNoKernel where none did (small launches fuse stages).
constexpr int kNumStages = 6;
enum Kernel : uint8_t {
    kHist, kScan, kScatter, kCluster, kOffsets, kCopy, kBucket, kScatterWide, kClusterHash, kFinish, kNumKernels,
    kNoKernel = 0xFF
};
extern const char *const kKernelNames[kNumKernels];
struct StageMarks {
    cudaEvent_t ev[kNumStages + 1];
    uint8_t kernel[kNumStages];
};
// Queue the whole reconstruction of one launch on `stream` (memset + kernels).
cudaError_t launch_reconstruct(const Launch &L, cudaStream_t stream, uint64_t *kernel_count,
                               StageMarks *marks = nullptr);

// One request of a serving batch: its inputs in (mapped) pinned host memory
// and where they go in the batch's device arrays.
struct GatherEntry {
    const uint32_t *words;
    const uint16_t *modules;
    uint64_t n;
    uint64_t off;
};
// Copy every request's inputs into the batch's device arrays (reads the host
// buffers over the C2C link; `table` must be device-accessible).
cudaError_t launch_gather(const GatherEntry *table, uint32_t n_requests, uint64_t max_n, uint32_t *words,
                          uint16_t *modules, cudaStream_t stream);

// Module placement for the clusters -> hits step, as the device holds it:
// per module three affine rows (r_i0, r_i1, o_i, 0), i = x, y, z, so that
// a hit is row_i . (u, v, 1).  Only the first two rotation columns matter
// because the local point has w = 0.
struct Placement {
    const float4 *rows;  // [3 * M]
    uint32_t M;
    float pitch_row, pitch_col;
    float half_rows, half_cols; // (rows - 1) / 2 and (cols - 1) / 2: the module centre in pixel units
};

// One hits launch: clusters in, hits out (all device-accessible pointers).
struct HitsLaunch {
    Placement p;
    uint32_t E;
    uint64_t capacity;                 // room in the cluster and hit arrays
    const uint64_t *cluster_offsets;   // [E + 1]
    const int32_t *event_status;       // [E] or null
    const uint32_t *module;            // [capacity]
    const float *x, *y;                // [capacity] centroids (pixel units)
    uint64_t *hit_offsets;             // [E + 1] or null: copy of cluster_offsets
    int32_t *hit_status;               // [E] or null: copy of event_status
    uint32_t *hit_module;              // [capacity] or null: copy of module
    float *hx, *hy, *hz;               // [capacity] global position
};
// Queue the hits kernel on `stream` (grid-stride; the cluster count is read
// on the device, so nothing waits for the clusters to exist).
cudaError_t launch_hits(const HitsLaunch &h, int max_blocks, cudaStream_t stream);

// Transfer on demand: copy a product's outputs (`src`, device memory) to
// `dst` (mapped pinned host memory): cluster offsets and event statuses
// always, and, if `clusters`, the cluster arrays of the clusters that exist
// (their count is read on the device, so only those bytes cross the link).
cudaError_t launch_copy_out(const Outputs &src, const Outputs &dst, uint32_t E, bool clusters, int max_blocks,
                            cudaStream_t stream);

// Launch parameters of a context (implemented by the runtime): geometry with
// device calibration pointers, device ordinal, clustering grid size and SM
// count; false if the context has failed.
bool context_launch_params(hp_ctx *ctx, Geometry *g, int *device, int *cc_grid, int *sm_count);
// Argument checks shared by the device-resident entry points: 0 (HP_OK) or
// the hp_status to return.
int check_device_call(hp_ctx *ctx, uint32_t n_events, uint64_t n_digis, const uint64_t *d_offsets,
                      const uint32_t *d_words, const uint16_t *d_module_ids, const struct hp_device_clusters *out);
// Mark the context failed after a CUDA error (every later call reports
// HP_ECUDA); returns HP_ECUDA.
int context_fail(hp_ctx *ctx);

} // namespace hp
