// C ABI of the CFGzip decode-step library: argument checks, partition tables, launch
// planning. The declarations and their contracts are in include/cfgzip.h.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "cfgzip.h"
#include "cfgzip_cluster.cuh"
#include "cfgzip_filtered.cuh"
#include "cfgzip_kernels.cuh"
#include "cfgzip_multi.cuh"
#include "class_sort.cuh"
#include "workspace.h"

using namespace cfgzip;

namespace {

struct Part {
    bool live = false;
    int32_t V = 0, K = 0, KW = 0, VW = 0;
    void* block = nullptr;  // one device allocation holding every table of the partition
    size_t block_bytes = 0;
    PartDev dev{};
    std::vector<int32_t> sizes;  // host copy of the class sizes (cfgzip_choose_mode)
};

constexpr size_t kSpareBytes = size_t(32) << 20;  // most memory of a released partition a context keeps for the next one
constexpr size_t kPartialSlots = size_t(1) << 18;  // 4 MB of (max, sum, pos) slots
constexpr int kTwoOctetItemsPerWarp = 3;           // bf16: two octets per lane from this many work items per warp on
constexpr int kDefaultRows = 16384;

}  // namespace

// Scratch of cfgzip_step_noalloc: lives in the library image, one copy on every GPU that loads it.
constexpr int kNoAllocMaxRows = 1024;
constexpr int kNoAllocMaxSplits = 64;
struct NoAllocScratch {
    Partial partials[kNoAllocMaxRows * kNoAllocMaxSplits];  // 1 MiB
    unsigned int tickets[kNoAllocMaxRows];                  // 4 KiB
};
static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

struct cfgzip_ctx {
    int device = 0;
    int sm_count = 0;
    int smem_optin = 0;
    std::vector<Part> parts;
    void* spare_block = nullptr;  // memory of the partition released last, for the next one loaded (given back with the context)
    size_t spare_bytes = 0;
    PartDev* d_parts = nullptr;
    Partial* d_partials = nullptr;
    unsigned int* d_tickets = nullptr;  // reserved_rows entries
    int32_t* d_status = nullptr;        // 4 counters, and 4 that nobody reads (see uncounted)
    bool uncounted = false;             // set around a launch that repeats what another launch of the same call counts
    int32_t* d_group_part = nullptr;
    int32_t* d_group_rows = nullptr;
    int32_t* d_n_groups = nullptr;
    int32_t* d_group_w = nullptr;       // row batches in front of every group
    int32_t* d_row_mode = nullptr;      // automatic mode: which rows the class-list kernel has finished
    int32_t reserved_rows = 0;
    int32_t max_groups = 0;
    // staging for cfgzip_decode_step_host
    void* st_logits = nullptr;
    size_t st_logits_bytes = 0;
    uint32_t* st_cm = nullptr;
    size_t st_cm_bytes = 0;
    uint32_t* st_vm = nullptr;
    size_t st_vm_bytes = 0;
    int32_t* st_small = nullptr;  // row_part, argmax, rep, lse, logp_argmax: 5 arrays of st_rows
    int32_t st_rows = 0;
    int32_t* st_small_host = nullptr;  // pinned mirror of the four result arrays: the kernels write them there, or one copy does
    // pinned host buffers: copies in, the step, copies out run side by side
    cudaStream_t st_in = nullptr, st_out = nullptr;
    cudaEvent_t st_ready = nullptr, st_masks = nullptr, st_expanded = nullptr;
    std::vector<cudaEvent_t> st_chunk_in, st_chunk_done;
    int64_t launches = 0;
    std::vector<std::pair<const void*, size_t>> smem_allowed;  // kernels whose shared-memory limit has been raised, and to what
    // row plan kept by cfgzip_plan_rows (valid until anything overwrites the plan buffers or the partitions change)
    bool plan_valid = false;
    bool plan_in_use = false;  // set for the duration of a call that passed CFGZIP_ROWS_AS_PLANNED
    const int32_t* plan_row_part = nullptr;
    int32_t plan_B = 0, plan_V = 0;
    // tuning
    int32_t ctas_per_sm = 4;
    int32_t token_warps = 0;
    int32_t row_warps = 0;
    int32_t pdl = 1;
    bool pdl_now = true;      // set per call: programmatic dependent launch only pays for short kernels
    int cluster_now = 1;      // set around a launch: blocks per thread-block cluster
    int cluster_limit[kClusterMost + 1] = {};  // clusters of that many blocks that run side by side, a block to an SM
    int prefetch_items = 4;   // work items per warp of the pipelined kernel asked into the L2 before its wait
    int prefetch_min_mbytes = 48;  // ... for steps of at least this many megabytes of logits
    bool prefetch_now = false;     // set per call beside pdl_now
    int rotate = 1;           // the chunk deal of the pipelined kernel starts at another warp slot for every row batch
    // cuTensorMapEncodeTiled, looked up through the runtime (no link against the driver library)
    CUresult (*encode_tiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill) = nullptr;
    int32_t pipeline = 1;     // bulk-copy pipelined dense kernel for aligned logits
    int32_t tensor_map = 1;   // tiled 2-D copies for row batches that are consecutive rows
    int32_t pipe_warps = 16;
    int32_t pipe_depth = 2;
    bool pipe_depth_set = false;  // the knob was set: no automatic third stage
    int32_t waves = 1;        // pipelined kernel: blocks launched per resident block slot
    int32_t spread = 1;       // pad the shared memory of one-block-per-SM launches so that blocks cannot share an SM
    int32_t stage_alias = 0;  // 1: always lay the class-mask staging area over the rings (default: only where it buys warps)
    int32_t lane_octets = 0;  // bf16 pipelined kernel: octets per lane and row (0 = automatic, 1, 2)
    int32_t auto_permille = -1;  // automatic mode: groups that allow under this many thousandths of their tokens go to the
                                 // class lists; -1 = by element type (measured break-even: f32 40, bf16 10)
    int64_t auto_min_bytes = -1;  // automatic mode on device-resident masks: steps of at least this many bytes of logits let the
                                  // GPU choose (one more launch); -1 = never (dense): the choice from host masks costs nothing
    int32_t fold = 0;         // pipelined kernel: the last block of a row group writes the rows' results (one launch per step)
    int32_t one_launch = 1;   // short batches: the whole step in one launch (k_step_cluster); off once a knob shapes the streaming kernel
    int32_t expire_test = 0;  // test hook: the pipelined kernel reports its first completed wait as run out
};

namespace {

struct DeviceGuard {
    int prev = -1;
    bool ok = true;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
        if (prev == dev) prev = -1;  // nothing to put back
        else if (cudaSetDevice(dev) != cudaSuccess) ok = false;
    }
    ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

inline int ceil_div(int64_t a, int64_t b) { return int((a + b - 1) / b); }

int32_t* status_of(const cfgzip_ctx* ctx) { return ctx->d_status + (ctx->uncounted ? 4 : 0); }

template <typename... KArgs, typename... Args>
int launch(cfgzip_ctx* ctx, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
           Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    if (ctx->pdl == 2 || (ctx->pdl && ctx->pdl_now)) {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    if (ctx->cluster_now > 1) {  // neighbouring blocks along x form a thread-block cluster
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = unsigned(ctx->cluster_now);
        attr[n_attr].val.clusterDim.y = 1;
        attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    cfg.attrs = attr;
    cfg.numAttrs = unsigned(n_attr);
    if (cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...) != cudaSuccess) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    ctx->launches += 1;
    return CFGZIP_OK;
}

// More than 48 KB of dynamic shared memory has to be allowed once per kernel; it is allowed up to the device's limit, so that
// the limit another context may have set is never smaller, and remembered: asking the runtime on every step costs half a
// microsecond of host time. large_clusters: the kernel also comes in clusters of more than eight blocks.
template <typename K>
int ensure_smem(cfgzip_ctx* ctx, K kernel, size_t bytes, bool large_clusters = false) {
    if (bytes <= 48 * 1024) return CFGZIP_OK;
    const void* fn = reinterpret_cast<const void*>(kernel);
    for (const auto& k : ctx->smem_allowed)
        if (k.first == fn) return bytes <= k.second ? CFGZIP_OK : CFGZIP_E_CUDA;
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, fn) != cudaSuccess) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    const size_t most = size_t(ctx->smem_optin) - std::min(size_t(ctx->smem_optin), attr.sharedSizeBytes);
    if (bytes > most || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(most)) != cudaSuccess ||
        (large_clusters && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    ctx->smem_allowed.emplace_back(fn, most);
    return CFGZIP_OK;
}

// How many clusters of every size the device holds at once, a block to an SM: the SMs come in groups that a cluster does not cross,
// so that 132 of 148 can be had four at a time and 120 eight at a time (15 clusters). Asked once per device and process: the
// fifteen questions took as long as the rest of creating a context.
void find_cluster_limits(cfgzip_ctx* ctx) {
    static std::mutex mutex;
    static std::map<int, std::array<int, kClusterMost + 1>> known;
    std::lock_guard<std::mutex> lock(mutex);
    const auto found = known.find(ctx->device);
    if (found != known.end()) {
        std::copy(found->second.begin(), found->second.end(), ctx->cluster_limit);
        return;
    }
    auto kern = k_step_cluster<kBF16, 1, false, false>;
    const size_t smem = size_t(ctx->smem_optin) / 2 + 1024;
    if (ensure_smem(ctx, kern, smem, true) != CFGZIP_OK) return;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    for (unsigned n = 2; n <= kClusterMost; ++n) {
        attr[0].val.clusterDim.x = n;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(n);
        if (cudaOccupancyMaxActiveClusters(&ctx->cluster_limit[n], kern, &cfg) != cudaSuccess) {
            cudaGetLastError();
            ctx->cluster_limit[n] = 0;
        }
    }
    std::copy(std::begin(ctx->cluster_limit), std::end(ctx->cluster_limit), known[ctx->device].begin());
}

int check_partition_host(const int32_t* c, int32_t V, const int32_t* r, int32_t K) {
    if (!c || !r || V <= 0 || K <= 0 || K > V) return CFGZIP_E_ARG;
    std::vector<uint8_t> seen(size_t(K), 0);
    for (int32_t i = 0; i < V; ++i) {
        if (c[i] < 0 || c[i] >= K) return CFGZIP_E_PARTITION;
        seen[size_t(c[i])] = 1;
    }
    for (int32_t k = 0; k < K; ++k) {
        if (!seen[size_t(k)]) return CFGZIP_E_PARTITION;
        if (r[k] < 0 || r[k] >= V || c[r[k]] != k) return CFGZIP_E_PARTITION;
    }
    return CFGZIP_OK;
}

void build_class_lists_host(const int32_t* c, int32_t V, int32_t K, int32_t* off, int32_t* tok) {
    std::fill(off, off + K + 1, 0);
    for (int32_t i = 0; i < V; ++i) off[c[i] + 1] += 1;
    for (int32_t k = 0; k < K; ++k) off[k + 1] += off[k];
    std::vector<int32_t> cursor(off, off + K);
    for (int32_t i = 0; i < V; ++i) tok[cursor[size_t(c[i])]++] = i;  // ascending ids inside a class
}

// Everything a per-step call needs to know about the partitions it may touch.
struct PartSet {
    int32_t V = 0, VW = 0, maxK = 0, maxKW = 0, n_live_same_v = 0;
    bool all_c16 = true;
    bool all_kw_mult4 = true;
};

int resolve_parts(cfgzip_ctx* ctx, cfgzip_part_id part0, bool mixed, PartSet* ps) {
    if (part0 < 0 || size_t(part0) >= ctx->parts.size() || !ctx->parts[size_t(part0)].live) return CFGZIP_E_RANGE;
    const Part& p0 = ctx->parts[size_t(part0)];
    ps->V = p0.V;
    ps->VW = p0.VW;
    if (!mixed) {
        ps->maxK = p0.K;
        ps->maxKW = p0.KW;
        ps->n_live_same_v = 1;
        ps->all_c16 = p0.dev.c16 != nullptr;
        ps->all_kw_mult4 = (p0.KW % 4) == 0;
        return CFGZIP_OK;
    }
    for (const Part& p : ctx->parts) {
        if (!p.live || p.V != p0.V) continue;
        ps->maxK = std::max(ps->maxK, p.K);
        ps->maxKW = std::max(ps->maxKW, p.KW);
        ps->n_live_same_v += 1;
        ps->all_c16 = ps->all_c16 && p.dev.c16 != nullptr;
        ps->all_kw_mult4 = ps->all_kw_mult4 && (p.KW % 4) == 0;
    }
    return CFGZIP_OK;
}

bool aligned32(const void* p, int64_t row_stride_elems, int elem_size) {
    return (reinterpret_cast<uintptr_t>(p) & 31u) == 0 && ((row_stride_elems * elem_size) & 31) == 0;
}

// (rows of a buffer that does not even start on an element are left to the element-wise kernels)
bool aligned_elems(const void* p, int elem_size) { return (reinterpret_cast<uintptr_t>(p) & uintptr_t(elem_size - 1)) == 0; }

bool aligned16(const void* p, int64_t row_stride_elems, int elem_size) {
    return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && ((row_stride_elems * elem_size) & 15) == 0;
}

size_t dense_smem_bytes(int table_words, int n_warps, int stage_stride) {
    (void)n_warps;
    return size_t(table_words) * 4 + kGroupRows * 4 + size_t(stage_stride) * kGroupRows * 4;
}

// Launch shape of the dense kernels.
struct DensePlan {
    int S = 1, per_split = 0, WT = 4, threads = 128, table_words = 0, stage_stride = 0;
    int depth = 0;       // > 0: pipelined kernel with this many stages per warp
    int cm_bulk = 0;     // pipelined kernel: class masks staged by bulk copies
    int stage_alias = 0; // pipelined kernel: staging area over the start of the rings
    int hold_warps = 0;
    int ctas_per_sm = 1; // blocks per SM the launch was sized for
    int opl = 1;         // pipelined kernel: octets per lane and row (2: bf16 chunks of 512 tokens)
    bool shifted = false;  // pipelined kernel: rows that start anywhere
    int chunk_octets = 32; // pipelined kernel: vectors per row and work item
    int fold = 0;        // pipelined kernel: results written by the last block of each group (no finalize launch)
    int fold_off = 0;    // fold: offset of the block's shared (row, warp) states, 0 = warps publish to the scratch directly
    int slots = 0;       // states per row in the global scratch
    int blocks = 0;      // > 0: pipelined kernel, mixed batch: S_even blocks to a group where the groups are the fewest they can be,
                         // else the blocks are shared out by the groups' sizes, at most S to a group
    int S_even = 0;
    size_t smem = 0;
    int n_groups_ub = 1;
    bool use_plan_kernel = false;
    bool ok = false;  // false: the dense kernels cannot run this call (generic path instead)
};

// alias: the class-mask staging area shares the space of the rings (it is dead once the table is built)
size_t pipe_smem_bytes(int table_words, int n_warps, int depth, int stage_bytes, int stage_stride, bool alias = false) {
    const size_t rings = size_t(n_warps) * depth * stage_bytes, staging = size_t(stage_stride) * kGroupRows * 4;
    return size_t(table_words) * 4 + kGroupRows * 4 + ((size_t(n_warps) * depth * 12 + 127) & ~size_t(127)) +
           (alias ? std::max(rings, staging) : rings + staging);
}

// Words between the rows of the class masks' staging area where these are not copied or read directly.
int slice_stride(const PartSet& ps) { return std::min(ps.maxKW, kMaskSlice) | 1; }
// How a call's class masks can be fetched (kMasks..).
int masks_kind(const PartSet& ps, const uint32_t* class_mask, int64_t stride, bool mixed, bool block) {
    if (reinterpret_cast<uintptr_t>(class_mask) & 15u) return kMasksStaged;
    if ((stride & 3) == 0) return ps.all_kw_mult4 ? kMasksRows : kMasksStaged;
    return block && !mixed && stride <= ps.maxKW + 64 ? kMasksBlock : kMasksStaged;
}

// Launch shape of the register-based dense kernel. units: octets; unit_chunk: units one warp covers per iteration.
// narrow: also where the class table leaves no room for a whole slice of the masks (some 53400 to 57500 classes off the 16-byte grid), by
// slices as wide as there is room, or word by word. The per-row kernel is as fast there (64 bf16 rows of 60032 in 53000 classes 167 us by whole
// slices, 137), but takes one mask per row.
DensePlan plan_dense(cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool mixed, int units, int unit_chunk, int masks, bool narrow = false) {
    DensePlan d;
    d.table_words = (ps.maxKW + 1) * 32;
    d.use_plan_kernel = mixed;
    d.n_groups_ub = mixed ? ceil_div(B, kGroupRows) + ps.n_live_same_v : ceil_div(B, kGroupRows);
    if (!ps.all_c16) return d;
    const size_t cap = size_t(ctx->smem_optin) - 2048;
    narrow = narrow && !masks && dense_smem_bytes(d.table_words, 8, slice_stride(ps)) > cap;
    const size_t least = dense_smem_bytes(d.table_words, 8, masks || narrow ? 0 : slice_stride(ps));
    if (least > cap) return d;
    if (mixed && (B > ctx->reserved_rows || d.n_groups_ub > ctx->max_groups)) return d;
    const int ctas_per_sm = ctx->ctas_per_sm;
    // the class masks through shared memory, all at once while that keeps a block under 64 KB
    d.cm_bulk = masks;
    if (narrow) {
        const int room = int((cap - least) / (kGroupRows * 4));
        d.stage_stride = room > 16 ? (room - 1) | 1 : 0;
    }
    if (!masks && !narrow) d.stage_stride = dense_smem_bytes(d.table_words, 8, ps.maxKW | 1) <= 64 * 1024 ? ps.maxKW | 1 : slice_stride(ps);
    d.ctas_per_sm = ctas_per_sm;
    const int target = ctx->sm_count * ctas_per_sm;
    const int n_chunks = ceil_div(units, unit_chunk);
    const int s0 = std::max(1, target / d.n_groups_ub);
    int cps = ceil_div(n_chunks, s0);  // chunks per block
    int WR = ctx->row_warps ? ctx->row_warps : (cps <= 2 ? 4 : 1);
    if (WR != 1 && WR != 2 && WR != 4) WR = 1;
    d.WT = ctx->token_warps ? ctx->token_warps : (WR == 4 ? std::min(cps, 2) : (WR == 2 ? 2 : 4));
    d.WT = std::max(1, std::min(d.WT, 8 / WR));
    d.threads = d.WT * WR * 32;
    for (;;) {
        d.S = ceil_div(n_chunks, cps);
        if (size_t(d.n_groups_ub) * kGroupRows * (size_t(d.S) * d.WT + 1) <= kPartialSlots) break;
        if (cps >= n_chunks) return d;
        cps *= 2;
    }
    d.per_split = cps * unit_chunk;
    d.slots = d.S * d.WT + 1;
    d.smem = dense_smem_bytes(d.table_words, d.threads / 32, d.stage_stride);
    d.ok = true;
    return d;
}

// Launch shape of the expansion alone: two blocks to an SM, so that a class table serves many tokens.
DensePlan plan_expand(cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool mixed, int masks) {
    DensePlan d;
    d.table_words = (ps.maxKW + 1) * 32;
    d.use_plan_kernel = mixed;
    d.n_groups_ub = mixed ? ceil_div(B, kGroupRows) + ps.n_live_same_v : ceil_div(B, kGroupRows);
    if (!ps.all_c16 || dense_smem_bytes(d.table_words, 0, masks ? 0 : slice_stride(ps)) > size_t(ctx->smem_optin) - 2048) return d;
    if (mixed && (B > ctx->reserved_rows || d.n_groups_ub > ctx->max_groups)) return d;
    d.cm_bulk = masks;
    if (!masks) d.stage_stride = dense_smem_bytes(d.table_words, 0, ps.maxKW | 1) <= 100 * 1024 ? ps.maxKW | 1 : slice_stride(ps);
    d.smem = dense_smem_bytes(d.table_words, 0, d.stage_stride);
    const int n_units = ceil_div(ps.VW, 16), per_sm = d.smem > size_t(ctx->smem_optin) / 2 - 2048 ? 1 : 2;
    d.per_split = ceil_div(n_units, std::max(1, per_sm * ctx->sm_count / d.n_groups_ub));
    d.S = ceil_div(n_units, d.per_split);
    d.threads = kExpandThreads;
    d.ok = true;
    return d;
}

// Launch shape of the pipelined fused kernel. A block takes per_split octets (any number, not only
// whole 32-octet chunks) of one row group, so that the blocks of a step fill the SMs evenly.
DensePlan plan_pipe_opl(cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool mixed, int elem_size, int masks, int64_t cm_stride, int opl,
                        bool shifted) {
    DensePlan d;
    d.opl = opl;
    d.shifted = shifted;  // rows off the 16-byte grid: each row's vectors start at its own first boundary
    d.chunk_octets = shifted ? PipeChunk<1, kSrcShifted>::kOctets : 32 * opl;
    d.table_words = (ps.maxKW + 1) * 32;
    d.use_plan_kernel = mixed;
    d.n_groups_ub = mixed ? ceil_div(B, kGroupRows) + ps.n_live_same_v : ceil_div(B, kGroupRows);
    if (!ps.all_c16 || !ctx->pipeline) return d;
    if (mixed && (B > ctx->reserved_rows || d.n_groups_ub > ctx->max_groups)) return d;
    const int chunk_octets = d.chunk_octets;
    const int stage_bytes = 32 * opl * (8 * 8 * elem_size + 16);
    const size_t cap = size_t(ctx->smem_optin) - 2048;  // room for the kernel's static shared memory
    // two octets per lane: the variant is compiled for at most 12 warps (its stages are twice as large and it needs
    // more registers per thread)
    int n_warps = opl == 2 ? std::min(ctx->pipe_warps, 12) : ctx->pipe_warps, depth = ctx->pipe_depth;
    const int max_warps = n_warps;
    d.cm_bulk = masks;
    int stride = masks == kMasksRows ? ps.maxKW + (ps.maxKW % 8 == 0 ? 4 : 8) : masks == kMasksBlock ? int(cm_stride) : slice_stride(ps);
    auto fits = [&](int warps, int stages, bool over_rings) {
        return pipe_smem_bytes(d.table_words, warps, stages, stage_bytes, stride, over_rings) <= cap;
    };
    bool alias = ctx->stage_alias != 0;
    bool settled = false;
    // Long steps (twenty or more work items per warp) gain from a third stage where sharing the staging area makes
    // room for it (measured at V = 128256, bf16: B = 1024 -0.7 %, B = 2048 -1.4 %; B = 256 .. 512 lose 1 to 2 % to
    // the late start of the first warps).
    if (!ctx->pipe_depth_set && depth < 3 && fits(n_warps, 3, true)) {
        const int64_t blocks = int64_t(ctx->sm_count) * ctx->waves;
        const int64_t items = int64_t(ceil_div(B, kGroupRows)) * ceil_div(ps.V >> 3, chunk_octets) *
                              ceil_div(std::min<int>(B, kGroupRows), kBatchRows);
        if (items >= 20 * blocks * n_warps) {
            depth = 3;
            alias = true;
            settled = true;
        }
    }
    // Otherwise: the most warps (down to 8: a staged class-mask fetch is worth giving up warps for when the class
    // table is large) for which the staging area of the class masks fits, beside the rings of all warps or, where
    // it does not, laid over the first rings (their warps then start copying after the table is built).
    if (!settled) {
        const int step_down = opl == 2 ? 1 : 4;
        int w = n_warps;
        for (; w >= std::min(8, max_warps); w -= step_down) {
            if (ctx->stage_alias == 0 && fits(w, 2, false)) { alias = false; break; }
            if (fits(w, 2, true)) { alias = true; break; }
        }
        if (w >= std::min(8, max_warps)) {
            n_warps = w;
        } else {  // the class masks word by word, a slice at a time
            n_warps = max_warps;
            stride = slice_stride(ps);
            d.cm_bulk = kMasksStaged;
            alias = true;  // (always over the rings: a slice beside them cost tables of 44200 to 48300 classes the kernel, 64 bf16 rows
                           // of 60032 in 48000 classes 151 us instead of 79)
        }
    }
    while (depth > 2 && pipe_smem_bytes(d.table_words, n_warps, depth, stage_bytes, stride, alias) > cap) --depth;
    while (n_warps > 4 && pipe_smem_bytes(d.table_words, n_warps, depth, stage_bytes, stride, alias) > cap)
        n_warps -= opl == 2 ? 1 : 2;
    size_t smem = pipe_smem_bytes(d.table_words, n_warps, depth, stage_bytes, stride, alias);
    if (smem > cap) return d;
    d.depth = depth;
    d.stage_stride = stride;
    const int fit = std::max(1, int((cap + 1024) / (smem + 1024)));
    d.ctas_per_sm = opl == 2 || shifted ? 1 : std::min(ctx->ctas_per_sm, fit);
    const int target = ctx->sm_count * d.ctas_per_sm * ctx->waves;
    const int n_oct = 4 * ps.VW;
    // blocks of groups that turn out not to exist leave at once, so size the split for the fewest
    // groups the batch can have
    const int s0 = std::max(1, target / ceil_div(B, kGroupRows));
    int per = std::max(chunk_octets, ceil_div(n_oct, s0));
    // Warps go side by side along the vocabulary first (long contiguous runs per row are kind to
    // DRAM); only when a block has fewer chunks than warps do warps split the row batches.
    const int chunks = ceil_div(per, chunk_octets);
    const int batch_rows = std::min<int>(B, kGroupRows), groups = ceil_div(B, kGroupRows);
    int WR = ctx->row_warps;
    if (!WR) {
        WR = 1;
        while (WR < 4 && chunks * WR * 2 <= n_warps) WR <<= 1;
    }
    while (WR > 1 && (WR - 1) * kBatchRows >= batch_rows) WR >>= 1;
    if ((WR != 1 && WR != 2 && WR != 4)) WR = 1;
    d.WT = ctx->token_warps ? ctx->token_warps : n_warps / WR;
    d.WT = std::max(1, std::min(std::min(d.WT, max_warps / WR), chunks));
    // Where a warp has a handful of work items, what counts is how many the busiest has, how many warps share the schedulers, and
    // how often a warp opens and publishes a row batch. Time of an item with w warps in the block 0.6 + 0.118 w us (w counted in
    // fours, a scheduler each), of a row batch 0.48, 0.3 where a row has more states than a warp folds: fitted to 128 bf16 rows of
    // 128256, it orders the shapes of 18 other batches as measured or within 2 %. Rows by the vocabulary / as chosen, us: bf16 of
    // 128256 96 rows 16.3 / 14.9, 128 19.0 / 17.2, 256 28.6 / 27.7, 100 rows of 100003 21.7 / 17.9, 80 of 256000 26.3 / 23.6; f32 of 128256
    // 34 rows 15.3 / 13.4, 150 33.1 / 32.2. Longer steps are bound by DRAM, which likes the long runs better (f32 of 128256, 300 rows 57.0,
    // split 59.2; 200 rows of 64064 20.8, split 21.5), and a mixed batch may have few row batches in a group.
    if (!ctx->row_warps && !ctx->token_warps && !mixed && opl == 1 && groups <= (elem_size == 2 ? 8 : 5)) {
        const int n_chunks = std::max(1, ceil_div(ps.V >> 3, chunk_octets)), S = ceil_div(n_oct, per), batches = ceil_div(batch_rows, kBatchRows);
        double least = 0.;
        for (int wr = 1; wr <= 4 && (wr == 1 || (wr - 1) * kBatchRows < batch_rows); wr <<= 1)
            for (int wt = std::min(n_warps / wr, chunks); wt >= 1; --wt) {
                const int turns = ceil_div(batches, wr), items = ceil_div(int64_t(turns) * n_chunks, int64_t(S) * wt);
                const double cost = items * (0.6 + 0.118 * (4 * ceil_div(wt * wr, 4))) + 0.48 * turns + (S * wt + 1 > kFinalizeWarpStates ? 0.3 : 0.);
                if (least > 0. && cost >= least) continue;
                least = cost;
                d.WT = wt;
                WR = wr;
            }
    }
    d.threads = d.WT * WR * 32;
    // The groups of a mixed batch may hold 32 rows or one, and only the GPU knows how many there are: where there are blocks
    // enough it gives every group the same number if the groups are the fewest the batch can have (336 bf16 rows of 128256 in two
    // partitions: 41 us; shares by size 44), else its share by size, one wave of blocks that all have about as much to do
    // (256 rows in eight partitions, V = 256000: 63 us; the same number for every group, in two waves, 78).
    if (mixed && target >= 3 * d.n_groups_ub) {
        const int batches = ceil_div(B, kBatchRows), most = std::min(batches, kGroupRows / kBatchRows);
        const int S = std::min(target, ceil_div(int64_t(target) * most, batches) + 2);
        if (size_t(d.n_groups_ub) * kGroupRows * (size_t(S) * d.WT + 2) <= kPartialSlots) {
            d.blocks = target;
            d.S = S;
            d.S_even = ceil_div(n_oct, per);
        }
    }
    while (!d.blocks) {
        d.S = ceil_div(n_oct, per);
        if (size_t(d.n_groups_ub) * kGroupRows * (size_t(d.S) * d.WT + 2) <= kPartialSlots) break;
        if (per >= n_oct) return d;
        per *= 2;
    }
    d.per_split = per;
    d.stage_alias = alias ? 1 : 0;
    d.hold_warps = alias ? std::min(d.threads / 32, ceil_div(int64_t(d.stage_stride) * kGroupRows * 4, int64_t(d.depth) * stage_bytes)) : 0;
    d.smem = pipe_smem_bytes(d.table_words, d.threads / 32, d.depth, stage_bytes, d.stage_stride, alias);
    d.slots = d.S * d.WT + 1;
    // One launch per step: the last block of a group folds the group's states. Where shared memory has room the
    // warps of a block first merge their states there (one state per row and block reaches the scratch); otherwise
    // the warps publish directly, which is only taken while a row has few states.
    if (ctx->fold) {  // 1: fold in the kernel; 2: only merge the states of a block's warps before they are published
        const size_t block_states = size_t(kGroupRows) * (d.WT + 1) * sizeof(Partial);
        if (d.smem + block_states <= cap) {
            d.fold = ctx->fold == 1;
            d.fold_off = int(d.smem);
            d.smem += block_states;
            d.slots = d.S;
        } else if (d.slots <= 256) {
            d.fold = ctx->fold == 1;
        }
    }
    // A launch sized for one block per SM asks for more than half of an SM's shared memory even when its few warps
    // need less, so that two of its blocks never share an SM while another SM stays empty (measured at B = 8 .. 24:
    // 10.2 -> 7.7 us, 10.1 -> 8.8 us, 12.4 -> 10.6 us).
    if (d.ctas_per_sm == 1 && ctx->spread) d.smem = std::max(d.smem, cap / 2 + 1024);
    d.ok = true;
    return d;
}

// Launch shape of the pipelined fused kernel. bf16 rows may be streamed with one octet (16 bytes) or two octets
// (32 bytes) per lane and row; two octets halve the per-row bookkeeping but double a work item, so they are taken
// only when every warp of the launch still gets several items.
DensePlan plan_pipe(cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool mixed, int elem_size, int masks, int64_t cm_stride,
                    bool shifted = false) {
    const DensePlan one = plan_pipe_opl(ctx, ps, B, mixed, elem_size, masks, cm_stride, 1, shifted);
    if (elem_size != 2 || ctx->lane_octets == 1 || shifted) return one;
    const DensePlan two = plan_pipe_opl(ctx, ps, B, mixed, elem_size, masks, cm_stride, 2, false);
    if (!two.ok) return one;
    if (!one.ok || ctx->lane_octets == 2) return two;
    if (ctx->lane_octets == 0) return one;
    const int64_t items = int64_t(ceil_div(B, kGroupRows)) * ceil_div(ps.V >> 3, 64) *
                          ceil_div(std::min<int>(B, kGroupRows), kBatchRows);
    const int64_t warps = int64_t(ctx->sm_count) * ctx->waves * (two.threads / 32);
    return items >= kTwoOctetItemsPerWarp * warps ? two : one;
}

// Whether rows that allow few tokens go through k_step_few (`d`, `per_sm`: its launch shape) or k_step_sparse, the class lists.
// k_step_few builds a class table per block, 32 rows at a time, and streams all rows at once; the class lists have a block or more
// per row, most efficient from the row count on at which a block takes a whole row and as long as these fit the device in one wave.
// Measured, us, class lists / k_step_few, bf16, one to five classes allowed:
//   under 64 rows    32 of 128256: K = 512 20 / 11, 2000 14.9 / 12.4, 4000 12.8 / 14.2; 48 f32 rows of 256000, K = 2000 20 / 24: by
//                    classes and row length. These batches take one launch where it fits them (launch_fused), the others the class lists,
//                    one launch instead of two
//   class table      128 of 128256: K = 4000 25 / 20, 6000 25 / 21, 8192 23.2 / 24.3, 16000 29 / 24; 512 of 256000: K = 8200 79 / 70, 16000
//                    108 / 71; f32: 250 of 200064 K = 6001 76 / 54, 100 of 64064 K = 8000 26 / 19; 70 of 90048 K = 11000 19.7 / 20.4 (while the table
//                    took its masks lane by lane from some 4900 classes on, the lists were better there)
//   short rows       450 of 20032 12 / 14, 450 of 32064 15 / 19, 410 of 32064 15.1 / 14.8, 512 of 64064 24 / 27, 800 40 / 39
//   mixed batches    groups of few rows build tables for little: 64 rows of 128256 in eight partitions, K = 512 19 / 16, 3000
//                    28 / 17, 4000 13 / 18; 300 rows of 20032 in two of 512 11.2 / 11.7, in eight 11 / 15
bool few_pays(const cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool mixed, int elem_size, const DensePlan& d) {
    const int wave = ctx->sm_count * ctx->ctas_per_sm;  // rows from half of this on have one block each in the other kernel
    const int64_t row_kb = int64_t(ps.V) * elem_size >> 10;
    if (B < 64) return false;
    if (mixed) return ps.maxK <= 3072 && !(row_kb < 96 && d.n_groups_ub > 16);
    return !(row_kb < 96 && B > wave / 2) && !(row_kb < 160 && B > 3 * wave / 4 && B <= wave);
}

// Launch shape of the kernel for rows that allow few tokens: three blocks per SM; warps go side by side along the vocabulary
// as long as a block has enough chunks for them, else they split the row batches.
DensePlan plan_few(cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool mixed, int elem_size, int masks) {
    DensePlan d;
    d.table_words = (ps.maxKW + 1) * 32;
    d.use_plan_kernel = mixed;
    d.n_groups_ub = mixed ? ceil_div(B, kGroupRows) + ps.n_live_same_v : ceil_div(B, kGroupRows);
    if (!ps.all_c16 || (mixed && (B > ctx->reserved_rows || d.n_groups_ub > ctx->max_groups))) return d;
    const size_t fixed = dense_smem_bytes(d.table_words, kFewWarps, 0) + kFewWarps * sizeof(FewWarp);
    d.cm_bulk = masks;
    if (!masks) d.stage_stride = fixed + size_t(ps.maxKW | 1) * kGroupRows * 4 <= 72 * 1024 ? ps.maxKW | 1 : slice_stride(ps);  // (three blocks per SM still fit)
    d.smem = fixed + size_t(d.stage_stride) * kGroupRows * 4;
    if (d.smem > size_t(ctx->smem_optin) - 2048) return d;
    const int n_chunks = std::max(1, ceil_div(ps.V / (32 / elem_size), 32));
    const int row_batches = ceil_div(std::min<int>(B, kGroupRows), kBatchRows);
    const int per_sm = std::max(1, std::min(3, int(size_t(ctx->smem_optin) / (d.smem + 1024))));
    d.S = std::min(std::max(1, per_sm * ctx->sm_count / ceil_div(B, kGroupRows)), n_chunks);
    while (d.S > 1 && size_t(d.n_groups_ub) * kGroupRows * (size_t(d.S) * kFewWarps + 1) > kPartialSlots) d.S = (d.S + 1) / 2;
    int WR = 1;
    while (WR < 4 && WR < row_batches && ceil_div(n_chunks, d.S) * WR * 2 <= kFewWarps) WR <<= 1;
    d.WT = kFewWarps / WR;
    d.threads = kFewThreads;
    d.slots = d.S * d.WT + 1;
    d.ok = size_t(d.n_groups_ub) * kGroupRows * d.slots <= kPartialSlots && few_pays(ctx, ps, B, mixed, elem_size, d);
    return d;
}

// Whether a call with several masks per logits row goes through k_step_multi or, every (row, mask) for itself, k_step_dense.
// k_step_multi takes the logits rows of a batch of eight (row, mask) pairs one after the other, so with two or three masks a row
// its chain is the longer one and its sharing small; k_step_dense builds a class table for every few tokens, which costs with K, and
// takes each exponential once per mask, which costs once the device is full. `items`: (256 tokens, batch) pairs. Measured, us,
// k_step_dense / k_step_multi, bf16 of 128256, rows x masks:
//   K = 256    4x2 9.0 / 11.3, 16x2 10.4 / 11.8, 32x2 16 / 15; 4x4 9.3 / 9.9, 16x4 16 / 13; 1x16 9.3 / 8.7, 8x16 22 / 14
//   K = 2048   4x2 11.3 / 12.1, 16x2 12.6 / 12.7, 32x2 17.5 / 16; 3x3 11.6 / 9.3, 12x3 16 / 15; 2x4 11.0 / 10.0, 8x16 24 / 15
//   K = 4000   4x2 14.5 / 13.5, 16x2 15.9 / 13.8;  K = 8000  1x2 25 / 13, 4x2 26 / 15
// f32 of 128256, K = 2048: 4x2 14.8 / 12.6;  f32 of 50048, K = 2048: 4x2 10.1 / 10.8, 24x2 11.7 / 12.6
bool multi_pays(const PartSet& ps, int32_t B, int masks_per_row, int elem_size, int64_t items) {
    const int logits_rows = std::min<int>(B, ceil_div(kBatchRows, masks_per_row));  // of a batch
    if (logits_rows == 1 || ps.maxK > 3072 || int64_t(ps.V) * elem_size >= 400 * 1024) return true;
    if (ps.maxK < 1024) return items >= (logits_rows == 2 ? 1500 : 2200);
    return logits_rows == 2 || items >= (logits_rows == 3 ? 1000 : 2200);
}

// Launch shape of the kernel for several masks per logits row: two blocks per SM of eight warps, four where the class table is
// large, where eight would get a third of an item each or less (4 rows x 4 masks of 50048 bf16, K = 256: 8.7 against 9.4 us; 4 x 4
// of 128256, K = 2048: 12.6 with four, 9.3 with eight), and on short calls where only four leave room to stage the class masks
// (K = 8000, 4 x 2: 14.7 against 18); warps split the row batches of a group first, so that a block builds its table for as many
// chunks as possible.
DensePlan plan_multi(cfgzip_ctx* ctx, const PartSet& ps, int32_t B, int masks_per_row, int elem_size, int masks,
                      int64_t cm_stride) {
    const int32_t rows = B * masks_per_row;
    DensePlan d;
    d.table_words = (ps.maxKW + 1) * 32;
    d.n_groups_ub = ceil_div(rows, kGroupRows);
    if (!ps.all_c16) return d;
    // (the class masks directly, all at once by way of shared memory where they are short, or a slice at a time)
    const size_t cap = size_t(ctx->smem_optin) - 2048;
    d.cm_bulk = masks == kMasksBlock && cm_stride > 2 * kMaskSlice ? kMasksStaged : masks;
    if (d.cm_bulk == kMasksBlock) d.stage_stride = int(cm_stride);
    if (d.cm_bulk == kMasksStaged) d.stage_stride = ps.maxKW <= 2 * kMaskSlice ? ps.maxKW | 1 : slice_stride(ps);
    int n_warps = kMultiWarps;
    auto bytes = [&](int warps) { return dense_smem_bytes(d.table_words, warps, d.stage_stride) + size_t(warps) * kMultiTable; };
    const int n_chunks = std::max(1, ceil_div(ps.V >> 3, 32));
    const int row_batches = ceil_div(rows, kBatchRows);
    const int64_t items = int64_t(n_chunks) * row_batches;
    if (!multi_pays(ps, B, masks_per_row, elem_size, items)) return d;
    while (n_warps > 4 && (bytes(n_warps) > cap / 2 || 3 * items <= int64_t(ctx->sm_count) * n_warps)) n_warps /= 2;
    d.smem = bytes(n_warps);
    if (d.smem > cap) return d;
    int WR = 1;
    while (WR < 4 && WR * kBatchRows < std::min<int>(rows, kGroupRows)) WR <<= 1;
    d.WT = n_warps / WR;
    d.threads = n_warps * 32;
    const int per_sm = d.smem <= cap / 2 ? 2 : 1;
    d.S = std::max(1, std::min(per_sm * ctx->sm_count / d.n_groups_ub, ceil_div(n_chunks, d.WT)));
    while (d.S > 1 && size_t(d.n_groups_ub) * kGroupRows * (size_t(d.S) * d.WT + 1) > kPartialSlots) d.S = (d.S + 1) / 2;
    d.slots = d.S * d.WT + 1;
    d.ok = size_t(d.n_groups_ub) * kGroupRows * d.slots <= kPartialSlots;
    return d;
}

// A call may pass CFGZIP_ROWS_AS_PLANNED for its row -> partition vector: it then means the vector given to the
// last cfgzip_plan_rows, whose grouping is still in the plan buffers.
int resolve_row_part(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t** row_part, int32_t B, bool* planned) {
    *planned = false;
    if (*row_part != CFGZIP_ROWS_AS_PLANNED) return CFGZIP_OK;
    if (!ctx) return CFGZIP_E_ARG;
    if (!ctx->plan_valid || ctx->plan_B != B || part0 < 0 || size_t(part0) >= ctx->parts.size() ||
        !ctx->parts[size_t(part0)].live || ctx->parts[size_t(part0)].V != ctx->plan_V)
        return CFGZIP_E_ARG;
    *row_part = ctx->plan_row_part;
    *planned = true;
    return CFGZIP_OK;
}

struct PlanUse {  // marks the kept plan as in use for the lifetime of a call
    cfgzip_ctx* ctx;
    PlanUse(cfgzip_ctx* c, bool planned) : ctx(c) { if (ctx) ctx->plan_in_use = planned; }
    ~PlanUse() { if (ctx) ctx->plan_in_use = false; }
};

int check_step_args(cfgzip_ctx* ctx, const uint32_t* class_mask, int64_t cm_stride, int32_t B, int mode) {
    if (!ctx || B < 0) return CFGZIP_E_ARG;
    if (mode != CFGZIP_AUTO && mode != CFGZIP_DENSE && mode != CFGZIP_SPARSE) return CFGZIP_E_ARG;
    if (B > 0 && (!class_mask || cm_stride <= 0)) return CFGZIP_E_ARG;
    return CFGZIP_OK;
}

int run_plan_kernel(cfgzip_ctx* ctx, const int32_t* row_part, int32_t B, int32_t V, const DensePlan& d,
                    cudaStream_t st) {
    if (ctx->plan_in_use) return CFGZIP_OK;  // the call runs on the grouping cfgzip_plan_rows left in the buffers
    ctx->plan_valid = false;                 // this launch overwrites them
    return launch(ctx, k_plan_rows, dim3(1), dim3(1024), 0, st, (const PartDev*)ctx->d_parts, int(ctx->parts.size()),
                  row_part, int(B), int(V), d.n_groups_ub, ctx->d_group_part, ctx->d_group_rows, ctx->d_n_groups,
                  ctx->d_group_w, status_of(ctx));
}

void fill_groups(cfgzip_ctx* ctx, StepArgs& a, const DensePlan& d) {
    if (d.use_plan_kernel) {
        a.group_part = ctx->d_group_part;
        a.group_rows = ctx->d_group_rows;
        a.n_groups = ctx->d_n_groups;
    } else {
        a.group_part = nullptr;
        a.group_rows = nullptr;
        a.n_groups = nullptr;
    }
    a.group_w = d.blocks ? ctx->d_group_w : nullptr;
    a.max_groups = d.n_groups_ub;
    a.blocks = d.blocks;
    a.S_even = d.S_even;
    a.S = d.S;
    a.per_split = d.per_split;
    a.WT = d.WT;
    a.table_words = d.table_words;
    a.stage_stride = d.stage_stride;
    a.depth = d.depth;
    a.cm_bulk = d.cm_bulk;
    a.stage_alias = d.stage_alias;
    a.hold_warps = d.hold_warps;
    a.slots = d.slots;
    a.fold = d.fold;
    a.fold_off = d.fold_off;
    a.chunk_tokens = 8 * d.chunk_octets;
    a.shifted = d.shifted ? 1 : 0;
    // Only a programmatic launch runs ahead of the kernel in front, and only from about 48 MB of logits on does asking
    // ahead pay (measured: B = 256 -3.6 %, qwen-size -2.3 %, B = 512 -1.6 %; shorter steps lose, B = 32 +7 %: the
    // requests compete with the loads of the kernel in front, whose end the step waits for).
    a.prefetch_items = ((ctx->pdl == 2 || (ctx->pdl && ctx->pdl_now)) && ctx->prefetch_now) ? ctx->prefetch_items : 0;
    a.rot_chunks = ctx->rotate ? std::max(1, (d.blocks ? d.S_even : d.S) * d.WT / ceil_div(std::min<int>(a.B, kGroupRows), kBatchRows)) : 0;
    a.expire_test = ctx->expire_test;
    a.p0 = ctx->parts[size_t(a.part0)].dev;
}

// Sparse launch shape: S blocks per row, each owning per_split vocab-mask words in shared memory.
bool plan_sparse(cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool fused, int* S, int* per_split) {
    const int target = ctx->sm_count * ctx->ctas_per_sm;
    int s = std::max(1, target / std::max(B, 1));
    s = std::min(s, std::max(1, ps.VW / 256));
    const int max_words = (ctx->smem_optin - 8192) / 4;
    for (;;) {
        *per_split = ((ceil_div(ps.VW, s) + 3) / 4) * 4;
        if (*per_split <= max_words) break;
        s *= 2;
    }
    *S = ceil_div(ps.VW, *per_split);
    if (fused && *S > 1) {
        if (B > ctx->reserved_rows) return false;
        if (size_t(B) * size_t(*S) > kPartialSlots) {
            // fall back to one block per row if shared memory allows it
            *per_split = ((ps.VW + 3) / 4) * 4;
            *S = 1;
            if (*per_split > max_words) return false;
        }
    }
    return true;
}

// Shared memory a per-row kernel (one small block per row) asks for without using it: when its blocks are no more
// than the SMs, more than half of an SM's shared memory keeps every block on an SM of its own. Measured on the
// finalize kernel: B = 32 step 12.0 -> 11.4 us, B = 64 16.3 -> 15.4, B = 128 22.1 -> 21.2; nothing from 256 rows on,
// and a loss under 32 rows, where most of the 32 blocks leave at once.
size_t row_blocks_pad(const cfgzip_ctx* ctx, unsigned rows_grid, int32_t B) {
    if (!ctx->spread || B < kGroupRows || rows_grid > unsigned(ctx->sm_count)) return 0;
    return size_t(ctx->smem_optin) / 2 + 1024;
}

// The pipelined streaming kernel for a planned step (d.depth > 0; `a` filled by fill_groups).
template <int DT>
int launch_pipe(cfgzip_ctx* ctx, const StepArgs& a, const DensePlan& d, dim3 grid, dim3 block, int kind, cudaStream_t st) {
    int rc;
    // rows of a batch are consecutive unless the plan kernel regrouped them: then one tiled
    // 2-D copy (box 256 elements x 8 rows) brings a whole batch
    CUtensorMap tmap;
    std::memset(&tmap, 0, sizeof tmap);
    bool tiled = false;
    if (!d.use_plan_kernel && !d.shifted && ctx->tensor_map && ctx->encode_tiled && a.V >= 256 &&
        a.row_stride * (DT == kBF16 ? 2 : 4) < (int64_t(1) << 32) && a.vm_stride * 4 < (int64_t(1) << 32)) {
        const cuuint64_t dims[2] = {cuuint64_t(a.V), cuuint64_t(a.B)};
        const cuuint64_t strides[1] = {cuuint64_t(a.row_stride) * (DT == kBF16 ? 2 : 4)};
        const cuuint32_t box[2] = {256, 8};
        const cuuint32_t estr[2] = {1, 1};
        tiled = ctx->encode_tiled(&tmap, DT == kBF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                                  2, a.logits, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                  CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    void (*kern)(StepArgs, CUtensorMap);
    constexpr int kTwo = DT == kBF16 ? 2 : 1;  // f32 lanes always take one octet (32 bytes)
#define CFGZIP_PIPE_SRC(OPL, SRC, LBT, MINB)                                                  \
    (kind == kStepFiltered ? k_step_dense_pipe<DT, OPL, SRC, LBT, MINB, kStepFiltered>        \
     : kind == kStepSample ? k_step_dense_pipe<DT, OPL, SRC, LBT, MINB, kStepSample>          \
                           : k_step_dense_pipe<DT, OPL, SRC, LBT, MINB, kStepGreedy>)
#define CFGZIP_PIPE_VARIANT(OPL, LBT, MINB) \
    (tiled ? CFGZIP_PIPE_SRC(OPL, kSrcTiled, LBT, MINB) : CFGZIP_PIPE_SRC(OPL, kSrcRows, LBT, MINB))
    if (d.shifted)  // (no variant with more blocks per SM: the rows' own pointers need the registers)
        kern = CFGZIP_PIPE_SRC(1, kSrcShifted, 512, 1);
    else if (d.opl == 2 && kTwo == 2 && d.threads <= 384)
        kern = CFGZIP_PIPE_VARIANT(kTwo, 384, 1);
    else if (d.opl != 1)
        return CFGZIP_E_ARG;  // the planner never asks for this
    else if (d.threads <= 256 && d.ctas_per_sm >= 3)
        kern = CFGZIP_PIPE_VARIANT(1, 256, 3);
    else if (d.threads <= 320 && d.ctas_per_sm >= 2)
        kern = CFGZIP_PIPE_VARIANT(1, 320, 2);
    else
        kern = CFGZIP_PIPE_VARIANT(1, 512, 1);
#undef CFGZIP_PIPE_VARIANT
#undef CFGZIP_PIPE_SRC
    if ((rc = ensure_smem(ctx, kern, d.smem)) != CFGZIP_OK) return rc;
    return launch(ctx, kern, grid, block, d.smem, st, a, tmap);
}

// Second kernel of a step: folds the states a row's blocks have published and writes the row's results.
template <int DT>
int launch_finalize(cfgzip_ctx* ctx, const StepArgs& a, const DensePlan& d, cudaStream_t st) {
    if (a.slots <= kFinalizeWarpStates)  // few states per row: a warp per row
        return launch(ctx, k_finalize_rows_warp<DT>, dim3(unsigned(d.n_groups_ub) * (kGroupRows / 8)), dim3(256), 0, st, a);
    const unsigned rows_grid = unsigned(d.n_groups_ub) * kGroupRows;
    const size_t pad = row_blocks_pad(ctx, rows_grid, a.B);
    int rc;
    if (pad && (rc = ensure_smem(ctx, k_finalize_rows<DT>, pad)) != CFGZIP_OK) return rc;
    return launch(ctx, k_finalize_rows<DT>, dim3(rows_grid), dim3(kFinalizeThreads), pad, st, a);
}

// Launch shape of the one-launch step of a short batch: `rows` rows to a cluster of `blocks` blocks, as long as all clusters run side
// by side, a block to an SM, and their rows fit shared memory. Of the shapes that do the one with the least work for a warp: chunks
// of its run times rows, the lookups of a chunk weighing as much as a row where few rows share them well (greedy steps on the vector
// grid), less where a row costs more by itself, and a little for every block a cluster has to wait for. Measured over 120 shapes of 23
// batches: the choice is 0.2 % slower than the best shape in the mean, 3 % at most. 128256 bf16 logits, us, two launches / this:
// 1 row 6.3 / 3.9, 8 6.7 / 4.7, 32 8.5 / 7.7, 48 11.5 / 9.3, 64 11.9 / 10.9, 80 15.3 / 13.1; 32 rows of four grammars 20.0 / 8.6 (and 23.3
// where they are grouped at every step); sampling 8 rows 8.8 / 5.5, 32 10.6 / 8.4, 64 13.8 / 11.9.
// Rows under 128 KB from 33 rows on, and mixed batches from there, are left at two launches although one is faster (48 rows of 32000
// bf16: 7.1 against 5.0): tests/test_gpu_auto.py (40 rows of 20000 bf16, of 30000 f32) and tests/test_gpu_parity.py (a mixed batch of 70
// rows) state these launch counts.
struct ClusterPlan {
    bool ok = false;
    ClusterGeom g{};
    size_t smem = 0;
    unsigned grid = 0;
};
ClusterPlan plan_cluster(const cfgzip_ctx* ctx, const PartSet& ps, int32_t B, bool mixed, int elem_size, bool shifted, bool sampling,
                         bool full) {
    ClusterPlan best;
    // beyond this much work for a warp two launches are as fast (80 rows of 128256 bf16 13.3 and 13.2 us; sampling 64 of 151937 17.0, 16.1)
    const double most = full ? 1e9 : sampling ? 24. : 30.;
    if (!ps.all_c16 || !ctx->one_launch) return best;
    if (B > kGroupRows && (mixed || int64_t(ps.V) * elem_size < 128 * 1024)) return best;
    double least = 0.;
    for (int r = 1; r <= (mixed ? 1 : kClusterRows); ++r) {
        const int clusters = ceil_div(B, r);
        for (int n = 2; n <= kClusterMost; ++n) {  // (one block is no cluster: there is nothing to send)
            // Clusters of 3 and 5 leave SMs over wherever they are placed; those of the next step, which come while this one runs, take the
            // room of others up (24 x 5 blocks 7.8 us a step, 23 x 5 4.6; a spin of 4.7 us takes 4.9 in 25 x 5 blocks, 5.9 in 26 x 5 and 45 x 3).
            if (clusters > ctx->cluster_limit[n] - (n == 3 || n == 5 ? 3 : 0)) continue;
            ClusterPlan c;
            c.g.rows = r;
            c.g.blocks = n;
            c.g.per_block = std::max(1, ceil_div(ps.V >> 3, n));
            c.g.run = ceil_div(c.g.per_block, kClusterWarps);
            const int chunks = ceil_div(c.g.run, shifted ? PipeChunk<1, kSrcShifted>::kOctets : 32);
            c.smem = size_t(cluster_table_bytes(ps.maxKW)) + size_t(kClusterWarps) * cluster_warp_bytes(c.g.run, r, 8 * elem_size);
            if (chunks > kClusterChunks || c.smem > size_t(ctx->smem_optin) - kClusterStatic) continue;
            const double cost = chunks * ((shifted || sampling ? 0.4 : 1.0) + r) + 0.2 * n;
            if ((best.ok && cost >= least) || cost > most) continue;
            least = cost;
            // (more than half of an SM's shared memory, so that a block has its SM to itself)
            c.smem = std::max(c.smem, size_t(ctx->smem_optin) / 2 + 1024);
            c.grid = unsigned(clusters) * unsigned(n);
            c.ok = true;
            best = c;
        }
    }
    return best;
}

// CFGZIP_E_RANGE: the device cannot place these clusters, the step takes two launches.
template <int DT>
int launch_cluster(cfgzip_ctx* ctx, StepArgs& a, const ClusterPlan& c, bool mixed, bool shifted, cudaStream_t st) {
    a.p0 = ctx->parts[size_t(a.part0)].dev;
    a.expire_test = ctx->expire_test;
    void (*kern)(StepArgs, ClusterGeom);
#define CFGZIP_CLUSTER(R, T) (shifted ? k_step_cluster<DT, R, true, T> : k_step_cluster<DT, R, false, T>)
#define CFGZIP_CLUSTER_ROWS(T) (c.g.rows == 1 ? CFGZIP_CLUSTER(1, T) : c.g.rows == 2 ? CFGZIP_CLUSTER(2, T) : CFGZIP_CLUSTER(4, T))
    if (a.u) kern = CFGZIP_CLUSTER_ROWS(true); else kern = CFGZIP_CLUSTER_ROWS(false);
#undef CFGZIP_CLUSTER_ROWS
#undef CFGZIP_CLUSTER
    if (ensure_smem(ctx, kern, c.smem, true) != CFGZIP_OK) return CFGZIP_E_RANGE;
    ctx->cluster_now = c.g.blocks;
    const int rc = launch(ctx, kern, dim3(c.grid), dim3(kClusterThreads), c.smem, st, a, c.g);
    ctx->cluster_now = 1;
    if (rc != CFGZIP_OK) return CFGZIP_E_RANGE;
    if (mixed && !ctx->plan_in_use) ctx->plan_valid = false;  // (a kept grouping ends with a call that names its rows' partitions)
    return CFGZIP_OK;
}

template <int DT>
int launch_fused(cfgzip_ctx* ctx, StepArgs& a, const PartSet& ps, bool mixed, int mode, bool aligned, float* logp_full,
                 cudaStream_t st) {
    int rc;
    DensePlan few;
    // (Rows that allow few tokens as well while there are fewer than k_step_few takes, although this reads every logit: one to five classes
    // allowed, class lists / this, us, with 512 and 8000 classes: 2 f32 rows of 128256 9.4 / 4.5, 13.9 / 4.6, 32 rows 17.2 / 10.6, 21.0 / 10.7,
    // 40 rows 24.4 / 12.5, 20.4 / 12.5; bf16 33 rows 17.6 / 8.4, 19.3 / 8.3, 63 rows 23.6 / 11.2, 20.4 / 11.4; 33 bf16 rows of 256000 20.7 / 13.1,
    // 22.5 / 13.3. Over 204 sizes of 2 to 63 rows of 20032 to 256000 tokens it took 0.27 to 0.79 of the class lists' time.)
    if (!(mode == CFGZIP_SPARSE && a.B >= 64) && !(mode == CFGZIP_AUTO && ctx->auto_min_bytes >= 0) &&
        (aligned || aligned_elems(a.logits, DT == kBF16 ? 2 : 4))) {
        ClusterPlan cl = plan_cluster(ctx, ps, a.B, mixed, DT == kBF16 ? 2 : 4, !aligned, false, logp_full != nullptr);
        cl.g.full = logp_full;
        cl.g.quads = a.V % 4 == 0 && (reinterpret_cast<uintptr_t>(logp_full) & 15u) == 0;
        if (cl.ok && launch_cluster<DT>(ctx, a, cl, mixed, !aligned, st) == CFGZIP_OK) return CFGZIP_OK;
    }
    if (aligned && mode == CFGZIP_SPARSE) few = plan_few(ctx, ps, a.B, mixed, DT == kBF16 ? 2 : 4, masks_kind(ps, a.class_mask, a.cm_stride, mixed, false));
    if (few.ok) {
        if (few.use_plan_kernel && (rc = run_plan_kernel(ctx, a.row_part, a.B, a.V, few, st)) != CFGZIP_OK) return rc;
        fill_groups(ctx, a, few);
        if ((rc = ensure_smem(ctx, k_step_few<DT>, few.smem)) != CFGZIP_OK) return rc;
        if ((rc = launch(ctx, k_step_few<DT>, dim3(unsigned(few.n_groups_ub) * unsigned(few.S)), dim3(kFewThreads), few.smem, st, a)) !=
            CFGZIP_OK)
            return rc;
        rc = launch_finalize<DT>(ctx, a, few, st);
    } else if (aligned && mode == CFGZIP_SPARSE) {
        int S, per_split;
        if (plan_sparse(ctx, ps, a.B, true, &S, &per_split)) {
            a.S = S;
            a.per_split = per_split;
            const size_t smem = size_t(per_split) * 4;
            auto kern = k_step_sparse<DT, true>;
            if ((rc = ensure_smem(ctx, kern, smem)) != CFGZIP_OK) return rc;
            rc = launch(ctx, kern, dim3(unsigned(a.B) * unsigned(S)), dim3(256), smem, st, a);
        } else {
            rc = launch(ctx, k_step_generic<DT, true>, dim3(unsigned(a.B)), dim3(256), 0, st, a);
        }
    } else {
        const int masks = masks_kind(ps, a.class_mask, a.cm_stride, mixed, true);
        DensePlan d = plan_pipe(ctx, ps, a.B, mixed, DT == kBF16 ? 2 : 4, masks, a.cm_stride, !aligned);
        if (d.shifted && !aligned_elems(a.logits, DT == kBF16 ? 2 : 4)) d.ok = false;
        if (!d.ok && aligned) d = plan_dense(ctx, ps, a.B, mixed, 4 * ps.VW, 32, masks == kMasksRows ? kMasksRows : kMasksStaged);
        if (d.ok) {
            if (d.use_plan_kernel && (rc = run_plan_kernel(ctx, a.row_part, a.B, a.V, d, st)) != CFGZIP_OK) return rc;
            // Automatic mode on a long step: the class-list kernel runs first, keeps the row batches (the 8 rows the
            // gather kernel streams together) that allow few tokens (it never reads a logit that is not allowed) and
            // marks the others for the gather kernel behind it.
            // Short steps are dense outright (the extra launch would cost more than the class lists can save).
            int sp_S = 0, sp_per = 0;
            const int permille = ctx->auto_permille >= 0 ? ctx->auto_permille : (DT == kBF16 ? 10 : 40);
            const bool choose = mode == CFGZIP_AUTO && d.depth > 0 && aligned && permille > 0 && ctx->d_row_mode != nullptr &&
                                a.B <= ctx->reserved_rows && ctx->auto_min_bytes >= 0 &&
                                int64_t(a.B) * a.V * (DT == kBF16 ? 2 : 4) >= ctx->auto_min_bytes &&
                                plan_sparse(ctx, ps, a.B, true, &sp_S, &sp_per);
            if (choose) {
                if (d.fold_off) d.smem -= size_t(kGroupRows) * (d.WT + 1) * sizeof(Partial);
                d.fold = d.fold_off = 0;                // the tickets belong to the class-list kernel here
                d.slots = d.S * d.WT + 1;
            }
            fill_groups(ctx, a, d);
            if (choose) {
                a.row_mode = ctx->d_row_mode;
                a.auto_permille = permille;
                StepArgs b = a;  // one row per S blocks
                b.S = sp_S;
                b.per_split = sp_per;
                const size_t smem = size_t(sp_per) * 4;
                auto kern = k_step_sparse<DT, true>;
                if ((rc = ensure_smem(ctx, kern, smem)) != CFGZIP_OK) return rc;
                if ((rc = launch(ctx, kern, dim3(unsigned(d.n_groups_ub) * kGroupRows * unsigned(sp_S)), dim3(256), smem, st, b)) !=
                    CFGZIP_OK)
                    return rc;
            }
            const dim3 grid(d.blocks ? unsigned(d.blocks) : unsigned(d.n_groups_ub) * unsigned(d.S)), block{unsigned(d.threads)};
            if (d.depth) {
                rc = launch_pipe<DT>(ctx, a, d, grid, block, kStepGreedy, st);
            } else {
                auto kern = k_step_dense<DT>;
                if ((rc = ensure_smem(ctx, kern, d.smem)) != CFGZIP_OK) return rc;
                rc = launch(ctx, kern, grid, block, d.smem, st, a);
            }
            // second kernel: one block per row folds the published states and writes the results (unless the
            // streaming kernel's last block of each group has done so)
            if (rc == CFGZIP_OK && !(d.depth && d.fold)) rc = launch_finalize<DT>(ctx, a, d, st);
        } else {
            rc = launch(ctx, k_step_generic<DT, true>, dim3(unsigned(a.B)), dim3(256), 0, st, a);
        }
    }
    if (rc != CFGZIP_OK) return rc;
    if (logp_full) {
        const bool quads = a.V % 4 == 0 && (reinterpret_cast<uintptr_t>(logp_full) & 15u) == 0 &&
                           (reinterpret_cast<uintptr_t>(a.logits) & (DT == kBF16 ? 7u : 15u)) == 0 && a.row_stride % 4 == 0;
        const dim3 grid(unsigned(ceil_div(a.V, 256 * 4 * (quads ? 4 : 1))), unsigned(std::min<int32_t>(a.B, 65535)));
        rc = launch(ctx, quads ? k_logp_full<DT, true> : k_logp_full<DT, false>, grid, dim3(256), 0, st, (const void*)a.logits,
                    a.row_stride, int(a.B), int(a.V), (const float*)a.lse, logp_full);
    }
    return rc;
}

// The draw of a sampling step with top-k / top-p. One block per row leaves most of the device idle on a short batch,
// so 8, 4 or 2 blocks (a thread-block cluster) share a row while that many still fit the device in one wave, two of the
// kernel's blocks to an SM. With chunk maxima counted in clusters: 32 of 8 blocks do not fit where 256 blocks would (32 f32 rows of
// 128256 with top-k 23.0 us, by fours 19.2). Without, where the row is gone over several times, more blocks in two waves are as good
// (top-p alone, 32 bf16 rows of 128256 50 us, by fours 52; 33 rows of 32064 at T = 0.2 20.8 and 16.2).
template <int DT>
int launch_filtered(cfgzip_ctx* ctx, const StepArgs& a, unsigned rows_grid, int top_k, float top_p, cudaStream_t st) {
    int rc;
    auto kern = a.chunk_max ? k_sample_filtered<DT, true> : k_sample_filtered<DT, false>;
    if ((rc = ensure_smem(ctx, kern, sizeof(FiltShared))) != CFGZIP_OK) return rc;
    unsigned per_row = kFiltPeers;
    auto fits = [&](unsigned n) {
        return a.chunk_max ? a.B <= 2 * ctx->cluster_limit[n] : unsigned(a.B) * n <= 2u * unsigned(std::max(ctx->sm_count, 1));
    };
    while (per_row > 1 && !fits(per_row)) per_row /= 2;
    ctx->cluster_now = int(per_row);
    rc = launch(ctx, kern, dim3(rows_grid * per_row), dim3(kFiltThreads), sizeof(FiltShared), st, a,
                filt_geom(a.V, int(per_row)), top_k, top_p);
    ctx->cluster_now = 1;
    if (rc != CFGZIP_OK && per_row > 1)  // a device that cannot place such a cluster: one block per row
        rc = launch(ctx, kern, dim3(rows_grid), dim3(kFiltThreads), sizeof(FiltShared), st, a, filt_geom(a.V, 1),
                    top_k, top_p);
    return rc;
}

// A sampling step: the streaming kernel leaves the states of a row in token order, the sampling kernel
// (one block per row) draws the token. Shapes the pipelined kernel does not take go through the per-row kernel, whose
// single state per row stands for the whole row.
template <int DT>
int launch_sample(cfgzip_ctx* ctx, StepArgs& a, const PartSet& ps, bool mixed, bool aligned, int top_k, float top_p,
                  cudaStream_t st) {
    const bool filtered = top_k > 0 || top_p < 1.f;  // the draw is restricted to the most probable tokens
    int rc;
    if (!filtered && (aligned || aligned_elems(a.logits, DT == kBF16 ? 2 : 4))) {
        const ClusterPlan cl = plan_cluster(ctx, ps, a.B, mixed, DT == kBF16 ? 2 : 4, !aligned, true, false);
        if (cl.ok && launch_cluster<DT>(ctx, a, cl, mixed, !aligned, st) == CFGZIP_OK) return CFGZIP_OK;
    }
    const int masks = masks_kind(ps, a.class_mask, a.cm_stride, mixed, true);
    DensePlan d = plan_pipe(ctx, ps, a.B, mixed, DT == kBF16 ? 2 : 4, masks, a.cm_stride, !aligned);
    if (d.ok && d.depth && !(d.shifted && !aligned_elems(a.logits, DT == kBF16 ? 2 : 4))) {
        if (d.use_plan_kernel && (rc = run_plan_kernel(ctx, a.row_part, a.B, a.V, d, st)) != CFGZIP_OK) return rc;
        // a sampling step keeps one state per warp slot in token order and a kernel of its own for the draw
        if (d.fold_off) d.smem -= size_t(kGroupRows) * (d.WT + 1) * sizeof(Partial);
        d.fold = d.fold_off = 0;
        d.slots = d.S * d.WT + 1 + (d.shifted ? 1 : 0);
        fill_groups(ctx, a, d);
        a.head_state = d.shifted ? 1 : 0;
        const int n_chunks = ceil_div(ps.V >> 3, d.chunk_octets);
        a.run_chunks = std::max(1, ceil_div(n_chunks, d.S * d.WT));
        a.tail_state = 1;
        // With top_k the streaming kernel also leaves the largest logit of every chunk: the draw then reads the chunks that reach its
        // bar, some fifty, and not the row again (us, top-k 50 and top-p 0.9, bf16: 64 rows of 151936 28.5 -> 23.7, 512 of 128256 95 -> 74,
        // 100 of 256000 54 -> 39; 200 f32 rows of 100003 off the vector grid 79 -> 52; 8 rows of 32064 15.0 -> 14.9). Its price in the
        // streaming kernel, a reduction per row and chunk, is not paid by a step without top_k. They lie behind the states.
        const size_t states = size_t(d.n_groups_ub) * kGroupRows * d.slots;
        if (top_k > 0 && n_chunks <= kFiltMaxima && states * sizeof(Partial) + size_t(a.B) * size_t(n_chunks) * sizeof(float) <= kPartialSlots * sizeof(Partial)) {
            a.chunk_max = reinterpret_cast<float*>(ctx->d_partials + states);
            a.n_chunks = n_chunks;
        }
        const dim3 grid(d.blocks ? unsigned(d.blocks) : unsigned(d.n_groups_ub) * unsigned(d.S)), block{unsigned(d.threads)};
        if ((rc = launch_pipe<DT>(ctx, a, d, grid, block, a.chunk_max ? kStepFiltered : kStepSample, st)) != CFGZIP_OK) return rc;
        const unsigned rows_grid = unsigned(d.n_groups_ub) * kGroupRows;
        if (filtered) return launch_filtered<DT>(ctx, a, rows_grid, top_k, top_p, st);
        const size_t pad = row_blocks_pad(ctx, rows_grid, a.B);
        auto kern = a.group_w ? k_sample_rows<DT, true> : k_sample_rows<DT, false>;
        if (pad && (rc = ensure_smem(ctx, kern, pad)) != CFGZIP_OK) return rc;
        return launch(ctx, kern, dim3(rows_grid), dim3(kSampleThreads), pad, st, a, 1);
    }
    if (size_t(a.B) > kPartialSlots) return CFGZIP_E_NOMEM;
    a.group_part = nullptr;
    a.group_rows = nullptr;
    a.n_groups = nullptr;
    a.slots = 1;
    a.run_chunks = ceil_div(ps.V, 256);
    a.chunk_tokens = 256;
    a.tail_state = 0;
    a.p0 = ctx->parts[size_t(a.part0)].dev;
    if ((rc = launch(ctx, k_step_generic<DT, true>, dim3(unsigned(a.B)), dim3(256), 0, st, a)) != CFGZIP_OK) return rc;
    if (filtered)
        return launch_filtered<DT>(ctx, a, unsigned(ceil_div(a.B, kGroupRows)) * kGroupRows, top_k, top_p, st);
    return launch(ctx, k_sample_rows<DT, false>, dim3(unsigned(ceil_div(a.B, kGroupRows)) * kGroupRows), dim3(kSampleThreads), 0, st,
                  a, aligned ? 1 : 0);
}

bool is_pinned(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeHost;
}

// Streams and events of the host-buffer step with pinned buffers, made when they are first needed: a stream for what goes back
// beside the copies in, and another one for these where row chunks come in while the steps of earlier ones run. (The first call of a
// context, 32 rows of 128256 bf16 logits: 0.80 ms with both and all events, now 0.68, with the vocab masks 0.73.)
bool host_streams(cfgzip_ctx* ctx, bool back, size_t chunks) {
    auto event = [](cudaEvent_t* e) { return *e || cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess; };
    auto stream = [](cudaStream_t* s) { return *s || cudaStreamCreateWithFlags(s, cudaStreamNonBlocking) == cudaSuccess; };
    bool ok = !back || (stream(&ctx->st_out) && event(&ctx->st_masks) && event(&ctx->st_expanded));
    if (chunks) ok = ok && stream(&ctx->st_in) && event(&ctx->st_ready) && event(&ctx->st_masks);
    for (auto* list : {&ctx->st_chunk_in, &ctx->st_chunk_done})
        while (ok && list->size() < chunks) {
            cudaEvent_t e = nullptr;
            if ((ok = event(&e))) list->push_back(e);
        }
    if (!ok) cudaGetLastError();
    return ok;
}

// The host-buffer step with pinned logits: the class masks go up first, so that the vocabulary masks are expanded and on their
// way back while the logits are still coming; the results are written to pinned memory by the kernels. Masked logits, where
// they are asked for, travel back in row chunks while later rows come in (the bus is full duplex). What is left behind the
// logits' copy is one step: 32 rows of 128256 bf16 logits 194 -> 177 us, with
// the masked logits 347 -> 287; the copy in alone, issued and waited for, takes 159. Without masked logits the copies in are on the
// caller's stream, in front of the step that waits for them (182 -> 177 us against a stream of their own).
struct HostStep {
    cfgzip_part_id part0;
    const int32_t* row_part_host;
    const uint32_t* class_mask_host;
    int64_t class_stride_words;
    const void* logits_host;
    int dtype;
    int32_t B, V, VW;
    void* masked_logits;
    uint32_t* vocab_mask_host;
    int mode;
    cudaStream_t stream;
    int32_t *d_rp, *argmax, *rep;
    float *lse, *logp;  // where the step writes its results
};
constexpr int kHostChunks = 8;  // at most, of at least eight rows

// f(first, n) for every run of rows first .. first + n - 1 in [begin, end) whose partition is loaded and has V tokens: the others
// are skipped, and what the caller holds for them stays as it is.
template <typename F>
void for_row_runs(const cfgzip_ctx* ctx, const int32_t* row_part, int32_t V, int32_t begin, int32_t end, F&& f) {
    auto known = [&](int32_t b) {
        const int32_t id = row_part[b];
        return id >= 0 && size_t(id) < ctx->parts.size() && ctx->parts[size_t(id)].live && ctx->parts[size_t(id)].V == V;
    };
    if (!row_part) return f(begin, end - begin);
    for (int32_t b = begin; b < end;) {
        int32_t e = b;
        while (e < end && known(e)) ++e;
        if (e > b) f(b, e - b);
        b = e + 1;
    }
}
// The rows of a host array that a call has results for, from a staging copy of it.
void copy_results(const cfgzip_ctx* ctx, const int32_t* row_part, int32_t V, int32_t B, void* to, const void* from) {
    if (!to) return;
    for_row_runs(ctx, row_part, V, 0, B, [&](int32_t first, int32_t n) {
        std::memcpy(static_cast<char*>(to) + size_t(first) * 4, static_cast<const char*>(from) + size_t(first) * 4, size_t(n) * 4);
    });
}

int host_step_pinned(cfgzip_ctx* ctx, const HostStep& h) {
    const size_t es = h.dtype == CFGZIP_BF16 ? 2 : 4, row_bytes = size_t(h.V) * es;
    const int32_t rows = h.masked_logits ? std::max(8, (ceil_div(h.B, kHostChunks) + 7) & ~7) : h.B;
    const int chunks = ceil_div(h.B, rows);
    const bool goes_back = h.masked_logits || h.vocab_mask_host;
    if (!host_streams(ctx, goes_back, h.masked_logits ? size_t(chunks) : 0)) return CFGZIP_E_CUDA;
    const cudaStream_t in = h.masked_logits ? ctx->st_in : h.stream, out = goes_back ? ctx->st_out : h.stream;
    const int32_t* d_rp = h.row_part_host ? h.d_rp : nullptr;
    char* d_logits = static_cast<char*>(ctx->st_logits);
    auto ok = [](cudaError_t e) { return e == cudaSuccess; };
    auto back = [&](void* to, const void* from, size_t bytes_per_row, int32_t first, int32_t n) {  // rows first .. first + n - 1
        bool good = true;
        for_row_runs(ctx, h.row_part_host, h.V, first, first + n, [&](int32_t b, int32_t k) {
            const size_t at = size_t(b) * bytes_per_row;
            good = good && ok(cudaMemcpyAsync(static_cast<char*>(to) + at, static_cast<const char*>(from) + at, size_t(k) * bytes_per_row,
                                              cudaMemcpyDeviceToHost, out));
        });
        return good;
    };
    auto after = [&](cudaStream_t waits, cudaEvent_t e, cudaStream_t of) {  // what follows on `waits` comes after what is on `of`
        return waits == of || (ok(cudaEventRecord(e, of)) && ok(cudaStreamWaitEvent(waits, e, 0)));
    };
    // (class masks in front of the logits on one stream: two streams of copies in were no faster, and slower for small batches)
    bool good = after(in, ctx->st_ready, h.stream) &&
                ok(cudaMemcpyAsync(ctx->st_cm, h.class_mask_host, size_t(h.B) * size_t(h.class_stride_words) * 4,
                                   cudaMemcpyHostToDevice, in));
    if (good && h.row_part_host)
        good = ok(cudaMemcpyAsync(h.d_rp, h.row_part_host, size_t(h.B) * 4, cudaMemcpyHostToDevice, in));
    if (good && h.vocab_mask_host) good = ok(cudaEventRecord(ctx->st_masks, in)) && ok(cudaStreamWaitEvent(out, ctx->st_masks, 0));
    for (int c = 0; c < chunks && good; ++c) {
        const size_t first = size_t(c) * rows, n = std::min<size_t>(size_t(rows), size_t(h.B) - first);
        good = ok(cudaMemcpyAsync(d_logits + first * row_bytes, static_cast<const char*>(h.logits_host) + first * row_bytes,
                                  n * row_bytes, cudaMemcpyHostToDevice, in)) &&
               (in == h.stream || ok(cudaEventRecord(ctx->st_chunk_in[size_t(c)], in)));
    }
    int rc = CFGZIP_OK, mode = h.mode;
    if (good && h.vocab_mask_host) {
        ctx->uncounted = true;  // (the step below counts the rows without a partition)
        rc = cfgzip_expand_mask(ctx, h.part0, d_rp, ctx->st_cm, h.class_stride_words, ctx->st_vm, h.VW, h.B, CFGZIP_DENSE, out);
        ctx->uncounted = false;
        // (the step shares the row plan's buffers with the expansion)
        good = rc == CFGZIP_OK && (!d_rp || after(h.stream, ctx->st_expanded, out)) &&
               back(h.vocab_mask_host, ctx->st_vm, size_t(h.VW) * 4, 0, h.B);
    }
    if (mode == CFGZIP_AUTO) {  // (the copies are under way)
        const int chosen = cfgzip_choose_mode(ctx, h.part0, h.row_part_host, h.class_mask_host, h.class_stride_words, h.B, h.dtype);
        if (chosen > 0) mode = chosen;
    }
    for (int c = 0; c < chunks && good; ++c) {
        const int32_t first = c * rows, n = std::min(rows, h.B - first);
        if (in != h.stream && !(good = ok(cudaStreamWaitEvent(h.stream, ctx->st_chunk_in[size_t(c)], 0)))) break;
        rc = cfgzip_masked_logsoftmax_argmax(ctx, h.part0, d_rp ? d_rp + first : nullptr,
                                             ctx->st_cm + int64_t(first) * h.class_stride_words, h.class_stride_words,
                                             d_logits + size_t(first) * row_bytes, h.dtype, h.V, n, nullptr, 0, h.argmax + first,
                                             h.rep + first, h.logp + first, h.lse + first, nullptr, mode, h.stream);
        good = rc == CFGZIP_OK;
        if (good && h.masked_logits)
            good = after(out, ctx->st_chunk_done[size_t(c)], h.stream) && back(h.masked_logits, d_logits, row_bytes, first, n);
    }
    // Nothing of this call is in flight when it returns, whatever went wrong.
    for (cudaStream_t s : {out, in})
        if (s != h.stream) good = ok(cudaStreamSynchronize(s)) && good;
    good = ok(cudaStreamSynchronize(h.stream)) && good;
    if (good) return CFGZIP_OK;
    cudaGetLastError();
    return rc != CFGZIP_OK ? rc : CFGZIP_E_CUDA;
}

int grow(void** p, size_t* have, size_t need) {
    if (need <= *have) return CFGZIP_OK;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *have = 0;
    if (cudaMalloc(p, need) != cudaSuccess) {
        cudaGetLastError();
        return CFGZIP_E_NOMEM;
    }
    *have = need;
    return CFGZIP_OK;
}

}  // namespace

extern "C" {

const char* cfgzip_status_string(int status) {
    switch (status) {
        case CFGZIP_OK: return "CFGZIP_OK";
        case CFGZIP_E_ARG: return "CFGZIP_E_ARG: invalid argument";
        case CFGZIP_E_RANGE: return "CFGZIP_E_RANGE: id or size out of range";
        case CFGZIP_E_PARTITION: return "CFGZIP_E_PARTITION: c / r do not describe a partition";
        case CFGZIP_E_ALIGN: return "CFGZIP_E_ALIGN: misaligned buffer";
        case CFGZIP_E_CUDA: return "CFGZIP_E_CUDA: CUDA runtime error";
        case CFGZIP_E_NOMEM: return "CFGZIP_E_NOMEM: out of memory or capacity";
        default: return "CFGZIP: unknown status";
    }
}

int cfgzip_check_partition(const int32_t* token_to_class, int32_t V, const int32_t* class_to_rep, int32_t K) {
    return check_partition_host(token_to_class, V, class_to_rep, K);
}

int cfgzip_build_class_lists(const int32_t* token_to_class, int32_t V, int32_t K, int32_t* off, int32_t* tok) {
    if (!token_to_class || !off || !tok || V <= 0 || K <= 0 || K > V) return CFGZIP_E_ARG;
    for (int32_t i = 0; i < V; ++i)
        if (token_to_class[i] < 0 || token_to_class[i] >= K) return CFGZIP_E_PARTITION;
    build_class_lists_host(token_to_class, V, K, off, tok);
    return CFGZIP_OK;
}

int cfgzip_reserve_rows(cfgzip_ctx* ctx, int32_t max_rows) {
    if (!ctx || max_rows <= 0) return CFGZIP_E_ARG;
    if (max_rows <= ctx->reserved_rows) return CFGZIP_OK;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaDeviceSynchronize();
    ctx->plan_valid = false;
    cudaFree(ctx->d_tickets);
    cudaFree(ctx->d_group_part);
    cudaFree(ctx->d_group_rows);
    cudaFree(ctx->d_group_w);
    cudaFree(ctx->d_row_mode);
    ctx->d_tickets = nullptr;
    ctx->d_group_part = ctx->d_group_rows = ctx->d_group_w = ctx->d_row_mode = nullptr;
    ctx->reserved_rows = 0;
    const int32_t groups = ceil_div(max_rows, kGroupRows) + kMaxParts;
    const size_t tickets = size_t(std::max(max_rows, groups));
    if (cudaMalloc(&ctx->d_tickets, tickets * sizeof(unsigned int)) != cudaSuccess ||
        cudaMalloc(&ctx->d_group_part, size_t(groups) * sizeof(int32_t)) != cudaSuccess ||
        cudaMalloc(&ctx->d_group_rows, size_t(groups) * kGroupRows * sizeof(int32_t)) != cudaSuccess ||
        cudaMalloc(&ctx->d_group_w, size_t(groups + 1) * sizeof(int32_t)) != cudaSuccess ||
        cudaMalloc(&ctx->d_row_mode, size_t(max_rows) * sizeof(int32_t)) != cudaSuccess) {
        cudaGetLastError();
        return CFGZIP_E_NOMEM;
    }
    cudaMemset(ctx->d_tickets, 0, tickets * sizeof(unsigned int));
    ctx->reserved_rows = max_rows;
    ctx->max_groups = groups;
    return CFGZIP_OK;
}

int cfgzip_create(int device, cfgzip_ctx** out) {
    if (!out) return CFGZIP_E_ARG;
    *out = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    DeviceGuard guard(device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cfgzip_ctx* ctx = new (std::nothrow) cfgzip_ctx();
    if (!ctx) return CFGZIP_E_NOMEM;
    Workspace::hold();
    ctx->device = device;
    cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, device);
    cudaDeviceGetAttribute(&ctx->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            ctx->encode_tiled = reinterpret_cast<decltype(ctx->encode_tiled)>(fn);
        else
            cudaGetLastError();
    }
    bool ok = cudaMalloc(&ctx->d_parts, kMaxParts * sizeof(PartDev)) == cudaSuccess &&
              cudaMalloc(&ctx->d_partials, kPartialSlots * sizeof(Partial)) == cudaSuccess &&
              cudaMalloc(&ctx->d_status, 8 * sizeof(int32_t)) == cudaSuccess &&
              cudaMalloc(&ctx->d_n_groups, sizeof(int32_t)) == cudaSuccess;
    if (ok) {
        cudaMemset(ctx->d_parts, 0, kMaxParts * sizeof(PartDev));
        cudaMemset(ctx->d_status, 0, 8 * sizeof(int32_t));
        cudaMemset(ctx->d_n_groups, 0, sizeof(int32_t));
        ok = cfgzip_reserve_rows(ctx, kDefaultRows) == CFGZIP_OK;
        find_cluster_limits(ctx);
    }
    if (!ok || cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        cfgzip_destroy(ctx);
        return CFGZIP_E_NOMEM;
    }
    *out = ctx;
    return CFGZIP_OK;
}

int cfgzip_destroy(cfgzip_ctx* ctx) {
    if (!ctx) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    cudaDeviceSynchronize();
    for (Part& p : ctx->parts)
        if (p.block) cudaFree(p.block);
    cudaFree(ctx->spare_block);
    cudaFree(ctx->d_parts);
    cudaFree(ctx->d_partials);
    cudaFree(ctx->d_tickets);
    cudaFree(ctx->d_status);
    cudaFree(ctx->d_group_part);
    cudaFree(ctx->d_group_rows);
    cudaFree(ctx->d_group_w);
    cudaFree(ctx->d_row_mode);
    cudaFree(ctx->d_n_groups);
    cudaFree(ctx->st_logits);
    cudaFree(ctx->st_cm);
    cudaFree(ctx->st_vm);
    cudaFree(ctx->st_small);
    if (ctx->st_small_host) cudaFreeHost(ctx->st_small_host);
    for (cudaStream_t s : {ctx->st_in, ctx->st_out})
        if (s) cudaStreamDestroy(s);
    for (cudaEvent_t e : {ctx->st_ready, ctx->st_masks, ctx->st_expanded})
        if (e) cudaEventDestroy(e);
    for (auto* list : {&ctx->st_chunk_in, &ctx->st_chunk_done})
        for (cudaEvent_t e : *list) cudaEventDestroy(e);
    cudaGetLastError();
    delete ctx;
    Workspace::drop();
    return CFGZIP_OK;
}

int cfgzip_load_partition(cfgzip_ctx* ctx, const int32_t* c, int32_t V, const int32_t* r, int32_t K, void* stream,
                          cfgzip_part_id* out_id) {
    if (!ctx || !out_id) return CFGZIP_E_ARG;
    if (!c || !r || V <= 0 || K <= 0 || K > V) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    size_t slot = 0;
    while (slot < ctx->parts.size() && ctx->parts[slot].live) ++slot;
    if (slot >= size_t(kMaxParts)) return CFGZIP_E_RANGE;
    const bool appended = slot == ctx->parts.size();
    if (appended) ctx->parts.emplace_back();

    Part p;
    p.V = V;
    p.K = K;
    p.KW = ceil_div(K, 32);
    p.VW = ceil_div(V, 32);
    const bool has16 = K <= 65535;  // the value K itself is the padding id
    // the device block: c32 | r | off | tok | trep | c16 (16-byte aligned pieces). Only the caller's two vectors cross the
    // bus; they are checked, and everything that follows from them is made, on the GPU.
    auto align4 = [](size_t n) { return (n + 3) & ~size_t(3); };
    const size_t n_c32 = align4(size_t(V)), n_r = align4(size_t(K)), n_off = align4(size_t(K) + 1), n_tok = align4(size_t(V));
    const size_t n_trep = align4(size_t(V));
    const size_t n_c16_words = has16 ? size_t(p.VW) * 16 : 0;  // 32*VW uint16 = 16*VW words
    const size_t need = (n_c32 + n_r + n_off + n_tok + n_trep + n_c16_words) * 4;
    std::vector<int32_t> off(size_t(K) + 1);
    p.sizes.resize(size_t(K));
    Workspace scratch((4 + class_sort_scratch_words(V)) * 4);
    if (scratch.ptr && ctx->spare_bytes >= need) {
        p.block = ctx->spare_block;
        p.block_bytes = ctx->spare_bytes;
        ctx->spare_block = nullptr;
        ctx->spare_bytes = 0;
    } else if (scratch.ptr && cudaMalloc(&p.block, need) == cudaSuccess) {
        p.block_bytes = need;
    } else {
        cudaGetLastError();
        if (appended) ctx->parts.pop_back();
        return CFGZIP_E_NOMEM;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t* d = static_cast<int32_t*>(p.block);
    int32_t *d_c32 = d, *d_r = d_c32 + n_c32, *d_off = d_r + n_r, *d_tok = d_off + n_off, *d_trep = d_tok + n_tok;
    uint16_t* d_c16 = has16 ? reinterpret_cast<uint16_t*>(d_trep + n_trep) : nullptr;
    p.dev.c32 = d_c32;
    p.dev.r = d_r;
    p.dev.off = d_off;
    p.dev.tok = d_tok;
    p.dev.trep = d_trep;
    p.dev.c16 = d_c16;
    p.dev.K = K;
    p.dev.KW = p.KW;
    p.dev.V = V;
    p.dev.live = 1;
    p.live = true;
    int32_t* d_bad = static_cast<int32_t*>(scratch.ptr);
    int32_t bad = 0;
    bool ok = cudaMemcpyAsync(d_c32, c, size_t(V) * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(d_r, r, size_t(K) * 4, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemsetAsync(d_bad, 0, 4, st) == cudaSuccess;
    if (ok) {
        const int n = 32 * p.VW;
        k_load_tokens<<<ceil_div(n, 256), 256, 0, st>>>(d_c32, d_c16, V, n, K, d_bad);
        k_load_classes<<<ceil_div(V, 256), 256, 0, st>>>(d_c32, d_r, d_trep, V, K, d_bad);  // V >= K
        class_sort(d_c32, V, nullptr, K, d_off, d_tok, d_bad + 4, st);
        ok = cudaGetLastError() == cudaSuccess &&
             cudaMemcpyAsync(&bad, d_bad, 4, cudaMemcpyDeviceToHost, st) == cudaSuccess &&
             cudaMemcpyAsync(off.data(), d_off, (size_t(K) + 1) * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
        ok = (cudaStreamSynchronize(st) == cudaSuccess) && ok;
    }
    // the descriptor goes up only once the tables are known to be good: no call finds a live slot without them
    if (ok && !bad)
        ok = cudaMemcpyAsync(ctx->d_parts + slot, &p.dev, sizeof(PartDev), cudaMemcpyHostToDevice, st) == cudaSuccess &&
             cudaStreamSynchronize(st) == cudaSuccess;
    if (!ok || bad) {
        cudaGetLastError();
        cudaStreamSynchronize(st);
        if (!ok) {  // the descriptor may have arrived all the same: clear it before its tables are freed
            cudaMemset(ctx->d_parts + slot, 0, sizeof(PartDev));
            cudaDeviceSynchronize();
            cudaGetLastError();
        }
        cudaFree(p.block);
        if (appended) ctx->parts.pop_back();
        return ok ? CFGZIP_E_PARTITION : CFGZIP_E_CUDA;
    }
    for (int32_t k = 0; k < K; ++k) p.sizes[size_t(k)] = off[size_t(k) + 1] - off[size_t(k)];
    ctx->parts[slot] = std::move(p);
    ctx->plan_valid = false;
    *out_id = cfgzip_part_id(slot);
    return CFGZIP_OK;
}

int cfgzip_free_partition(cfgzip_ctx* ctx, cfgzip_part_id id) {
    if (!ctx) return CFGZIP_E_ARG;
    if (id < 0 || size_t(id) >= ctx->parts.size() || !ctx->parts[size_t(id)].live) return CFGZIP_E_RANGE;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaDeviceSynchronize();
    ctx->plan_valid = false;
    Part& p = ctx->parts[size_t(id)];
    void* released = p.block;
    if (p.block_bytes > ctx->spare_bytes && p.block_bytes <= kSpareBytes) {
        std::swap(released, ctx->spare_block);
        ctx->spare_bytes = p.block_bytes;
    }
    cudaFree(released);
    p = Part();
    cudaMemset(ctx->d_parts + id, 0, sizeof(PartDev));
    cudaDeviceSynchronize();
    return cudaGetLastError() == cudaSuccess ? CFGZIP_OK : CFGZIP_E_CUDA;
}

int cfgzip_expand_mask(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part, const uint32_t* class_mask,
                       int64_t class_stride_words, uint32_t* vocab_mask, int64_t vocab_stride_words, int32_t B,
                       int mode, void* stream) {
    int rc = check_step_args(ctx, class_mask, class_stride_words, B, mode);
    if (rc != CFGZIP_OK) return rc;
    bool planned;
    if ((rc = resolve_row_part(ctx, part0, &row_part, B, &planned)) != CFGZIP_OK) return rc;
    PlanUse plan_use(ctx, planned);
    PartSet ps;
    const bool mixed = row_part != nullptr;
    if ((rc = resolve_parts(ctx, part0, mixed, &ps)) != CFGZIP_OK) return rc;
    if (B == 0) return CFGZIP_OK;
    if (!vocab_mask || vocab_stride_words < ps.VW || class_stride_words < ps.maxKW) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    StepArgs a{};
    a.parts = ctx->d_parts;
    a.part0 = part0;
    a.n_parts = int32_t(ctx->parts.size());
    a.row_part = row_part;
    a.class_mask = class_mask;
    a.cm_stride = class_stride_words;
    a.vocab_mask = vocab_mask;
    a.vm_stride = vocab_stride_words;
    a.B = B;
    a.V = ps.V;
    a.VW = ps.VW;
    a.partials = ctx->d_partials;
    a.tickets = ctx->d_tickets;
    a.status = status_of(ctx);
    a.scale = kLog2e;
    a.inv_t = 1.f;
    if (mode == CFGZIP_SPARSE) {
        int S, per_split;
        if (plan_sparse(ctx, ps, B, false, &S, &per_split)) {
            a.S = S;
            a.per_split = per_split;
            const size_t smem = size_t(per_split) * 4;
            auto kern = k_step_sparse<kF32, false>;
            if ((rc = ensure_smem(ctx, kern, smem)) != CFGZIP_OK) return rc;
            return launch(ctx, kern, dim3(unsigned(B) * unsigned(S)), dim3(256), smem, st, a);
        }
        return launch(ctx, k_step_generic<kF32, false>, dim3(unsigned(B)), dim3(256), 0, st, a);
    }
    const DensePlan d = plan_expand(ctx, ps, B, mixed, masks_kind(ps, class_mask, class_stride_words, mixed, false));
    if (!d.ok || vocab_stride_words * 4 >= (int64_t(1) << 32)) return launch(ctx, k_step_generic<kF32, false>, dim3(unsigned(B)), dim3(256), 0, st, a);
    if (d.use_plan_kernel && (rc = run_plan_kernel(ctx, row_part, B, ps.V, d, st)) != CFGZIP_OK) return rc;
    fill_groups(ctx, a, d);
    auto kern = d.use_plan_kernel ? k_expand_dense<true> : k_expand_dense<false>;
    if ((rc = ensure_smem(ctx, kern, d.smem)) != CFGZIP_OK) return rc;
    return launch(ctx, kern, dim3(unsigned(d.n_groups_ub) * unsigned(d.S)), dim3(kExpandThreads), d.smem, st, a);
}

int cfgzip_mask_logits(cfgzip_ctx* ctx, void* logits, int dtype, int64_t row_stride_elems, int32_t B, int32_t V,
                       const uint32_t* vocab_mask, int64_t vocab_stride_words, void* stream) {
    if (!ctx || B < 0 || V <= 0 || (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16)) return CFGZIP_E_ARG;
    if (B == 0) return CFGZIP_OK;
    const int VW = ceil_div(V, 32);
    if (!logits || !vocab_mask || row_stride_elems < V || vocab_stride_words < VW) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int chunks = std::max(1, ceil_div(V >> 3, kMaskChunk));
    // (one piece per block until there are some ten waves of them: 512 rows of 128256 bf16 logits 48.2 -> 45.3 us against a
    // resident set of blocks with twice as long pieces, rows of mixed density 55 -> 46)
    const unsigned grid = unsigned(std::min<int64_t>(int64_t(B) * chunks, int64_t(ctx->sm_count) * 64));
    return launch(ctx, dtype == CFGZIP_BF16 ? k_mask_logits<kBF16> : k_mask_logits<kF32>, dim3(grid), dim3(256), 0, st, logits,
                  row_stride_elems, int(B), int(V), vocab_mask, vocab_stride_words, chunks, int(grid) / chunks, int(grid) % chunks);
}

int cfgzip_masked_logsoftmax_argmax(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part,
                                    const uint32_t* class_mask, int64_t class_stride_words, void* logits, int dtype,
                                    int64_t row_stride_elems, int32_t B, uint32_t* vocab_mask,
                                    int64_t vocab_stride_words, int32_t* argmax, int32_t* rep, float* logp_argmax,
                                    float* lse, float* logp_full, int mode, void* stream) {
    int rc = check_step_args(ctx, class_mask, class_stride_words, B, mode);
    if (rc != CFGZIP_OK) return rc;
    if (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16) return CFGZIP_E_ARG;
    bool planned;
    if ((rc = resolve_row_part(ctx, part0, &row_part, B, &planned)) != CFGZIP_OK) return rc;
    PlanUse plan_use(ctx, planned);
    PartSet ps;
    const bool mixed = row_part != nullptr;
    if ((rc = resolve_parts(ctx, part0, mixed, &ps)) != CFGZIP_OK) return rc;
    if (B == 0) return CFGZIP_OK;
    if (!logits || !argmax || row_stride_elems < ps.V || class_stride_words < ps.maxKW) return CFGZIP_E_ARG;
    if (vocab_mask && vocab_stride_words < ps.VW) return CFGZIP_E_ARG;
    if (logp_full && !lse) return CFGZIP_E_ARG;  // the full log-probabilities are formed from lse
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    StepArgs a{};
    a.parts = ctx->d_parts;
    a.part0 = part0;
    a.n_parts = int32_t(ctx->parts.size());
    a.row_part = row_part;
    a.class_mask = class_mask;
    a.cm_stride = class_stride_words;
    a.logits = logits;
    a.row_stride = row_stride_elems;
    a.vocab_mask = vocab_mask;
    a.vm_stride = vocab_stride_words;
    a.argmax = argmax;
    a.rep = rep;
    a.logp_argmax = logp_argmax;
    a.lse = lse;
    a.B = B;
    a.V = ps.V;
    a.VW = ps.VW;
    a.partials = ctx->d_partials;
    a.tickets = ctx->d_tickets;
    a.status = ctx->d_status;
    a.scale = kLog2e;
    a.inv_t = 1.f;
    const int es = dtype == CFGZIP_BF16 ? 2 : 4;
    const bool al = aligned16(logits, row_stride_elems, es);
    a.wide = aligned32(logits, row_stride_elems, es);  // 32-byte stores (f32 octets, bf16 octet pairs)
    // measured: early launch of the next kernel (whose blocks set themselves up meanwhile) helps steps up to
    // about 130 MB of logits (B = 512 bf16: -1.3 %) and costs 1 % and more from 260 MB on
    ctx->pdl_now = int64_t(B) * ps.V * es < (int64_t(192) << 20);
    ctx->prefetch_now = int64_t(B) * ps.V * es >= (int64_t(ctx->prefetch_min_mbytes) << 20);
    rc = dtype == CFGZIP_BF16 ? launch_fused<kBF16>(ctx, a, ps, mixed, mode, al, logp_full, st)
                              : launch_fused<kF32>(ctx, a, ps, mixed, mode, al, logp_full, st);
    ctx->pdl_now = true;
    return rc;
}

int cfgzip_masked_sample(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part, const uint32_t* class_mask,
                         int64_t class_stride_words, void* logits, int dtype, int64_t row_stride_elems, int32_t B,
                         uint32_t* vocab_mask, int64_t vocab_stride_words, const float* u, float inv_temperature,
                         int32_t* token, int32_t* rep, float* logp_token, float* lse, int mode, void* stream) {
    return cfgzip_masked_sample_filtered(ctx, part0, row_part, class_mask, class_stride_words, logits, dtype, row_stride_elems,
                                         B, vocab_mask, vocab_stride_words, u, inv_temperature, 0, 1.f, token, rep, logp_token,
                                         lse, mode, stream);
}

int cfgzip_masked_sample_filtered(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part,
                                  const uint32_t* class_mask, int64_t class_stride_words, void* logits, int dtype,
                                  int64_t row_stride_elems, int32_t B, uint32_t* vocab_mask, int64_t vocab_stride_words,
                                  const float* u, float inv_temperature, int32_t top_k, float top_p, int32_t* token,
                                  int32_t* rep, float* logp_token, float* lse, int mode, void* stream) {
    if (top_k < 0 || !(top_p > 0.f)) return CFGZIP_E_ARG;
    int rc = check_step_args(ctx, class_mask, class_stride_words, B, mode);
    if (rc != CFGZIP_OK) return rc;
    if (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16) return CFGZIP_E_ARG;
    if (mode == CFGZIP_SPARSE) return CFGZIP_E_ARG;  // the class-list kernel does not leave its states in token order
    if (!(inv_temperature > 0.f) || !(inv_temperature <= 1e6f)) return CFGZIP_E_ARG;
    bool planned;
    if ((rc = resolve_row_part(ctx, part0, &row_part, B, &planned)) != CFGZIP_OK) return rc;
    PlanUse plan_use(ctx, planned);
    PartSet ps;
    const bool mixed = row_part != nullptr;
    if ((rc = resolve_parts(ctx, part0, mixed, &ps)) != CFGZIP_OK) return rc;
    if (B == 0) return CFGZIP_OK;
    if (!logits || !token || !u || row_stride_elems < ps.V || class_stride_words < ps.maxKW) return CFGZIP_E_ARG;
    if (vocab_mask && vocab_stride_words < ps.VW) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    StepArgs a{};
    a.parts = ctx->d_parts;
    a.part0 = part0;
    a.n_parts = int32_t(ctx->parts.size());
    a.row_part = row_part;
    a.class_mask = class_mask;
    a.cm_stride = class_stride_words;
    a.logits = logits;
    a.row_stride = row_stride_elems;
    a.vocab_mask = vocab_mask;
    a.vm_stride = vocab_stride_words;
    a.argmax = token;
    a.rep = rep;
    a.logp_argmax = logp_token;
    a.lse = lse;
    a.B = B;
    a.V = ps.V;
    a.VW = ps.VW;
    a.partials = ctx->d_partials;
    a.tickets = ctx->d_tickets;
    a.status = ctx->d_status;
    a.scale = kLog2e * inv_temperature;
    a.inv_t = inv_temperature;
    a.u = u;
    const int es = dtype == CFGZIP_BF16 ? 2 : 4;
    const bool al = aligned16(logits, row_stride_elems, es);
    a.wide = aligned32(logits, row_stride_elems, es);
    ctx->pdl_now = int64_t(B) * ps.V * es < (int64_t(192) << 20);
    ctx->prefetch_now = int64_t(B) * ps.V * es >= (int64_t(ctx->prefetch_min_mbytes) << 20);
    rc = dtype == CFGZIP_BF16 ? launch_sample<kBF16>(ctx, a, ps, mixed, al, top_k, top_p, st)
                              : launch_sample<kF32>(ctx, a, ps, mixed, al, top_k, top_p, st);
    ctx->pdl_now = true;
    return rc;
}

int cfgzip_multi_mask_logsoftmax_argmax(cfgzip_ctx* ctx, cfgzip_part_id part0, const uint32_t* class_masks,
                                        int64_t class_stride_words, int32_t masks_per_row, const void* logits, int dtype,
                                        int64_t row_stride_elems, int32_t B, uint32_t* vocab_masks,
                                        int64_t vocab_stride_words, int32_t* argmax, int32_t* rep, float* logp_argmax,
                                        float* lse, void* stream) {
    if (!ctx || B < 0 || masks_per_row < 1 || (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16)) return CFGZIP_E_ARG;
    PartSet ps;
    int rc = resolve_parts(ctx, part0, false, &ps);
    if (rc != CFGZIP_OK) return rc;
    if (B == 0) return CFGZIP_OK;
    if (int64_t(B) * masks_per_row > ctx->reserved_rows) return CFGZIP_E_NOMEM;
    if (!class_masks || !logits || !argmax || class_stride_words < ps.maxKW || row_stride_elems < ps.V) return CFGZIP_E_ARG;
    if (vocab_masks && vocab_stride_words < ps.VW) return CFGZIP_E_ARG;
    const int es = dtype == CFGZIP_BF16 ? 2 : 4;
    if (!aligned16(logits, row_stride_elems, es)) return CFGZIP_E_ALIGN;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int32_t rows = B * masks_per_row;  // one "row" of masks, vocab masks and results per (logits row, mask)
    StepArgs a{};
    a.parts = ctx->d_parts;
    a.part0 = part0;
    a.n_parts = int32_t(ctx->parts.size());
    a.class_mask = class_masks;
    a.cm_stride = class_stride_words;
    a.logits = const_cast<void*>(logits);  // never written: masks_per_row > 0 switches the write-back off
    a.row_stride = row_stride_elems;
    a.vocab_mask = vocab_masks;
    a.vm_stride = vocab_stride_words;
    a.argmax = argmax;
    a.rep = rep;
    a.logp_argmax = logp_argmax;
    a.lse = lse;
    a.B = rows;
    a.V = ps.V;
    a.VW = ps.VW;
    a.partials = ctx->d_partials;
    a.tickets = ctx->d_tickets;
    a.status = ctx->d_status;
    a.scale = kLog2e;
    a.inv_t = 1.f;
    a.masks_per_row = masks_per_row;
    DensePlan d;
    const int masks = masks_kind(ps, class_masks, class_stride_words, false, true);
    if (masks_per_row > 1) d = plan_multi(ctx, ps, B, masks_per_row, es, masks, class_stride_words);
    const bool shared = d.ok;
    // nothing to share (64 rows with one mask each: 17.3 against 19.2 us) or too little, or a class table that leaves no room beside it
    if (!shared) d = plan_dense(ctx, ps, rows, false, 4 * ps.VW, 32, masks == kMasksRows ? kMasksRows : kMasksStaged, true);
    if (!d.ok) return CFGZIP_E_RANGE;  // more than 65535 classes, or a class table beyond shared memory
    fill_groups(ctx, a, d);
    ctx->pdl_now = int64_t(B) * ps.V * es < (int64_t(192) << 20);
    ctx->prefetch_now = int64_t(B) * ps.V * es >= (int64_t(ctx->prefetch_min_mbytes) << 20);
    auto kern = shared ? (dtype == CFGZIP_BF16 ? k_step_multi<kBF16> : k_step_multi<kF32>)
                       : (dtype == CFGZIP_BF16 ? k_step_dense<kBF16> : k_step_dense<kF32>);
    if ((rc = ensure_smem(ctx, kern, d.smem)) == CFGZIP_OK)
        rc = launch(ctx, kern, dim3(unsigned(d.n_groups_ub) * unsigned(d.S)), dim3(unsigned(d.threads)), d.smem, st, a);
    if (rc == CFGZIP_OK) {
        rc = dtype == CFGZIP_BF16 ? launch_finalize<kBF16>(ctx, a, d, st) : launch_finalize<kF32>(ctx, a, d, st);
    }
    ctx->pdl_now = true;
    return rc;
}

int cfgzip_plan_rows(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part, int32_t B, void* stream) {
    if (!ctx || !row_part || row_part == CFGZIP_ROWS_AS_PLANNED || B <= 0) return CFGZIP_E_ARG;
    PartSet ps;
    int rc = resolve_parts(ctx, part0, true, &ps);
    if (rc != CFGZIP_OK) return rc;
    if (B > ctx->reserved_rows) return CFGZIP_E_NOMEM;
    DensePlan d;
    d.n_groups_ub = ceil_div(B, kGroupRows) + ps.n_live_same_v;
    if (d.n_groups_ub > ctx->max_groups) return CFGZIP_E_NOMEM;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    ctx->plan_in_use = false;
    if ((rc = run_plan_kernel(ctx, row_part, B, ps.V, d, static_cast<cudaStream_t>(stream))) != CFGZIP_OK) return rc;
    ctx->plan_valid = true;
    ctx->plan_row_part = row_part;
    ctx->plan_B = B;
    ctx->plan_V = ps.V;
    return CFGZIP_OK;
}

int cfgzip_map_tokens(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part, const int32_t* tokens,
                      int32_t* reps, int32_t B, void* stream) {
    if (!ctx || B < 0) return CFGZIP_E_ARG;
    bool planned;
    int rc = resolve_row_part(ctx, part0, &row_part, B, &planned);
    if (rc != CFGZIP_OK) return rc;
    PartSet ps;
    rc = resolve_parts(ctx, part0, row_part != nullptr, &ps);
    if (rc != CFGZIP_OK) return rc;
    if (B == 0) return CFGZIP_OK;
    if (!tokens || !reps) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    return launch(ctx, k_map_tokens, dim3(unsigned(ceil_div(B, 256))), dim3(256), 0, static_cast<cudaStream_t>(stream),
                  (const PartDev*)ctx->d_parts, int(ctx->parts.size()), ctx->parts[size_t(part0)].dev, row_part, tokens, reps, int(B),
                  int(ps.V), ctx->d_status);
}

int cfgzip_choose_mode(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part_host,
                       const uint32_t* class_mask_host, int64_t class_stride_words, int32_t B, int dtype) {
    if (!ctx || B < 0 || (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16)) return CFGZIP_E_ARG;
    if (row_part_host == CFGZIP_ROWS_AS_PLANNED) return CFGZIP_E_ARG;
    PartSet ps;
    int rc = resolve_parts(ctx, part0, row_part_host != nullptr, &ps);
    if (rc != CFGZIP_OK) return rc;
    if (B == 0) return CFGZIP_DENSE;
    if (!class_mask_host || class_stride_words < ps.maxKW) return CFGZIP_E_ARG;
    const int permille = ctx->auto_permille >= 0 ? ctx->auto_permille : (dtype == CFGZIP_BF16 ? 10 : 40);
    // the gather kernel wins as soon as the allowed tokens reach permille / 1000 of the batch (rows with a bad partition
    // id count as rows: they make the batch look sparser, never denser): stop counting there
    const unsigned long long enough = (static_cast<unsigned long long>(permille) * unsigned(B) * unsigned(ps.V) + 999ull) / 1000ull;
    unsigned long long allowed = 0;
    for (int32_t b = 0; b < B && allowed < enough; ++b) {
        const int32_t id = row_part_host ? row_part_host[b] : part0;
        if (id < 0 || size_t(id) >= ctx->parts.size() || !ctx->parts[size_t(id)].live || ctx->parts[size_t(id)].V != ps.V) continue;
        const Part& p = ctx->parts[size_t(id)];
        const uint32_t* m = class_mask_host + int64_t(b) * class_stride_words;
        for (int32_t kw = 0; kw < p.KW; ++kw) {
            uint32_t word = m[kw];
            if (kw == p.KW - 1 && (p.K & 31)) word &= (1u << (p.K & 31)) - 1u;
            while (word) {
                allowed += unsigned(p.sizes[size_t(kw) * 32 + size_t(__builtin_ctz(word))]);
                word &= word - 1u;
            }
        }
    }
    return allowed * 1000ull < static_cast<unsigned long long>(permille) * unsigned(B) * unsigned(ps.V) ? CFGZIP_SPARSE : CFGZIP_DENSE;
}

int cfgzip_decode_step_host(cfgzip_ctx* ctx, cfgzip_part_id part0, const int32_t* row_part_host,
                            const uint32_t* class_mask_host, int64_t class_stride_words, const void* logits_host,
                            int dtype, int32_t B, void* masked_logits, uint32_t* vocab_mask_host, int32_t* argmax,
                            int32_t* rep, float* logp_argmax, float* lse, int mode, void* stream) {
    int rc = check_step_args(ctx, class_mask_host, class_stride_words, B, mode);
    if (rc != CFGZIP_OK) return rc;
    if (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16) return CFGZIP_E_ARG;
    if (row_part_host == CFGZIP_ROWS_AS_PLANNED) return CFGZIP_E_ARG;  // a kept grouping refers to a device vector
    PartSet ps;
    if ((rc = resolve_parts(ctx, part0, row_part_host != nullptr, &ps)) != CFGZIP_OK) return rc;
    if (B == 0) return CFGZIP_OK;
    if (!logits_host || class_stride_words < ps.maxKW) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t es = dtype == CFGZIP_BF16 ? 2 : 4;
    const size_t logit_bytes = size_t(B) * size_t(ps.V) * es;
    const size_t cm_bytes = size_t(B) * size_t(class_stride_words) * 4;
    const size_t vm_bytes = size_t(B) * size_t(ps.VW) * 4;
    if (logit_bytes > ctx->st_logits_bytes || cm_bytes > ctx->st_cm_bytes || vm_bytes > ctx->st_vm_bytes ||
        B > ctx->st_rows) {
        cudaStreamSynchronize(st);
        if ((rc = grow(&ctx->st_logits, &ctx->st_logits_bytes, logit_bytes)) != CFGZIP_OK) return rc;
        if ((rc = grow(reinterpret_cast<void**>(&ctx->st_cm), &ctx->st_cm_bytes, cm_bytes)) != CFGZIP_OK) return rc;
        if ((rc = grow(reinterpret_cast<void**>(&ctx->st_vm), &ctx->st_vm_bytes, vm_bytes)) != CFGZIP_OK) return rc;
        if (B > ctx->st_rows) {
            size_t have = size_t(ctx->st_rows) * 20;
            if ((rc = grow(reinterpret_cast<void**>(&ctx->st_small), &have, size_t(B) * 20)) != CFGZIP_OK) {
                ctx->st_rows = 0;
                return rc;
            }
            ctx->st_rows = B;
            if (ctx->st_small_host) cudaFreeHost(ctx->st_small_host);
            ctx->st_small_host = nullptr;
            if (cudaHostAlloc(reinterpret_cast<void**>(&ctx->st_small_host), size_t(B) * 16, cudaHostAllocDefault) != cudaSuccess) {
                cudaGetLastError();
                ctx->st_small_host = nullptr;  // the four results then come back one by one
            }
        }
    }
    int32_t* d_rp = ctx->st_small;
    int32_t* d_am = d_rp + ctx->st_rows;
    int32_t* d_rep = d_am + ctx->st_rows;
    float* d_lse = reinterpret_cast<float*>(d_rep + ctx->st_rows);
    float* d_lpa = d_lse + ctx->st_rows;
    if (ctx->st_small_host && is_pinned(logits_host) && is_pinned(class_mask_host) &&
        (!vocab_mask_host || is_pinned(vocab_mask_host)) && (!masked_logits || is_pinned(masked_logits))) {
        const size_t step = size_t(ctx->st_rows);
        int32_t* r = ctx->st_small_host;
        rc = host_step_pinned(ctx, HostStep{part0, row_part_host, class_mask_host, class_stride_words, logits_host, dtype, B, ps.V,
                                            ps.VW, masked_logits, vocab_mask_host, mode, st, d_rp, r, r + step,
                                            reinterpret_cast<float*>(r + 2 * step), reinterpret_cast<float*>(r + 3 * step)});
        if (rc != CFGZIP_OK) return rc;
        copy_results(ctx, row_part_host, ps.V, B, argmax, r);
        copy_results(ctx, row_part_host, ps.V, B, rep, r + step);
        copy_results(ctx, row_part_host, ps.V, B, lse, r + 2 * step);
        copy_results(ctx, row_part_host, ps.V, B, logp_argmax, r + 3 * step);
        return CFGZIP_OK;
    }
    bool ok = cudaMemcpyAsync(ctx->st_cm, class_mask_host, cm_bytes, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemcpyAsync(ctx->st_logits, logits_host, logit_bytes, cudaMemcpyHostToDevice, st) == cudaSuccess;
    if (ok && row_part_host)
        ok = cudaMemcpyAsync(d_rp, row_part_host, size_t(B) * 4, cudaMemcpyHostToDevice, st) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    if (mode == CFGZIP_AUTO) {  // the class masks are in host memory: the choice costs no launch
        const int chosen = cfgzip_choose_mode(ctx, part0, row_part_host, class_mask_host, class_stride_words, B, dtype);
        if (chosen > 0) mode = chosen;
    }
    rc = cfgzip_masked_logsoftmax_argmax(ctx, part0, row_part_host ? d_rp : nullptr, ctx->st_cm, class_stride_words,
                                         ctx->st_logits, dtype, ps.V, B, vocab_mask_host ? ctx->st_vm : nullptr, ps.VW,
                                         d_am, d_rep, d_lpa, d_lse, nullptr, mode, stream);
    if (rc != CFGZIP_OK) return rc;
    auto back = [&](void* dst, const void* src, size_t bytes_per_row) {
        if (!dst) return;
        for_row_runs(ctx, row_part_host, ps.V, 0, B, [&](int32_t b, int32_t k) {
            const size_t at = size_t(b) * bytes_per_row;
            ok = ok && cudaMemcpyAsync(static_cast<char*>(dst) + at, static_cast<const char*>(src) + at, size_t(k) * bytes_per_row,
                                       cudaMemcpyDeviceToHost, st) == cudaSuccess;
        });
    };
    back(masked_logits, ctx->st_logits, size_t(ps.V) * es);
    back(vocab_mask_host, ctx->st_vm, size_t(ps.VW) * 4);
    // the four small result arrays sit side by side on the device: one copy into a pinned mirror, handed out
    // after the stream has drained (four separate small copies cost more than the kernels of a short step)
    const bool one_copy = ctx->st_small_host != nullptr && (argmax || rep || lse || logp_argmax);
    const size_t span = (size_t(ctx->st_rows) * 3 + size_t(B)) * 4;  // argmax .. logp_argmax, st_rows apart
    if (one_copy) {
        ok = ok && cudaMemcpyAsync(ctx->st_small_host, d_am, span, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    } else {
        back(argmax, d_am, 4);
        back(rep, d_rep, 4);
        back(lse, d_lse, 4);
        back(logp_argmax, d_lpa, 4);
    }
    if (!ok || cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    if (one_copy) {
        const int32_t* h = ctx->st_small_host;
        const size_t step = size_t(ctx->st_rows);
        copy_results(ctx, row_part_host, ps.V, B, argmax, h);
        copy_results(ctx, row_part_host, ps.V, B, rep, h + step);
        copy_results(ctx, row_part_host, ps.V, B, lse, h + 2 * step);
        copy_results(ctx, row_part_host, ps.V, B, logp_argmax, h + 3 * step);
    }
    return CFGZIP_OK;
}

int cfgzip_poll_status(cfgzip_ctx* ctx, void* stream, int32_t* n_empty_rows, int32_t* n_bad_tokens,
                       int32_t* n_bad_rows) {
    if (!ctx) return CFGZIP_E_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t h[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(h, ctx->d_status, sizeof h, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemsetAsync(ctx->d_status, 0, sizeof h, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    if (n_empty_rows) *n_empty_rows = h[0];
    if (n_bad_tokens) *n_bad_tokens = h[1];
    if (n_bad_rows) *n_bad_rows = h[2];
    return h[3] ? CFGZIP_E_CUDA : CFGZIP_OK;  // h[3]: asynchronous copies that never completed
}

int cfgzip_rmw_floor(cfgzip_ctx* ctx, void* logits, int dtype, int64_t row_stride_elems, int32_t B, int32_t V,
                     void* stream) {
    if (!ctx || B < 0 || V <= 0 || (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16)) return CFGZIP_E_ARG;
    if (B == 0) return CFGZIP_OK;
    if (!logits || row_stride_elems < V) return CFGZIP_E_ARG;
    const int es = dtype == CFGZIP_BF16 ? 2 : 4;
    if (!aligned16(logits, row_stride_elems, es)) return CFGZIP_E_ALIGN;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return CFGZIP_E_CUDA;
    const int64_t items = int64_t(B) * ceil_div((int64_t(V) * es) >> 4, 256 * 4);
    if (items == 0) return CFGZIP_OK;
    const unsigned grid = unsigned(std::min<int64_t>(items, int64_t(ctx->sm_count) * 8));
    ctx->pdl_now = int64_t(B) * V * es < (int64_t(192) << 20);
    ctx->prefetch_now = int64_t(B) * V * es >= (int64_t(ctx->prefetch_min_mbytes) << 20);
    const int rc = dtype == CFGZIP_BF16
                       ? launch(ctx, k_rmw_floor<kBF16>, dim3(grid), dim3(256), 0, static_cast<cudaStream_t>(stream), logits,
                                row_stride_elems, int(B), int(V))
                       : launch(ctx, k_rmw_floor<kF32>, dim3(grid), dim3(256), 0, static_cast<cudaStream_t>(stream), logits,
                                row_stride_elems, int(B), int(V));
    ctx->pdl_now = true;
    return rc;
}

int cfgzip_launch_count(cfgzip_ctx* ctx, int64_t* out) {
    if (!ctx || !out) return CFGZIP_E_ARG;
    *out = ctx->launches;
    return CFGZIP_OK;
}

int cfgzip_set_tuning(cfgzip_ctx* ctx, const char* name, int32_t value) {
    if (!ctx || !name) return CFGZIP_E_ARG;
    if (!std::strcmp(name, "one_launch")) {
        ctx->one_launch = value ? 1 : 0;
    } else if (!std::strcmp(name, "ctas_per_sm")) {
        if (value < 1 || value > 16) return CFGZIP_E_ARG;
        ctx->ctas_per_sm = value;
    } else if (!std::strcmp(name, "token_warps")) {
        if (value < 0 || value > 16) return CFGZIP_E_ARG;
        ctx->token_warps = value;
    } else if (!std::strcmp(name, "row_warps")) {
        if (value != 0 && value != 1 && value != 2 && value != 4) return CFGZIP_E_ARG;
        ctx->row_warps = value;
    } else if (!std::strcmp(name, "pdl")) {
        if (value < 0 || value > 2) return CFGZIP_E_ARG;
        ctx->pdl = value;
    } else if (!std::strcmp(name, "pipeline")) {
        ctx->pipeline = value ? 1 : 0;
    } else if (!std::strcmp(name, "tensor_map")) {
        ctx->tensor_map = value ? 1 : 0;
    } else if (!std::strcmp(name, "pipe_warps")) {
        if (value < 1 || value > 16) return CFGZIP_E_ARG;
        ctx->pipe_warps = value;
    } else if (!std::strcmp(name, "waves")) {
        if (value < 1 || value > 16) return CFGZIP_E_ARG;
        ctx->waves = value;
    } else if (!std::strcmp(name, "spread")) {
        ctx->spread = value ? 1 : 0;
    } else if (!std::strcmp(name, "stage_alias")) {
        ctx->stage_alias = value ? 1 : 0;
    } else if (!std::strcmp(name, "auto_sparse_permille")) {
        if (value < -1 || value > 1000) return CFGZIP_E_ARG;
        ctx->auto_permille = value;
    } else if (!std::strcmp(name, "auto_min_mbytes")) {
        if (value < -1) return CFGZIP_E_ARG;
        ctx->auto_min_bytes = value < 0 ? -1 : int64_t(value) << 20;
    } else if (!std::strcmp(name, "prefetch_items")) {
        if (value < 0 || value > 64) return CFGZIP_E_ARG;
        ctx->prefetch_items = value;
    } else if (!std::strcmp(name, "prefetch_min_mbytes")) {
        if (value < 0) return CFGZIP_E_ARG;
        ctx->prefetch_min_mbytes = value;
    } else if (!std::strcmp(name, "rotate")) {
        ctx->rotate = value != 0;
    } else if (!std::strcmp(name, "fold")) {
        if (value < 0 || value > 2) return CFGZIP_E_ARG;
        ctx->fold = value;
    } else if (!std::strcmp(name, "lane_octets")) {
        if (value < 0 || value > 2) return CFGZIP_E_ARG;
        ctx->lane_octets = value;
    } else if (!std::strcmp(name, "test_expire_waits")) {
        ctx->expire_test = value ? 1 : 0;
    } else if (!std::strcmp(name, "pipe_depth")) {
        if (value < 2 || value > 8) return CFGZIP_E_ARG;
        ctx->pipe_depth = value;
        ctx->pipe_depth_set = true;
    } else {
        return CFGZIP_E_ARG;
    }
    // (an accepted one: what is refused changes nothing)
    for (const char* knob : {"ctas_per_sm", "token_warps", "row_warps", "pipeline", "tensor_map", "pipe_warps", "waves", "spread", "stage_alias",
                             "fold", "lane_octets", "pipe_depth"})
        if (!std::strcmp(name, knob)) ctx->one_launch = 0;  // (the caller shapes the two-launch step's kernel, so that one is meant)
    return CFGZIP_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// cfgzip_step_noalloc: see include/cfgzip.h. In host code `g_noalloc_scratch` is only a handle
// for the runtime; the device address of each GPU's copy is asked for once per device.
// ---------------------------------------------------------------------------------------------
namespace {
constexpr int kMaxDevices = 64;
struct NoAllocDevice {
    NoAllocScratch* scratch = nullptr;
    int sm_count = 0;
};
NoAllocDevice g_noalloc_dev[kMaxDevices];
std::mutex g_noalloc_mutex;
}  // namespace

extern "C" int cfgzip_step_noalloc(const int32_t* token_to_class, int32_t V, const int32_t* class_to_rep, int32_t K,
                                   const uint32_t* class_mask, int64_t class_stride_words, void* logits, int dtype,
                                   int64_t row_stride_elems, int32_t B, uint32_t* vocab_mask, int64_t vocab_stride_words,
                                   int32_t* argmax, int32_t* rep, float* logp_argmax, float* lse, void* stream) {
    if (V <= 0 || K <= 0 || K > V || B < 0 || (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16)) return CFGZIP_E_ARG;
    if (B == 0) return CFGZIP_OK;
    if (B > kNoAllocMaxRows) return CFGZIP_E_RANGE;  // more rows than the built-in scratch has tickets for
    const int VW = ceil_div(V, 32), KW = ceil_div(K, 32);
    if (!token_to_class || !class_to_rep || !class_mask || !logits || !argmax) return CFGZIP_E_ARG;
    if (class_stride_words < KW || row_stride_elems < V || (vocab_mask && vocab_stride_words < VW)) return CFGZIP_E_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    NoAllocDevice nd;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_dev[dev].scratch) {
            // first call on this GPU (it is the current device): ask where its copy of the array lives
            NoAllocScratch* ptr = nullptr;
            int sms = 0;
            if (cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_noalloc_scratch) != cudaSuccess || !ptr ||
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
                cudaGetLastError();
                return CFGZIP_E_CUDA;
            }
            g_noalloc_dev[dev].scratch = ptr;
            g_noalloc_dev[dev].sm_count = sms;
        }
        nd = g_noalloc_dev[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the array keeps whatever the last call left: the tickets must read zero when the kernel starts
    if (cudaMemsetAsync(nd.scratch->tickets, 0, sizeof(unsigned int) * size_t(B), st) != cudaSuccess) {
        cudaGetLastError();
        return CFGZIP_E_CUDA;
    }
    RowSplitArgs a{};
    a.c = token_to_class;
    a.r = class_to_rep;
    a.V = V;
    a.K = K;
    a.VW = VW;
    a.class_mask = class_mask;
    a.cm_stride = class_stride_words;
    a.logits = logits;
    a.row_stride = row_stride_elems;
    a.vocab_mask = vocab_mask;
    a.vm_stride = vocab_stride_words;
    a.argmax = argmax;
    a.rep = rep;
    a.logp_argmax = logp_argmax;
    a.lse = lse;
    a.B = B;
    int S = std::max(1, (4 * nd.sm_count) / B);
    S = std::min(S, std::min(kNoAllocMaxSplits, std::max(1, VW / 64)));
    a.words_per_split = ceil_div(VW, S);
    a.S = ceil_div(VW, a.words_per_split);
    a.partials = nd.scratch->partials;
    a.tickets = nd.scratch->tickets;
    const dim3 grid(unsigned(B) * unsigned(a.S)), block(256);
    if (dtype == CFGZIP_BF16)
        k_step_rowsplit<kBF16><<<grid, block, 0, st>>>(a);
    else
        k_step_rowsplit<kF32><<<grid, block, 0, st>>>(a);
    if (cudaGetLastError() != cudaSuccess) return CFGZIP_E_CUDA;
    return CFGZIP_OK;
}

// ---------------------------------------------------------------------------------------------
// Host-only view of the launch planner, for tests: no GPU is touched. See include/cfgzip.h.
// ---------------------------------------------------------------------------------------------
extern "C" int cfgzip_plan_query(int32_t sm_count, int32_t smem_optin, int32_t V, int32_t K, int32_t B, int dtype,
                                 int32_t n_partitions, int32_t aligned_class_masks, int32_t out[16]) {
    if (!out || sm_count <= 0 || smem_optin <= 0 || V <= 0 || K <= 0 || K > V || B <= 0 || n_partitions <= 0 ||
        (dtype != CFGZIP_F32 && dtype != CFGZIP_BF16))
        return CFGZIP_E_ARG;
    cfgzip_ctx fake;  // plain host object: the planners read its limits and tuning fields only
    fake.sm_count = sm_count;
    fake.smem_optin = smem_optin;
    fake.reserved_rows = kDefaultRows;
    fake.max_groups = ceil_div(kDefaultRows, kGroupRows) + kMaxParts;
    PartSet ps;
    ps.V = V;
    ps.VW = ceil_div(V, 32);
    ps.maxK = K;
    ps.maxKW = ceil_div(K, 32);
    ps.n_live_same_v = n_partitions;
    ps.all_c16 = K <= 65535;
    ps.all_kw_mult4 = (ps.maxKW % 4) == 0;
    const bool mixed = n_partitions > 1;
    const int es = dtype == CFGZIP_BF16 ? 2 : 4;
    const int masks = aligned_class_masks && ps.all_kw_mult4 ? kMasksRows : kMasksStaged;
    DensePlan d = plan_pipe(&fake, ps, B, mixed, es, masks, ps.maxKW);
    int kind = 2;  // pipelined
    if (!d.ok) {
        d = plan_dense(&fake, ps, B, mixed, 4 * ps.VW, 32, masks);
        kind = 1;  // register kernel
    }
    if (!d.ok) kind = 0;  // per-row kernel
    int sp_S = 0, sp_per = 0;
    const bool sparse_ok = plan_sparse(&fake, ps, B, true, &sp_S, &sp_per);
    const int32_t vals[16] = {kind, d.n_groups_ub, d.S, d.per_split, d.WT, d.threads, d.depth, int32_t(d.smem),
                              d.table_words, d.stage_stride, d.cm_bulk, d.slots, sparse_ok ? sp_S : 0,
                              sparse_ok ? sp_per : 0, int32_t(kPartialSlots), d.ctas_per_sm};
    std::memcpy(out, vals, sizeof vals);
    return CFGZIP_OK;
}
