// Ahead-of-time instantiations of the fused probe kernel (the query is a descriptor interpreted at
// run time), result housekeeping kernels and the launch helpers used by the planner.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <unordered_map>

#include "sjq_fused_device.cuh"

namespace sjq {
namespace {

struct ClearParams {
    int64_t *sums;
    int64_t *counts;
    int64_t cells; // entries of sums / counts to zero
    int64_t *gkeys;
    int64_t gslots; // entries of gkeys to set to the empty marker
    int64_t *n_groups;
    int32_t *status;
    int32_t at_once; // the kernel behind this one may start at once (it waits on the device), else when the stores are out
};

// (every array starts on a 16-byte boundary; the odd last word is thread 0's)
__global__ void __launch_bounds__(256) clear_kernel(const ClearParams C)
{
    // Launched while the kernel before it still runs: that one, and all before it, first; then the pass may start, whose
    // reads of its tables rely on it.  (Filter and sum, 6 M rows, calls back to back: 18.4 -> 16.5 us; a call that nothing
    // runs before gains nothing.)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (C.at_once) asm volatile("griddepcontrol.launch_dependents;");
    const int64_t stride = (int64_t)blockDim.x * gridDim.x;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const longlong2 zero = make_longlong2(0, 0), empty = make_longlong2(kEmptyKey64, kEmptyKey64);
    for (int64_t i = t; i < C.cells / 2; i += stride) {
        reinterpret_cast<longlong2 *>(C.sums)[i] = zero;
        if (C.counts) reinterpret_cast<longlong2 *>(C.counts)[i] = zero;
    }
    for (int64_t i = t; i < C.gslots / 2; i += stride) reinterpret_cast<longlong2 *>(C.gkeys)[i] = empty;
    if (t == 0) {
        if (C.cells & 1) {
            C.sums[C.cells - 1] = 0;
            if (C.counts) C.counts[C.cells - 1] = 0;
        }
        if (C.gslots & 1) C.gkeys[C.gslots - 1] = kEmptyKey64;
        if (C.status) *C.status = 0;
        if (C.n_groups) *C.n_groups = 0;
    }
    if (!C.at_once) asm volatile("griddepcontrol.launch_dependents;");
}

struct CompactParams {
    const int64_t *gkeys;
    const longlong2 *cells; // {sum, count}
    int64_t dense_base; // indexed: cell number = key + dense_base
    int32_t indexed;    // the table is indexed by the key itself and has no key array
    int64_t ncells;     // indexed: all; otherwise the regular slots and the side slot after them
    int64_t tiles_per_block;
    int32_t ordered;            // indexed: the list comes out in key order
    unsigned int *block_counts; // ... from the used cells per block, counted by a kernel before; NULL: every block counts
    int64_t *keys, *sums, *counts;
    int64_t capacity;
    int64_t *n_groups;
    int32_t *status;
};

constexpr int kCompactThreads = 256;
constexpr int kCompactRounds = 8; // cells per thread and tile, all loaded before the first is used
constexpr int kCompactTile = kCompactThreads * kCompactRounds;
// Up to so many blocks each count the groups before their own themselves: a kernel for the counts costs a query over
// few rows 1 to 6 us (2 M rows, 1 % left, a list of 4000 groups: 15.4 us unordered, 20.0 with that kernel), the last
// of four blocks reads 96 KB more.
constexpr int kCompactAlone = 4;

// Cells of an indexed table that hold a group, [lo, hi), those of this thread.
__device__ __forceinline__ unsigned int used_cells(const CompactParams &C, int64_t lo, int64_t hi)
{
    unsigned int used = 0;
#pragma unroll 8
    for (int64_t i = lo + threadIdx.x; i < hi; i += kCompactThreads) used += C.cells[i].y != 0;
    return used;
}

__global__ void __launch_bounds__(kCompactThreads) compact_count_kernel(const CompactParams C)
{
    asm volatile("griddepcontrol.wait;" ::: "memory"); // the pass
    asm volatile("griddepcontrol.launch_dependents;"); // the listing may start and wait for the counts on the device
    const int64_t lo = (int64_t)blockIdx.x * C.tiles_per_block * kCompactTile;
    int64_t hi = lo + C.tiles_per_block * kCompactTile;
    hi = hi < C.ncells ? hi : C.ncells;
    unsigned int used = __reduce_add_sync(0xffffffffu, used_cells(C, lo, hi));
    __shared__ unsigned int part[kCompactThreads / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = used;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kCompactThreads / 32; ++w) used += part[w];
        C.block_counts[blockIdx.x] = used;
    }
}

// Group table -> list of (key, sum, count).  A block owns consecutive tiles of cells; a warp takes 256 consecutive
// cells of a tile.  The place of a block's groups is the number of groups before it (an indexed table: the list comes
// out in ascending key order), or is drawn from the common counter, once per tile.
// (Four blocks per SM at 64 registers: merge of eight lists of 200,000 with its sort 106.5 us, 107.9 with 80 registers.)
__global__ void __launch_bounds__(kCompactThreads, 4) compact_kernel(const CompactParams C)
{
    __shared__ unsigned int part[kCompactThreads / 32];
    __shared__ long long draw;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory"); // the pass, and the counts where a kernel forms them
    long long place = 0;
    if (C.ordered) {
        unsigned int before = 0;
        if (C.block_counts) {
            for (int b = threadIdx.x; b < (int)blockIdx.x; b += kCompactThreads) before += C.block_counts[b];
        } else {
            before = used_cells(C, 0, (int64_t)blockIdx.x * C.tiles_per_block * kCompactTile);
        }
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane == 0) part[warp] = before;
        __syncthreads();
        for (int w = 0; w < kCompactThreads / 32; ++w) place += part[w];
        __syncthreads();
    }
    const int64_t lo = (int64_t)blockIdx.x * C.tiles_per_block * kCompactTile;
    int64_t hi = lo + C.tiles_per_block * kCompactTile;
    hi = hi < C.ncells ? hi : C.ncells;
    for (int64_t tile = lo; tile < hi; tile += kCompactTile) {
        const int64_t first = tile + warp * (32 * kCompactRounds) + lane;
        longlong2 cell[kCompactRounds];
        long long key[kCompactRounds];
        unsigned int lanes[kCompactRounds], mine = 0;
#pragma unroll
        for (int r = 0; r < kCompactRounds; ++r) {
            const int64_t i = first + 32 * r;
            cell[r] = make_longlong2(0, 0);
            key[r] = kEmptyKey64;
            if (i < hi) {
                cell[r] = C.cells[i];
                key[r] = C.indexed ? i - C.dense_base : i == C.ncells - 1 ? kEmptyKey64 : C.gkeys[i];
            }
        }
#pragma unroll
        for (int r = 0; r < kCompactRounds; ++r) {
            const int64_t i = first + 32 * r;
            // a claimed slot holds a group whatever its count (merged lists may carry zeros); the side slot and the
            // cells of an indexed table do when a row was counted there
            const bool used = i < hi && (C.indexed || i == C.ncells - 1 ? cell[r].y != 0 : key[r] != kEmptyKey64);
            lanes[r] = __ballot_sync(0xffffffffu, used);
            mine += __popc(lanes[r]);
        }
        if (lane == 0) part[warp] = mine;
        __syncthreads();
        unsigned int before = 0, total = 0;
        for (int w = 0; w < kCompactThreads / 32; ++w) {
            before += w < warp ? part[w] : 0u;
            total += part[w];
        }
        if (!C.ordered) {
            if (threadIdx.x == 0)
                draw = (long long)atomicAdd(reinterpret_cast<unsigned long long *>(C.n_groups), (unsigned long long)total);
            __syncthreads();
            place = draw;
        }
        long long at = place + before;
#pragma unroll
        for (int r = 0; r < kCompactRounds; ++r) {
            if ((lanes[r] >> lane) & 1u) {
                const long long pos = at + __popc(lanes[r] & ((1u << lane) - 1u));
                if (pos < C.capacity) {
                    C.keys[pos] = key[r];
                    C.sums[pos] = cell[r].x;
                    C.counts[pos] = cell[r].y;
                } else {
                    set_status(C.status, SJQ_ERR_GROUP_OVERFLOW);
                }
            }
            at += __popc(lanes[r]);
        }
        place += total;
        __syncthreads(); // the shared words are written again for the next tile
    }
    if (C.ordered && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *C.n_groups = place;
}

struct MergeParams {
    const int64_t *keys, *sums, *counts; // the lists to merge, n entries
    int64_t n;
    int64_t *gkeys, *cells; // group table
    uint64_t gmask;
    int32_t *status;
};

// Lists of (key, sum, count) -> group table: one insert-or-find and two adds per entry.  Bound by the latency of the
// dependent steps (entry, slot, claim of a free slot, adds), hence all the warps an SM holds; the first entry is
// requested while the table is still being cleared, every other one before the probe of the one before it (merge of
// eight lists of 200,000 with its sort 110 -> 108 us, the kernel alone 33).  Four
// entries per thread, each step for all of them before the next: 66 us instead of 33 (claims and probes diverge, so
// that they come one after the other all the same, on half the warps).
__global__ void __launch_bounds__(256, 8) merge_kernel(const MergeParams M)
{
    const int64_t stride = (int64_t)blockDim.x * gridDim.x;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t key = 0, sum = 0, count = 0;
    if (first < M.n) key = M.keys[first], sum = M.sums[first], count = M.counts[first];
    asm volatile("griddepcontrol.wait;" ::: "memory"); // the cleared table
    for (int64_t i = first; i - (threadIdx.x & 31) < M.n; i += stride) { // whole warps stay together
        int64_t next_key = 0, next_sum = 0, next_count = 0;
        if (i + stride < M.n) next_key = M.keys[i + stride], next_sum = M.sums[i + stride], next_count = M.counts[i + stride];
        uint64_t cell = ~0ull;
        if (i < M.n) cell = group_cell(M.gkeys, M.gmask, M.status, key);
        unsigned long long *cells = reinterpret_cast<unsigned long long *>(M.cells);
        if (M.gmask < 0xFFFFFFFEull) {
            add_pairs<false>(cells, (uint32_t)cell, (uint64_t)sum, (uint64_t)count, cell != ~0ull);
        } else if (cell != ~0ull) {
            atomicAdd(cells + 2 * cell, (unsigned long long)sum);
            atomicAdd(cells + 2 * cell + 1, (unsigned long long)count);
        }
        key = next_key, sum = next_sum, count = next_count;
    }
}

struct SampleParams {
    const void *col[SJQ_MAX_PREDS];
    DPred preds[SJQ_MAX_PREDS];
    int32_t npreds;
    int64_t n;       // rows of the table
    int64_t groups;  // sampled groups of four consecutive rows
    int64_t stride;  // rows between the starts of two sampled groups (a multiple of 4)
    unsigned long long *counts; // [0] rows sampled, [1 + p] rows among them passing predicate p
};

// Every predicate evaluated on its own over an evenly spaced sample of the table: the marginal pass
// fractions the planner orders the stages by.  One 16- or 32-byte load per predicate and group.
__global__ void __launch_bounds__(256) sample_kernel(const __grid_constant__ SampleParams S)
{
    __shared__ unsigned int block_counts[SJQ_MAX_PREDS + 1];
    if (threadIdx.x <= SJQ_MAX_PREDS) block_counts[threadIdx.x] = 0;
    __syncthreads();
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < S.groups) {
        const int64_t r0 = g * S.stride;
        const int rows = (int)(S.n - r0 < 4 ? S.n - r0 : 4);
        atomicAdd(&block_counts[0], (unsigned int)rows);
        for (int p = 0; p < S.npreds; ++p) {
            const DPred &d = S.preds[p];
            unsigned int pass = 0;
            for (int r = 0; r < rows; ++r)
                pass += d.is64 ? pred_eval<int64_t>(d, static_cast<const int64_t *>(S.col[p])[r0 + r])
                               : pred_eval<int32_t>(d, static_cast<const int32_t *>(S.col[p])[r0 + r]);
            if (pass) atomicAdd(&block_counts[1 + p], pass);
        }
    }
    __syncthreads();
    if (threadIdx.x <= S.npreds && block_counts[threadIdx.x])
        atomicAdd(&S.counts[threadIdx.x], (unsigned long long)block_counts[threadIdx.x]);
}

const void *pick_kernel(int agg, bool mul, int form, bool few)
{
    const auto of = [few](fused_few_fn little, fused_fn any) {
        return few ? reinterpret_cast<const void *>(little) : reinterpret_cast<const void *>(any);
    };
    switch (agg) {
    case AGG_SCALAR: return of(fused_few_scalar(mul, form), fused_variant_scalar(mul, form));
    case AGG_SMEM: return of(fused_few_smem(mul, form), fused_variant_smem(mul, form));
    case AGG_GLOBAL: return of(fused_few_global(mul, form), fused_variant_global(mul, form));
    default: return of(fused_few_hash(mul, form), fused_variant_hash(mul, form));
    }
}

} // namespace

// ---- launch helpers used by the planner (sjq_run.cu) ----------------------

// Shared-memory opt-in and occupancy of a kernel variant; both answers are remembered per device, so a
// repeated query costs two map look-ups instead of two runtime calls.
namespace {
std::mutex g_occ_mutex;
std::unordered_map<uint64_t, int> g_occupancy; // (device, variant, block, smem) -> blocks per SM
std::unordered_map<uint32_t, int> g_opted;     // (device, variant) -> largest smem opted in for
} // namespace

int fused_cache_clear()
{
    std::lock_guard<std::mutex> lock(g_occ_mutex);
    const int n = (int)g_occupancy.size();
    g_occupancy.clear(); // the shared-memory opt-in of a kernel is a property of the function: kept
    return n;
}

sjq_status fused_occupancy(int agg, bool mul, int form, int nstages, int block, size_t smem, int *ctas_per_sm)
{
    const bool few = nstages <= kFewStages;
    std::mutex &mutex = g_occ_mutex;
    std::unordered_map<uint64_t, int> &occupancy = g_occupancy;
    std::unordered_map<uint32_t, int> &opted = g_opted;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SJQ_ERR_CUDA;
    const uint32_t variant = (uint32_t)(agg * 32 + form * 4 + (mul ? 2 : 0) + (few ? 1 : 0));
    const uint32_t fkey = (uint32_t)dev * 128u + variant;
    const uint64_t okey = ((uint64_t)fkey << 40) | ((uint64_t)block << 24) | (uint64_t)(smem & 0xFFFFFF);
    std::lock_guard<std::mutex> lock(mutex);
    const void *fn = pick_kernel(agg, mul, form, few);
    auto o = opted.find(fkey);
    if (o == opted.end() || o->second < (int)smem) {
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
            (void)cudaGetLastError();
            return SJQ_ERR_CUDA;
        }
        opted[fkey] = (int)smem;
    }
    auto it = occupancy.find(okey);
    if (it == occupancy.end()) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, block, smem) != cudaSuccess) {
            (void)cudaGetLastError();
            return SJQ_ERR_CUDA;
        }
        it = occupancy.emplace(okey, n).first;
    }
    *ctas_per_sm = it->second;
    return SJQ_OK;
}

sjq_status fused_launch(int agg, bool mul, int form, int grid, int block, size_t smem, bool behind,
                        const RunParams &P, cudaStream_t stream)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = behind ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    void *args[1];
    RunParamsFew little;
    if (P.nstages <= kFewStages) {
        std::memcpy(little.st, P.st, (size_t)P.nstages * sizeof(DStage));
        static_cast<RunCore &>(little) = P;
        args[0] = &little;
    } else {
        args[0] = const_cast<RunParams *>(&P);
    }
    if (cudaLaunchKernelExC(&cfg, pick_kernel(agg, mul, form, P.nstages <= kFewStages), args) != cudaSuccess) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    return SJQ_OK;
}

// `at_once`: the kernel behind starts beside a clear of so many blocks (of 256 threads) at most.
// Launched while the kernel before it still runs, a clear's blocks wait in the SMs: one per SM at most, which leaves other
// streams their room beside a long pass.  (Another stream's two joins over 2 M rows, a call, while filter and sum over 300 M
// rows and the clear of 8 M groups take turns: 206 us with eight waiting blocks per SM, 87 to 92 so, 99 to 103 with none
// launched early.)  The clear of a list's cells is held to that many blocks up to 32 MB (back to back, in its turn and so:
// a hundred thousand groups, 100 thousand rows 10.0 and 9.5 us; merge of eight lists of 58 thousand 22.2 and 21.8).  A dense
// result, which the pass adds to at once, needs all its blocks, and from half a block per SM on its clear waits for its turn
// (2 M rows, 5 thousand groups 6.65 in its turn and 6.35 early, 30 thousand 6.75 and 6.9, 60 thousand 6.75 and 7.05; a
// million 8.9 and, with one block per SM, 13.2; eight million, few rows, 28.7 and 39.2).
constexpr size_t kEarlyList = (size_t)32 << 20;
sjq_status clear_launch(int64_t *sums, int64_t *counts, int64_t cells, int64_t *gkeys, int64_t gslots,
                        int64_t *n_groups, int32_t *status, int at_once, int sm_count, cudaStream_t stream)
{
    const int64_t work = (cells > gslots ? cells : gslots) / 2;
    int64_t blocks = (work + 255) / 256;
    if (blocks > (int64_t)sm_count * 8) blocks = (int64_t)sm_count * 8;
    if (blocks < 1) blocks = 1;
    const ClearParams C{sums, counts, cells, gkeys, gslots, n_groups, status, blocks <= at_once ? 1 : 0};
    const bool list = gkeys != nullptr;
    if (list && blocks > sm_count && ((size_t)cells + (size_t)gslots) * 8 <= kEarlyList) blocks = sm_count;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = (list ? blocks : 2 * blocks) <= sm_count ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, clear_kernel, C) == cudaSuccess ? SJQ_OK : SJQ_ERR_CUDA;
}

// Enqueue the sampling kernel: `counts` (device, SJQ_MAX_PREDS + 1 words) is cleared first.
sjq_status sample_launch(const sjq_col *fact, const DPred *preds, int npreds, int64_t n, unsigned long long *counts,
                         cudaStream_t stream)
{
    if (cudaMemsetAsync(counts, 0, (SJQ_MAX_PREDS + 1) * sizeof(unsigned long long), stream) != cudaSuccess)
        return SJQ_ERR_CUDA;
    if (n <= 0 || npreds <= 0) return SJQ_OK;
    SampleParams S{};
    for (int p = 0; p < npreds; ++p) {
        S.col[p] = fact[preds[p].col].data;
        S.preds[p] = preds[p];
    }
    S.npreds = npreds;
    S.n = n;
    S.counts = counts;
    const int64_t quads = (n + 3) / 4;
    const int64_t want = (int64_t)1 << 16; // 65 536 groups of four rows
    S.groups = quads < want ? quads : want;
    S.stride = 4 * (quads / S.groups);
    sample_kernel<<<(int)((S.groups + 255) / 256), 256, 0, stream>>>(S);
    return cudaGetLastError() == cudaSuccess ? SJQ_OK : SJQ_ERR_CUDA;
}

sjq_status merge_launch(const int64_t *keys, const int64_t *sums, const int64_t *counts, int64_t n, int64_t *gkeys,
                        int64_t *cells, uint64_t gmask, int32_t *status, int sm_count, cudaStream_t stream)
{
    if (n <= 0) return SJQ_OK;
    MergeParams M{keys, sums, counts, n, gkeys, cells, gmask, status};
    const int64_t blocks = std::min((n + 255) / 256, (int64_t)sm_count * 8);
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization; // behind the clear, for which it waits on the device
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, merge_kernel, M) == cudaSuccess ? SJQ_OK : SJQ_ERR_CUDA;
}

// gslots: regular slots of the hash table (a side slot follows), or the cells of an indexed table.  `block_counts`
// (device, one word per 2048 cells): an indexed table is listed in key order; NULL: in no order.  `beside`: directly
// behind the fused kernel, which lets its successor start while it runs, so many blocks at most may wait beside it.
sjq_status compact_launch(const int64_t *gkeys, const int64_t *cells, int64_t gslots, bool indexed,
                          int64_t dense_base, unsigned int *block_counts, int64_t *keys, int64_t *sums,
                          int64_t *counts, int64_t capacity, int64_t *n_groups, int32_t *status, int sm_count,
                          int beside, cudaStream_t stream, int *launches)
{
    const int64_t ncells = indexed ? gslots : gslots + 1;
    const int64_t tiles = (ncells + kCompactTile - 1) / kCompactTile;
    const int64_t per = (tiles + (int64_t)sm_count * 8 - 1) / ((int64_t)sm_count * 8);
    const int blocks = (int)((tiles + per - 1) / per);
    const bool counted = block_counts && blocks > kCompactAlone;
    CompactParams C{gkeys, reinterpret_cast<const longlong2 *>(cells), dense_base, indexed ? 1 : 0, ncells, per,
                    block_counts ? 1 : 0, counted ? block_counts : nullptr, keys, sums, counts, capacity, n_groups, status};
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = blocks <= beside ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kCompactThreads);
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (counted) {
        if (cudaLaunchKernelEx(&cfg, compact_count_kernel, C) != cudaSuccess) return SJQ_ERR_CUDA;
        ++*launches;
        attr.val.programmaticStreamSerializationAllowed = 1; // the listing behind the counts
    }
    ++*launches;
    return cudaLaunchKernelEx(&cfg, compact_kernel, C) == cudaSuccess ? SJQ_OK : SJQ_ERR_CUDA;
}

} // namespace sjq
