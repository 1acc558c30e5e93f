// Dimension-table planning and build kernels.
//
// Section 3.3 of the paper: dense primary keys allow a directly indexed map
// whose build is a race-free direct store and whose probe is one load; the
// filter and the gathered attribute are fused into one narrow code per key
// with a reserved all-ones sentinel for "filtered out".  Sparse keys fall back
// to an open-addressing table populated with atomicCAS.  Section 4.3.1: the
// key range is verified at run time and the packed or unpacked form chosen.
#include <algorithm>
#include <mutex>
#include <new>
#include <type_traits>
#include <utility>

#include "sjq_internal.h"

namespace sjq {

namespace {

constexpr int kMaxDimCols = 32;

// A launch works on up to kBatchDims dimensions (and their filters, together at most kBatchPreds): the scans, the
// fills and the builds of a query's tables are one launch each.  A block belongs to one dimension; its threads take
// four consecutive rows at two places at a time (one where 64-bit values fill the registers), so that every column is
// read with 128-bit loads and six of them are in flight per thread before the first is used.  What bounds these
// kernels: latency for the small dimensions (2,556 to 200,000 rows), instructions as much as the columns' bytes for
// those of millions; so the code for 32-bit keys and payloads keeps to 32-bit arithmetic.
constexpr int kBatchDims = 8;
constexpr int kBatchPreds = 16;
constexpr int kFillThreads = 256;
constexpr int kBuildThreads = 256;
constexpr int kScanThreads = 512;

struct DimRows {
    int64_t n;
    const void *key;
    const void *pay[SJQ_MAX_PAYLOADS];
    int32_t npayload;
    int32_t pred0, npreds; // its conjunction in the launch's list
    uint32_t block0, blocks;
    uint8_t key64, pay64[SJQ_MAX_PAYLOADS];
};

struct DimFilters {
    DPred d[kBatchPreds];
    const void *col[kBatchPreds];
};

// Four consecutive values of a column as T (a 32-bit column may be read as 64-bit values, not the other way round).
// Evict first: the columns pass once and should not push the table that is being built out of the L2 (skewed keys asked
// once, 128 MB of columns beside an 84 MB table: 289 -> 279 us in all).
template <typename T>
__device__ __forceinline__ void load4(const void *col, bool is64, int64_t r, int rows, T *v)
{
    if (rows == 4) {
        if (sizeof(T) == 8 && is64) {
            const longlong2 a = __ldcs(static_cast<const longlong2 *>(col) + r / 2);
            const longlong2 b = __ldcs(static_cast<const longlong2 *>(col) + r / 2 + 1);
            v[0] = (T)a.x, v[1] = (T)a.y, v[2] = (T)b.x, v[3] = (T)b.y;
        } else {
            const int4 a = __ldcs(static_cast<const int4 *>(col) + r / 4);
            v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = k < rows ? (T)load_cell(col, sizeof(T) == 8 && is64, r + k) : (T)0;
}

// The rows a thread has in hand, Q groups of four: keys of type K and up to N payloads of type V, and which pass the
// filter.  Usual keeps to the tables of most dimensions: at most one payload, of 32 bits.
template <typename K, typename V, int N, int Q>
struct RowSet {
    static constexpr int kPayloads = N, kQuads = Q, kRows = 4 * Q;
    typedef K Key;
    typedef V Payload;
    K key[kRows];
    V pay[N][kRows];
    uint32_t m;
};
template <typename K>
using Usual = RowSet<K, int32_t, 1, 2>;
template <typename K>
using Wide = RowSet<K, int64_t, SJQ_MAX_PAYLOADS, 1>;
__host__ __device__ inline bool usual_payloads(const DimRows &D) { return D.npayload == 0 || (D.npayload == 1 && !D.pay64[0]); }

template <typename T>
__device__ __forceinline__ uint32_t filter4(const DPred &d, const T *v)
{
    uint32_t pass = 0;
    if (d.nset) {
        for (int i = 0; i < d.nset; ++i) {
            const int64_t lit = d.set[i];
#pragma unroll
            for (int k = 0; k < 4; ++k) pass |= (uint32_t)((int64_t)v[k] == lit) << k;
        }
        return pass;
    }
    if (sizeof(T) == 4) {
        const uint32_t lo = (uint32_t)d.lo32, width = (uint32_t)d.hi32 - lo;
        if (!d.never) {
#pragma unroll
            for (int k = 0; k < 4; ++k) pass |= (uint32_t)((uint32_t)v[k] - lo <= width) << k;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) pass |= (uint32_t)(((int64_t)v[k] >= d.lo) & ((int64_t)v[k] <= d.hi)) << k;
    }
    return d.neg ? ~pass : pass;
}

// Rows r .. r + 3 and r + apart .. r + apart + 3 (those below D.n).  The first filter's column is requested with the
// others; further filters are read one after the other.
template <typename Set>
__device__ __forceinline__ void read_rows(const DimRows &D, const DimFilters &F, int64_t r, int64_t apart, Set &R)
{
    typedef typename Set::Key K;
    typedef typename Set::Payload V;
    constexpr int kDimQuads = Set::kQuads;
    R.m = 0;
    int first[Set::kRows];
    const bool ahead = D.npreds > 0 && !F.d[D.pred0].is64;
#pragma unroll
    for (int q = 0; q < kDimQuads; ++q) {
        const int64_t at = r + q * apart, left = D.n - at;
        const int rows = left >= 4 ? 4 : left > 0 ? (int)left : 0;
        R.m |= ((1u << rows) - 1u) << (4 * q);
        if (!rows) continue;
        load4<K>(D.key, D.key64, at, rows, &R.key[4 * q]);
        if (ahead) load4<int>(F.col[D.pred0], false, at, rows, &first[4 * q]);
#pragma unroll
        for (int i = 0; i < Set::kPayloads; ++i)
            if (i < D.npayload) load4<V>(D.pay[i], D.pay64[i], at, rows, &R.pay[i][4 * q]);
    }
    if (ahead) {
#pragma unroll
        for (int q = 0; q < kDimQuads; ++q)
            if ((R.m >> (4 * q)) & 0xFu) R.m &= ~(0xFu << (4 * q)) | (filter4<int>(F.d[D.pred0], &first[4 * q]) & 0xFu) << (4 * q);
    }
    for (int p = D.pred0 + (ahead ? 1 : 0); p < D.pred0 + D.npreds; ++p) {
        const DPred &d = F.d[p];
#pragma unroll
        for (int q = 0; q < kDimQuads; ++q) {
            const int64_t at = r + q * apart, left = D.n - at;
            if (left <= 0) continue;
            int64_t v[4];
            load4<int64_t>(F.col[p], d.is64, at, left >= 4 ? 4 : (int)left, v);
            int v32[4] = {(int)v[0], (int)v[1], (int)v[2], (int)v[3]};
            const uint32_t pass = d.is64 ? filter4<int64_t>(d, v) : filter4<int>(d, v32);
            R.m &= ~(0xFu << (4 * q)) | (pass & 0xFu) << (4 * q);
        }
    }
}

// (a launch's tasks in the order of their blocks)
struct BuildTask;
struct FillTask;
__device__ __forceinline__ uint32_t first_block(const DimRows &t) { return t.block0; }
__device__ __forceinline__ uint32_t first_block(const BuildTask &t);
__device__ __forceinline__ uint32_t first_block(const FillTask &t);

template <typename Task>
__device__ __forceinline__ int task_of_block(const Task *tasks, int n)
{
    int t = 0;
    while (t + 1 < n && blockIdx.x >= first_block(tasks[t + 1])) ++t;
    return t;
}

__device__ __forceinline__ unsigned long long ordered(int64_t v) { return (unsigned long long)v ^ 0x8000000000000000ull; }
__device__ __forceinline__ int64_t unordered(unsigned long long v) { return (int64_t)(v ^ 0x8000000000000000ull); }

// Statistics of a dimension, kScratchWords words of scratch that start as zeros: while the blocks add to them, words
// 4 i, each in a sector of its own, hold i = 0 the largest of ~ordered(key) (so the smallest key), 1 of ordered(key),
// 2 the passing rows, 3..6 the payloads' like 0 and 1, 7 the blocks done; the block that comes last leaves kmin, kmax,
// count, p0min, p0max, p1min, p1max, 0 in words 0..7.
constexpr int kScratchWords = 32;
static_assert(kScratchWords * 8 == SJQ_PLAN_SCRATCH_BYTES, "one dimension's statistics fill the scratch of a plan");

struct ScanParams {
    DimRows dim[kBatchDims];
    DimFilters filters;
    int32_t ndims;
    unsigned long long *scratch;
    int64_t *host[kBatchDims]; // page-locked, eight words each, or NULL: the statistics stay in the scratch
};

constexpr int kExtremes = 2 + 2 * SJQ_MAX_PAYLOADS; // [min, max] of the key and of each payload

// Extremes (as ~ordered(min), ordered(max)) and count of the passing rows that this thread owns.
template <typename Set>
__device__ __forceinline__ void scan_rows(const DimRows &D, const DimFilters &F, unsigned long long (&ext)[kExtremes], unsigned int &cnt)
{
    typedef typename Set::Key K;
    typedef typename Set::Payload V;
    constexpr int kPayloads = Set::kPayloads;
    constexpr K kmost = sizeof(K) == 8 ? (K)INT64_MAX : (K)INT32_MAX;
    constexpr V vmost = sizeof(V) == 8 ? (V)INT64_MAX : (V)INT32_MAX;
    K kmin = kmost, kmax = -kmost - 1;
    V pmin[kPayloads], pmax[kPayloads];
#pragma unroll
    for (int i = 0; i < kPayloads; ++i) pmin[i] = vmost, pmax[i] = -vmost - 1;
    const int64_t apart = 4 * (int64_t)D.blocks * kScanThreads;
    for (int64_t r = 4 * ((int64_t)(blockIdx.x - D.block0) * kScanThreads + threadIdx.x); r < D.n; r += Set::kQuads * apart) {
        Set R;
        read_rows(D, F, r, apart, R);
        cnt += __popc(R.m);
#pragma unroll
        for (int k = 0; k < Set::kRows; ++k) {
            const bool on = (R.m >> k) & 1u;
            const K lo = on ? R.key[k] : kmost, hi = on ? R.key[k] : (K)(-kmost - 1);
            kmin = lo < kmin ? lo : kmin;
            kmax = hi > kmax ? hi : kmax;
#pragma unroll
            for (int i = 0; i < kPayloads; ++i) {
                if (i >= D.npayload) continue;
                const V plo = on ? R.pay[i][k] : vmost, phi = on ? R.pay[i][k] : (V)(-vmost - 1);
                pmin[i] = plo < pmin[i] ? plo : pmin[i];
                pmax[i] = phi > pmax[i] ? phi : pmax[i];
            }
        }
    }
    if (cnt == 0) return;
    ext[0] = ~ordered(kmin);
    ext[1] = ordered(kmax);
#pragma unroll
    for (int i = 0; i < kPayloads; ++i) {
        if (i >= D.npayload) continue;
        ext[2 + 2 * i] = ~ordered(pmin[i]);
        ext[3 + 2 * i] = ordered(pmax[i]);
    }
}

__global__ void __launch_bounds__(kScanThreads, 2) plan_scan_kernel(const __grid_constant__ ScanParams P)
{
    const int which = task_of_block(P.dim, P.ndims);
    const DimRows &D = P.dim[which];
    unsigned long long *const scratch = P.scratch + which * kScratchWords;
    unsigned long long ext[kExtremes];
#pragma unroll
    for (int i = 0; i < kExtremes; ++i) ext[i] = 0;
    unsigned int cnt = 0;
    if (!usual_payloads(D)) scan_rows<Wide<int64_t>>(D, P.filters, ext, cnt);
    else if (D.key64) scan_rows<Usual<int64_t>>(D, P.filters, ext, cnt);
    else scan_rows<Usual<int32_t>>(D, P.filters, ext, cnt);
    // one set of atomics per block: they all land on the same seven words
    __shared__ unsigned long long part[kScanThreads / 32][kExtremes + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cnt = __reduce_add_sync(0xffffffffu, cnt);
#pragma unroll
    for (int i = 0; i < kExtremes; ++i) {
        if (i >= 2 + 2 * D.npayload) continue;
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, ext[i], o);
            ext[i] = v > ext[i] ? v : ext[i];
        }
    }
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < kExtremes; ++i) part[warp][i] = ext[i];
        part[warp][kExtremes] = cnt;
    }
    __syncthreads();
    if (warp <= kExtremes) { // one warp per word
        unsigned long long v = lane < kScanThreads / 32 ? part[lane][warp] : 0ull;
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long t = __shfl_xor_sync(0xffffffffu, v, o);
            v = warp == kExtremes ? v + t : t > v ? t : v;
        }
        if (lane == 0) {
            if (warp == kExtremes) atomicAdd(&scratch[4 * 2], v);
            else if (warp < 2 + 2 * D.npayload) atomicMax(&scratch[4 * (warp < 2 ? warp : warp + 1)], v);
            __threadfence();
        }
    }
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&scratch[4 * 7], 1ull) == D.blocks - 1;
    __syncthreads();
    if (last && warp == 0) {
        const int i = lane & 7;
        const unsigned long long v = i < 7 ? atomicAdd(&scratch[4 * i], 0ull) : 0ull;
        const int64_t stat = i == 2 || i == 7 ? (int64_t)v : (i == 0 || i == 3 || i == 5) ? unordered(~v) : unordered(v);
        __syncwarp();
        if (lane < 8) {
            scratch[i] = (unsigned long long)stat;
            if (P.host[which]) P.host[which][i] = stat;
        }
    }
}

struct BuildTask {
    DimRows rows;
    int32_t kind;
    int32_t code_bits;
    int32_t usual; // no payload or a 32-bit one, slot indexes of a direct table below 2^32
    int64_t kmin;
    uint64_t span;  // direct
    uint32_t buckets; // hash: number of buckets
    int32_t bucket_k; // hash: keys per bucket
    int32_t code_off; // hash: byte offset of the codes inside a bucket
    int64_t pay_min[SJQ_MAX_PAYLOADS], pay_max[SJQ_MAX_PAYLOADS];
    int32_t pay_bits[SJQ_MAX_PAYLOADS];
    void *slots;
    unsigned int *filter; // presence bitmap words (hash: indexed by a hash of the key; direct with payloads: by slot)
    uint32_t fmask;       // hash: filter bits - 1
    long long expect_full; // >= 0: the layout promises that every key of the range is present: so many rows are stored
    unsigned long long *header; // [0] rows inserted, [1] blocks done (only with such a promise)
    int32_t *status;
};

__device__ __forceinline__ uint32_t first_block(const BuildTask &t) { return t.rows.block0; }

struct BuildParams {
    BuildTask task[kBatchDims];
    DimFilters filters;
    int32_t ntasks;
};

// One launch prepares the memory of the tables: the header counters and the presence bitmap to zero, the slot array
// to its empty pattern (bitmap: zeros; packed codes: all ones; open addressing: the empty key in every word).
// All regions start on 16-byte boundaries and are padded to a multiple of 16 bytes by the layout.
constexpr int kFillTile = 4 * kFillThreads; // 16-byte units per block and step

struct FillTask {
    uint4 *at;
    uint64_t units; // of 16 bytes
    uint4 pattern;
    uint32_t block0, blocks;
};

__device__ __forceinline__ uint32_t first_block(const FillTask &t) { return t.block0; }

struct FillParams {
    FillTask task[3 * kBatchDims];
    int32_t *clear_status[kBatchDims]; // NULL: left as it is
    int32_t ntasks;
};

__global__ void __launch_bounds__(kFillThreads) table_init_kernel(const __grid_constant__ FillParams P)
{
    cudaTriggerProgrammaticLaunchCompletion(); // the build is launched behind and waits for this kernel on the device
    if (blockIdx.x == 0 && threadIdx.x < kBatchDims && P.clear_status[threadIdx.x]) *P.clear_status[threadIdx.x] = 0;
    const FillTask &T = P.task[task_of_block(P.task, P.ntasks)];
    for (uint64_t base = (uint64_t)(blockIdx.x - T.block0) * kFillTile; base < T.units; base += (uint64_t)T.blocks * kFillTile) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint64_t i = base + k * kFillThreads + threadIdx.x;
            if (i < T.units) T.at[i] = T.pattern;
        }
    }
}

template <typename Set>
__device__ __forceinline__ bool pack_code(const BuildTask &B, const Set &R, int k, uint64_t *code)
{
    uint64_t c = 0;
    int shift = 0;
#pragma unroll
    for (int i = 0; i < Set::kPayloads; ++i) {
        if (i >= B.rows.npayload) continue;
        const int64_t v = R.pay[i][k];
        if (v < B.pay_min[i] || v > B.pay_max[i]) return false;
        c |= ((uint64_t)v - (uint64_t)B.pay_min[i]) << shift;
        shift += B.pay_bits[i];
    }
    *code = c;
    return true;
}
// (one 32-bit payload whose layout's bounds are 32-bit values)
template <typename Set>
__device__ __forceinline__ bool pack_code(const BuildTask &B, const Set &R, int k, uint32_t *code)
{
    *code = B.rows.npayload ? (uint32_t)R.pay[0][k] - (uint32_t)B.pay_min[0] : 0u;
    return *code <= (uint32_t)B.pay_max[0] - (uint32_t)B.pay_min[0];
}

// Set one bit per row of the warp in a bitmap and report a bit that two rows set.  All lanes call it.  A dimension
// that lists its keys in ascending order, as most do, gives a warp 128 neighbouring bits: the rows of a thread that
// share a word are joined first, then the words that several threads share (up to eight of them), so that five adds
// leave the warp instead of a hundred.
template <typename I>
__device__ __forceinline__ void set_bits(unsigned int *bits, const I *idx, uint32_t m, int32_t *status)
{
    const int lane = threadIdx.x & 31;
    I word = 0;
    unsigned int mine = 0, rows = 0, seen[4] = {0, 0, 0, 0};
    bool dup = false;
    // (nothing waits for an atomic's answer before the last of them is on its way)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!((m >> k) & 1u)) continue;
        const unsigned int bit = 1u << (idx[k] & 31);
        if (!rows) word = idx[k] >> 5;
        if (idx[k] >> 5 == word) {
            mine |= bit;
            ++rows;
        } else {
            seen[k] = atomicOr(bits + (idx[k] >> 5), bit);
        }
    }
    unsigned int joined = 0; // leader of a word that several threads share: their bits
    unsigned int pending = __ballot_sync(0xffffffffu, rows != 0);
    for (int it = 0; it < 8 && pending; ++it) {
        const int leader = __ffs((int)pending) - 1;
        const I w = __shfl_sync(0xffffffffu, word, leader);
        const bool in = rows && word == w;
        const unsigned int same = __ballot_sync(0xffffffffu, in);
        if (it == 0 && __popc(same) == 1 && __popc(pending) > 1) break; // scattered keys: every lane for itself
        const unsigned int all = __reduce_or_sync(0xffffffffu, in ? mine : 0u);
        const unsigned int n = __reduce_add_sync(0xffffffffu, in ? rows : 0u);
        if (lane == leader) {
            joined = all;
            dup = (int)n != __popc(all);
        }
        pending &= ~same;
    }
    if ((pending >> lane) & 1u) {
        joined = mine;
        dup = (int)rows != __popc(mine);
    }
    if (joined) dup |= (atomicOr(bits + word, joined) & joined) != 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) dup |= (seen[k] >> (idx[k] & 31)) & 1u;
    if (dup) set_status(status, SJQ_ERR_DUP_KEY);
}

// The packed codes of a thread's rows into a direct table.  A table with a presence bitmap finds repeated keys there;
// without one (wide codes only) the store itself tells, since a code is never all ones, which is what a slot starts as.
template <typename I, typename C>
__device__ __forceinline__ void store_codes(const BuildTask &B, const I *idx, const C *code, uint32_t m)
{
    const int bits = B.code_bits;
    if (bits < 8) {
        // several codes share a word that starts as all ones: clear this code's zero bits, the rows of a thread that
        // share a word at once (the keys are unique, so no two rows touch the same bits)
        const unsigned int per = 32u / (unsigned int)bits, low = (1u << bits) - 1u;
        unsigned int *const words = static_cast<unsigned int *>(B.slots);
        const int log_per = bits == 2 ? 4 : 3;
        I word = ~(I)0; // no slot's word
        unsigned int keep = ~0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (!((m >> k) & 1u)) continue;
            const I w = idx[k] >> log_per;
            const unsigned int sh = ((unsigned int)idx[k] & (per - 1u)) * (unsigned int)bits;
            if (w != word) {
                if (word != ~(I)0) atomicAnd(words + word, keep);
                word = w;
                keep = ~0u;
            }
            keep &= ~(low << sh) | ((unsigned int)code[k] << sh);
        }
        if (word != ~(I)0) atomicAnd(words + word, keep);
        return;
    }
    bool dup = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!((m >> k) & 1u)) continue;
        const uint64_t i = idx[k], c = code[k];
        if (B.filter) {
            if (bits == 8) static_cast<uint8_t *>(B.slots)[i] = (uint8_t)c;
            else if (bits == 16) static_cast<uint16_t *>(B.slots)[i] = (uint16_t)c;
            else if (bits == 32) static_cast<uint32_t *>(B.slots)[i] = (uint32_t)c;
            else static_cast<uint64_t *>(B.slots)[i] = c;
        } else if (bits == 64) {
            dup |= atomicExch(static_cast<unsigned long long *>(B.slots) + i, (unsigned long long)c) != ~0ull;
        } else if (bits == 32) {
            dup |= atomicExch(static_cast<unsigned int *>(B.slots) + i, (unsigned int)c) != ~0u;
        } else {
            const unsigned int per = 32u / (unsigned int)bits, sh = (unsigned int)(i % per) * (unsigned int)bits;
            const unsigned int low = ((1u << bits) - 1u) << sh;
            const unsigned int old = atomicAnd(static_cast<unsigned int *>(B.slots) + i / per, ~low | ((unsigned int)c << sh));
            dup |= (old & low) != low;
        }
    }
    if (dup) set_status(B.status, SJQ_ERR_DUP_KEY);
}

// Build a direct table from the rows that this thread owns; returns how many it stored.  I: type of a slot index of
// a direct table; C: of a code.
template <typename Set, typename I, typename C>
__device__ __forceinline__ unsigned int build_rows(const BuildTask &B, const DimFilters &F)
{
    constexpr int kRows = Set::kRows;
    const int64_t apart = 4 * (int64_t)B.rows.blocks * kBuildThreads;
    unsigned int inserted = 0;
    for (int64_t r = 4 * ((int64_t)(blockIdx.x - B.rows.block0) * kBuildThreads + threadIdx.x);
         r - 4 * (int64_t)(threadIdx.x & 31) < B.rows.n; r += Set::kQuads * apart) { // whole warps stay together
        Set R;
        read_rows(B.rows, F, r, apart, R);
        C code[kRows];
        uint32_t mismatch = 0;
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            code[k] = 0;
            if (((R.m >> k) & 1u) && !pack_code(B, R, k, &code[k])) mismatch |= 1u << k;
        }
        I idx[kRows];
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            const uint64_t i = (uint64_t)(int64_t)R.key[k] - (uint64_t)B.kmin;
            idx[k] = (I)i;
            if (((R.m >> k) & 1u) && i >= B.span) mismatch |= 1u << k;
        }
        if (mismatch) set_status(B.status, SJQ_ERR_LAYOUT_MISMATCH);
        R.m &= ~mismatch;
#pragma unroll
        for (int q = 0; q < Set::kQuads; ++q) {
            const uint32_t m = (R.m >> (4 * q)) & 0xFu;
            if (B.kind == SJQ_TABLE_DIRECT_BITMAP) {
                set_bits<I>(static_cast<unsigned int *>(B.slots), &idx[4 * q], m, B.status);
            } else {
                store_codes(B, &idx[4 * q], &code[4 * q], m);
                if (B.filter) set_bits<I>(B.filter, &idx[4 * q], m, B.status);
            }
        }
        inserted += __popc(R.m);
    }
    return inserted;
}

__global__ void __launch_bounds__(kBuildThreads, 4) direct_build_kernel(const __grid_constant__ BuildParams P)
{
    const BuildTask &B = P.task[task_of_block(P.task, P.ntasks)];
    const DimRows &D = B.rows;
    cudaGridDependencySynchronize(); // the tables' memory is prepared by the kernel before this one
    unsigned int inserted;
    if (B.usual && !D.key64) inserted = build_rows<Usual<int32_t>, uint32_t, uint32_t>(B, P.filters);
    else if (B.usual) inserted = build_rows<Usual<int64_t>, uint32_t, uint32_t>(B, P.filters);
    else if (!D.key64) inserted = build_rows<Wide<int32_t>, uint64_t, uint64_t>(B, P.filters);
    else inserted = build_rows<Wide<int64_t>, uint64_t, uint64_t>(B, P.filters);
    if (B.expect_full < 0) return;
    // A probe of this table trusts the range test alone, so exactly so many rows must have been stored: the block
    // that comes last compares (repeated keys have been reported by then).
    __shared__ unsigned int part[kBuildThreads / 32];
    inserted = __reduce_add_sync(0xffffffffu, inserted);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = inserted;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kBuildThreads / 32; ++w) inserted += part[w];
        if (inserted) atomicAdd(&B.header[0], (unsigned long long)inserted);
        __threadfence();
        if (atomicAdd(&B.header[1], 1ull) == B.rows.blocks - 1ull) {
            __threadfence();
            if (atomicAdd(&B.header[0], 0ull) != (unsigned long long)B.expect_full) set_status(B.status, SJQ_ERR_LAYOUT_MISMATCH);
        }
    }
}

// Open addressing.  A key claims the first free slot on its probe path (bucket after bucket from its home bucket, the
// slots of a bucket in order) with atomicCAS on the key word, one CAS a step and no look before it (at the default load
// 1.3 steps place a key), then its code goes beside it.  Bounded by the number of buckets; a key met on the way is a
// duplicate.  The latency of the CASes bounds the kernel, so a warp gathers its passing rows in shared memory and every
// lane whose key has found its place takes the next one from there: a step costs the warp one latency, nearly all lanes
// have a key in it, and a lane still walking when the queue is empty goes on with the keys of the warp's next rows.
// 2 M keys of 8 M rows of 16 bytes into 80 MB, planned, built and probed by 10 M rows: 277 us with a warp placing 32 keys
// at a time and waiting for the last of them, 264 so.  (The CASes alone, random, take 45, the rows 20.)
constexpr int kHashThreads = 256;
constexpr int kHashQueue = 128; // a warp's next rows: the queue is empty before they come

// A key on its way to its place.
template <typename W, typename C>
struct HashWalk {
    W key;
    C code;
    uint32_t bucket, tried; // tried: buckets seen full
    int slot;
    bool on;
};

template <typename W, typename C>
__device__ __forceinline__ void hash_start(const BuildTask &B, HashWalk<W, C> &H)
{
    const uint64_t hashed = sizeof(W) == 8 ? (uint64_t)H.key : (uint64_t)(int64_t)(int32_t)H.key;
    if (B.filter) {
        const uint32_t fb = filter_hash(hashed) & B.fmask;
        atomicOr(B.filter + (fb >> 5), 1u << (fb & 31));
    }
    H.bucket = home_bucket(hashed, B.buckets);
    H.tried = 0;
    H.slot = 0;
    H.on = true;
}

template <typename W, typename C>
__device__ __forceinline__ void hash_step(const BuildTask &B, HashWalk<W, C> &H)
{
    const W empty = sizeof(W) == 8 ? (W)kEmptyKey64 : (W)(uint32_t)kEmptyKey32;
    char *const at = static_cast<char *>(B.slots) + (size_t)H.bucket * kBucketBytes;
    const W old = atomicCAS(reinterpret_cast<W *>(at) + H.slot, empty, H.key);
    if (old == empty) {
        if (B.code_bits == 32) reinterpret_cast<uint32_t *>(at + B.code_off)[H.slot] = (uint32_t)H.code;
        else if (B.code_bits == 64) reinterpret_cast<uint64_t *>(at + B.code_off)[H.slot] = H.code;
        H.on = false;
    } else if (old == H.key) {
        set_status(B.status, SJQ_ERR_DUP_KEY);
        H.on = false;
    } else if (++H.slot == B.bucket_k) {
        H.slot = 0;
        H.bucket = H.bucket + 1 == B.buckets ? 0 : H.bucket + 1;
        if (++H.tried == B.buckets) {
            set_status(B.status, SJQ_ERR_TABLE_FULL);
            H.on = false;
        }
    }
}

template <typename Set, typename C>
__device__ __forceinline__ void hash_rows(const BuildTask &B, const DimFilters &F, void *queue)
{
    typedef typename std::conditional<sizeof(typename Set::Key) == 8, unsigned long long, unsigned int>::type W;
    static_assert(Set::kQuads == 1, "the queue takes 128 rows at a time");
    const W empty = sizeof(W) == 8 ? (W)kEmptyKey64 : (W)(uint32_t)kEmptyKey32;
    const int lane = threadIdx.x & 31;
    const unsigned int below = (1u << lane) - 1u;
    W *const qkey = static_cast<W *>(queue);
    C *const qcode = reinterpret_cast<C *>(qkey + kHashQueue);
    HashWalk<W, C> H;
    H.on = false;
    for (int64_t r = 4 * ((int64_t)(blockIdx.x - B.rows.block0) * kHashThreads + threadIdx.x);
         r - 4 * lane < B.rows.n; r += 4 * (int64_t)B.rows.blocks * kHashThreads) { // whole warps stay together
        Set R;
        read_rows(B.rows, F, r, 0, R);
        int waiting = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            bool on = (R.m >> k) & 1u;
            C code = 0;
            if (on && !pack_code(B, R, k, &code)) {
                set_status(B.status, SJQ_ERR_LAYOUT_MISMATCH);
                on = false;
            }
            if (on && (W)R.key[k] == empty) {
                set_status(B.status, SJQ_ERR_RESERVED_KEY);
                on = false;
            }
            const unsigned int lanes = __ballot_sync(0xffffffffu, on);
            if (on) {
                const int at = waiting + __popc(lanes & below);
                qkey[at] = (W)R.key[k];
                qcode[at] = code;
            }
            waiting += __popc(lanes);
        }
        __syncwarp();
        while (waiting > 0) {
            const unsigned int idle = __ballot_sync(0xffffffffu, !H.on);
            const int mine = waiting - 1 - __popc(idle & below);
            if (!H.on && mine >= 0) {
                H.key = qkey[mine];
                H.code = qcode[mine];
                hash_start(B, H);
            }
            waiting -= __popc(idle);
            if (H.on) hash_step(B, H);
        }
        __syncwarp(); // the queue has been read
    }
    while (H.on) hash_step(B, H);
}

template <typename K>
using UsualQuad = RowSet<K, int32_t, 1, 1>;

// FORMS: what the dimensions of the launch are, usual (at most one payload, of 32 bits), others, which need more registers,
// or both.  A kernel that holds both keeps the usual ones at their 32-bit payloads and costs the others 1 to 3 %: tables of
// 8 M rows, one in four kept, beside one of 1,000 of the other form, others alone and both: usual 153 and 141 us, the other
// 163 and 166; 8 M rows of each 336 and 340.
constexpr int kFormUsual = 1, kFormOther = 2;
template <int FORMS>
constexpr int kHashPerSm = FORMS == kFormUsual ? 5 : 4;
template <int FORMS>
__global__ void __launch_bounds__(kHashThreads, kHashPerSm<FORMS>) hash_build_kernel(const __grid_constant__ BuildParams P)
{
    __shared__ __align__(16) unsigned char queues[kHashThreads / 32][kHashQueue * 16];
    const BuildTask &B = P.task[task_of_block(P.task, P.ntasks)];
    void *const queue = queues[threadIdx.x >> 5];
    cudaGridDependencySynchronize(); // the tables' memory is prepared by the kernel before this one
    if (FORMS == kFormUsual || (FORMS != kFormOther && B.usual)) {
        if (!B.rows.key64) hash_rows<UsualQuad<int32_t>, uint32_t>(B, P.filters, queue);
        else hash_rows<UsualQuad<int64_t>, uint32_t>(B, P.filters, queue);
    } else if constexpr (FORMS != kFormUsual) {
        if (!B.rows.key64) hash_rows<Wide<int32_t>, uint64_t>(B, P.filters, queue);
        else hash_rows<Wide<int64_t>, uint64_t>(B, P.filters, queue);
    }
}

int bits_for(uint64_t range)
{
    int b = 0;
    while (b < 64 && (range >> b) != 0) ++b;
    return b;
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Bytes of a direct table's slot array (bitmap words or packed codes), spare entry included.
size_t direct_array_bytes(const sjq_dim_layout &L)
{
    const uint64_t span = (uint64_t)L.slots;
    const uint64_t bits = L.kind == SJQ_TABLE_DIRECT_BITMAP ? 1 : (uint64_t)L.code_bits;
    return align_up((size_t)(((span + 1) * bits + 31) / 32 * 4), 16); // whole 32-bit words
}

// Device bytes a table of this shape occupies, recomputed from kind, slots, code_bits and filter_bits (never
// taken from the struct); false when the fields contradict one another.  sjq_dim_plan_end sizes tables with
// it and sjq_build_dim checks a caller-supplied layout against it, so that a stale or hand-edited layout is
// rejected on the host instead of making the fills and the build kernel write past table_mem.
bool layout_table_bytes(const sjq_dim_layout &L, size_t *bytes)
{
    if (L.slots <= 0 || L.npayload < 0 || L.npayload > SJQ_MAX_PAYLOADS || L.filter_bits < 0) return false;
    if (is_direct_kind(L.kind)) {
        if ((uint64_t)L.slots > ((uint64_t)1 << 40)) return false;
        if (L.code_bits != direct_kind_bits(L.kind) || (L.kind == SJQ_TABLE_DIRECT_BITMAP) != (L.npayload == 0))
            return false;
        // a sub-byte table without its presence bitmap could not tell a repeated key from a missing one
        if (L.code_bits > 0 && L.code_bits < 8 && L.filter_bits == 0) return false;
        if (L.filter_bits != 0 &&
            (L.kind == SJQ_TABLE_DIRECT_BITMAP || L.filter_bits <= L.slots || L.filter_bits % 128 != 0))
            return false;
        *bytes = kTableHeaderBytes + align_up(direct_array_bytes(L), 256) + align_up((size_t)(L.filter_bits / 8), 256);
        return true;
    }
    if (L.kind == SJQ_TABLE_HASH_I32 || L.kind == SJQ_TABLE_HASH_I64) {
        if ((L.kind == SJQ_TABLE_HASH_I64) != (L.key_dtype == SJQ_I64)) return false;
        if (L.npayload == 0 ? L.code_bits != 0 : (L.code_bits != 32 && L.code_bits != 64)) return false;
        const int k = bucket_keys(L.key_dtype == SJQ_I64 ? 8 : 4, L.code_bits / 8);
        if (L.slots % k != 0 || L.slots > ((int64_t)1 << 31)) return false; // whole buckets
        if ((L.filter_bits & (L.filter_bits - 1)) || L.filter_bits > ((int64_t)1 << 32)) return false;
        *bytes = kTableHeaderBytes + align_up((size_t)(L.slots / k) * kBucketBytes, 256) +
                 align_up((size_t)(L.filter_bits / 8), 256);
        return true;
    }
    return false;
}

// What the kernels read of one dimension, checked; its filters are appended to the launch's list.
sjq_status fill_rows(const sjq_dim_desc &d, DimRows *D, DimFilters *F, int *nfilters)
{
    if (!d.cols || d.ncols <= 0 || d.ncols > kMaxDimCols || d.npreds < 0 || d.npreds > SJQ_MAX_PREDS ||
        (d.npreds && !d.preds) || d.key_col < 0 || d.key_col >= d.ncols || d.npayload < 0 ||
        d.npayload > SJQ_MAX_PAYLOADS || (d.npayload && !d.payload_cols))
        return SJQ_ERR_INVALID_ARG;
    const int64_t n = d.cols[d.key_col].n;
    if (n < 0) return SJQ_ERR_INVALID_ARG;
    for (int c = 0; c < d.ncols; ++c) {
        const sjq_col &col = d.cols[c];
        if (col.n != n || (col.dtype != SJQ_I32 && col.dtype != SJQ_I64)) return SJQ_ERR_INVALID_ARG;
        if (n > 0 && !col.data) return SJQ_ERR_INVALID_ARG;
        if (!aligned16(col.data)) return SJQ_ERR_ALIGN;
    }
    *D = DimRows{};
    D->n = n;
    D->key = d.cols[d.key_col].data;
    D->key64 = (uint8_t)d.cols[d.key_col].dtype;
    D->npayload = d.npayload;
    for (int i = 0; i < d.npayload; ++i) {
        if (d.payload_cols[i] < 0 || d.payload_cols[i] >= d.ncols) return SJQ_ERR_INVALID_ARG;
        D->pay[i] = d.cols[d.payload_cols[i]].data;
        D->pay64[i] = (uint8_t)d.cols[d.payload_cols[i]].dtype;
    }
    D->pred0 = *nfilters;
    D->npreds = d.npreds;
    for (int k = 0; k < d.npreds; ++k) {
        const int c = d.preds[k].col;
        if (c < 0 || c >= d.ncols) return SJQ_ERR_INVALID_ARG;
        if (!canon_pred(d.preds[k], d.cols[c].dtype, &F->d[*nfilters])) return SJQ_ERR_INVALID_ARG;
        F->col[*nfilters] = d.cols[c].data;
        ++*nfilters;
    }
    return SJQ_OK;
}

// (argument errors come before a missing device)
sjq_status check_dims(const sjq_dim_desc *dims, int ndims)
{
    for (int i = 0; i < ndims; ++i) {
        DimRows rows;
        DimFilters filters;
        int nfilters = 0;
        const sjq_status st = fill_rows(dims[i], &rows, &filters, &nfilters);
        if (st != SJQ_OK) return st;
    }
    return SJQ_OK;
}

// How many of the dimensions from `first` on one launch can take.
int batch_of(const sjq_dim_desc *dims, int ndims, int first)
{
    int n = 0, preds = 0;
    while (first + n < ndims && n < kBatchDims) {
        preds += std::max(0, dims[first + n].npreds);
        if (n > 0 && preds > kBatchPreds) break;
        ++n;
    }
    return n;
}

// Blocks for tasks of `second` steps each: about `room` of them in all, at least one per task.  Returns the grid.
template <typename Get>
uint32_t share_blocks(int ntasks, int64_t room, Get task)
{
    int64_t total = 0;
    for (int i = 0; i < ntasks; ++i) total += task(i).second;
    const int64_t per = std::max<int64_t>(1, (total + room - 1) / room);
    uint32_t at = 0;
    for (int i = 0; i < ntasks; ++i) {
        auto t = task(i);
        t.first->block0 = at;
        t.first->blocks = (uint32_t)std::max<int64_t>(1, (t.second + per - 1) / per);
        at += t.first->blocks;
    }
    return at;
}

// Enqueue the scans of a batch; the statistics of dimension i go to scratch + i * kScratchWords (and to host[i]).
sjq_status scan_launch(const sjq_dim_desc *dims, int ndims, unsigned long long *scratch, int64_t *const *host, int sm_count,
                       cudaStream_t stream)
{
    ScanParams P;
    int nfilters = 0;
    for (int i = 0; i < ndims; ++i) {
        const sjq_status st = fill_rows(dims[i], &P.dim[i], &P.filters, &nfilters);
        if (st != SJQ_OK) return st;
        P.host[i] = host ? host[i] : nullptr;
    }
    P.ndims = ndims;
    P.scratch = scratch;
    if (cudaMemsetAsync(scratch, 0, (size_t)ndims * kScratchWords * 8, stream) != cudaSuccess) return SJQ_ERR_CUDA;
    // (a dimension without rows has a block too, which writes its statistics)
    const uint32_t grid = share_blocks(ndims, 2 * sm_count, [&](int i) {
        return std::make_pair(&P.dim[i], (P.dim[i].n + 8 * kScanThreads - 1) / (8 * kScanThreads));
    });
    plan_scan_kernel<<<grid, kScanThreads, 0, stream>>>(P);
    return cudaGetLastError() == cudaSuccess ? SJQ_OK : SJQ_ERR_CUDA;
}

// Page-locked words for the statistics that a waiting plan reads back: a plan has a piece for as long as it waits, and
// the process keeps up to kKeptStats of them, so that threads that come and go leave none behind.
constexpr int kKeptStats = 8;
constexpr size_t kStatsBytes = kBatchDims * 8 * sizeof(int64_t);
std::mutex g_stats_mutex;
int64_t *g_stats[kKeptStats];
int g_nstats = 0;

struct HostStats {
    int64_t *words = nullptr;

    HostStats()
    {
        {
            std::lock_guard<std::mutex> lock(g_stats_mutex);
            if (g_nstats > 0) words = g_stats[--g_nstats];
        }
        if (!words && cudaHostAlloc(reinterpret_cast<void **>(&words), kStatsBytes,
                                    cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            (void)cudaGetLastError();
            words = nullptr;
        }
    }
    HostStats(const HostStats &) = delete;
    HostStats &operator=(const HostStats &) = delete;
    ~HostStats()
    {
        if (!words) return;
        {
            std::lock_guard<std::mutex> lock(g_stats_mutex);
            if (g_nstats < kKeptStats) {
                g_stats[g_nstats++] = words;
                return;
            }
        }
        if (cudaFreeHost(words) != cudaSuccess) (void)cudaGetLastError();
    }
    void abandon() { words = nullptr; } // after a failed wait: a kernel may still write there
};

} // namespace

bool canon_pred(const sjq_pred &p, int dtype, DPred *d)
{
    *d = DPred{};
    d->col = p.col;
    d->is64 = (uint8_t)(dtype == SJQ_I64);
    bool empty = false;
    switch (p.op) {
    case SJQ_EQ: d->lo = d->hi = p.lo; break;
    case SJQ_NE: d->lo = d->hi = p.lo; d->neg = 1; break;
    case SJQ_LT:
        if (p.lo == INT64_MIN) empty = true;
        else { d->lo = INT64_MIN; d->hi = p.lo - 1; }
        break;
    case SJQ_LE: d->lo = INT64_MIN; d->hi = p.lo; break;
    case SJQ_GT:
        if (p.lo == INT64_MAX) empty = true;
        else { d->lo = p.lo + 1; d->hi = INT64_MAX; }
        break;
    case SJQ_GE: d->lo = p.lo; d->hi = INT64_MAX; break;
    case SJQ_BETWEEN: d->lo = p.lo; d->hi = p.hi; break;
    case SJQ_IN:
        if (p.nset < 0 || p.nset > SJQ_MAX_IN_SET || (p.nset && !p.set)) return false;
        if (p.nset == 0) empty = true;
        for (int k = 0; k < p.nset; ++k) d->set[k] = p.set[k];
        d->nset = (uint8_t)p.nset;
        break;
    default: return false;
    }
    if (empty || d->lo > d->hi) {
        d->lo = 1;
        d->hi = 0;
    }
    // int32 view of the range
    if (d->lo > d->hi || d->lo > INT32_MAX || d->hi < INT32_MIN) {
        d->never = 1;
        d->lo32 = 1;
        d->hi32 = 0;
    } else {
        d->lo32 = d->lo < INT32_MIN ? INT32_MIN : (int32_t)d->lo;
        d->hi32 = d->hi > INT32_MAX ? INT32_MAX : (int32_t)d->hi;
    }
    return true;
}

sjq_status device_info(DeviceInfo *out)
{
    static thread_local DeviceInfo cache[64];
    static thread_local bool have[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    if (dev >= 0 && dev < 64 && have[dev]) {
        *out = cache[dev];
        return SJQ_OK;
    }
    DeviceInfo d{};
    d.device = dev;
    if (cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&d.max_smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&d.l2_bytes, cudaDevAttrL2CacheSize, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    if (dev >= 0 && dev < 64) {
        cache[dev] = d;
        have[dev] = true;
    }
    *out = d;
    return SJQ_OK;
}

} // namespace sjq

using namespace sjq;

extern "C" sjq_status sjq_dim_plan_begin(const sjq_col *cols, int ncols, const sjq_pred *preds, int npreds,
                                         int key_col, const int *payload_cols, int npayload, void *scratch_dev,
                                         int64_t *host_stats, void *stream_)
{
    if (!scratch_dev || !host_stats) return SJQ_ERR_INVALID_ARG;
    if (!aligned16(scratch_dev)) return SJQ_ERR_ALIGN;
    const sjq_dim_desc d{cols, ncols, preds, npreds, key_col, payload_cols, npayload, nullptr};
    DeviceInfo dev;
    sjq_status st = check_dims(&d, 1);
    if (st == SJQ_OK) st = device_info(&dev);
    if (st != SJQ_OK) return st;
    cudaStream_t stream = (cudaStream_t)stream_;
    st = scan_launch(&d, 1, static_cast<unsigned long long *>(scratch_dev), nullptr, dev.sm_count, stream);
    if (st == SJQ_OK &&
        cudaMemcpyAsync(host_stats, scratch_dev, 8 * sizeof(int64_t), cudaMemcpyDeviceToHost, stream) != cudaSuccess)
        st = SJQ_ERR_CUDA;
    if (st == SJQ_ERR_CUDA) (void)cudaGetLastError();
    return st;
}

namespace sjq {
int host_stats_release()
{
    std::lock_guard<std::mutex> lock(g_stats_mutex);
    const int n = g_nstats;
    while (g_nstats > 0)
        if (cudaFreeHost(g_stats[--g_nstats]) != cudaSuccess) (void)cudaGetLastError();
    return n;
}
} // namespace sjq

extern "C" sjq_status sjq_dims_plan(const sjq_dim_desc *dims, int ndims, void *scratch_dev, size_t scratch_bytes,
                                    void *stream_, sjq_dim_layout *layouts)
{
    if (!dims || ndims <= 0 || !scratch_dev || !layouts) return SJQ_ERR_INVALID_ARG;
    if (!aligned16(scratch_dev)) return SJQ_ERR_ALIGN;
    if (scratch_bytes < (size_t)ndims * SJQ_PLAN_SCRATCH_BYTES) return SJQ_ERR_BUFFER_SMALL;
    DeviceInfo dev;
    sjq_status st = check_dims(dims, ndims);
    if (st == SJQ_OK) st = device_info(&dev);
    if (st != SJQ_OK) return st;
    HostStats host;
    if (!host.words) return SJQ_ERR_CUDA;
    int64_t *words[kBatchDims];
    for (int i = 0; i < kBatchDims; ++i) words[i] = host.words + 8 * i;
    cudaStream_t stream = (cudaStream_t)stream_;
    for (int first = 0; first < ndims;) {
        const int n = batch_of(dims, ndims, first);
        st = scan_launch(dims + first, n, static_cast<unsigned long long *>(scratch_dev), words, dev.sm_count, stream);
        // the kernel writes the statistics into the page-locked words itself
        if (st == SJQ_OK && cudaStreamSynchronize(stream) != cudaSuccess) {
            host.abandon();
            st = SJQ_ERR_CUDA;
        }
        if (st != SJQ_OK) {
            (void)cudaGetLastError();
            return st;
        }
        for (int i = 0; i < n; ++i) {
            const sjq_dim_desc &d = dims[first + i];
            st = sjq_dim_plan_end(d.cols, d.ncols, d.key_col, d.npayload, d.opts, words[i], &layouts[first + i]);
            if (st != SJQ_OK) return st;
        }
        first += n;
    }
    return SJQ_OK;
}

extern "C" sjq_status sjq_dims_plan_begin(const sjq_dim_desc *dims, int ndims, void *scratch_dev, size_t scratch_bytes,
                                          int64_t *const *host_stats, void *stream_)
{
    if (!dims || ndims <= 0 || !scratch_dev || !host_stats) return SJQ_ERR_INVALID_ARG;
    if (!aligned16(scratch_dev)) return SJQ_ERR_ALIGN;
    if (scratch_bytes < (size_t)ndims * SJQ_PLAN_SCRATCH_BYTES) return SJQ_ERR_BUFFER_SMALL;
    DeviceInfo dev;
    sjq_status st = check_dims(dims, ndims);
    if (st == SJQ_OK) st = device_info(&dev);
    for (int first = 0; first < ndims && st == SJQ_OK;) {
        const int n = batch_of(dims, ndims, first);
        st = scan_launch(dims + first, n, static_cast<unsigned long long *>(scratch_dev) + (size_t)first * kScratchWords,
                         host_stats + first, dev.sm_count, (cudaStream_t)stream_);
        first += n;
    }
    if (st == SJQ_ERR_CUDA) (void)cudaGetLastError();
    return st;
}

extern "C" sjq_status sjq_dim_plan(const sjq_col *cols, int ncols, const sjq_pred *preds, int npreds, int key_col,
                                   const int *payload_cols, int npayload, const sjq_build_opts *opts,
                                   void *scratch_dev, void *stream, sjq_dim_layout *layout)
{
    const sjq_dim_desc d{cols, ncols, preds, npreds, key_col, payload_cols, npayload, opts};
    return sjq_dims_plan(&d, 1, scratch_dev, SJQ_PLAN_SCRATCH_BYTES, stream, layout);
}

extern "C" sjq_status sjq_dim_plan_end(const sjq_col *cols, int ncols, int key_col, int npayload,
                                       const sjq_build_opts *opts, const int64_t *h, sjq_dim_layout *layout)
{
    if (!layout || !h || !cols || ncols <= 0 || key_col < 0 || key_col >= ncols || npayload < 0 ||
        npayload > SJQ_MAX_PAYLOADS)
        return SJQ_ERR_INVALID_ARG;
    struct { int64_t n; } P{cols[key_col].n};

    sjq_dim_layout L{};
    L.key_dtype = cols[key_col].dtype;
    L.npayload = npayload;
    L.dim_rows = P.n;
    L.entries = h[2];
    if (L.entries > 0) {
        L.kmin = h[0];
        L.kmax = h[1];
    }
    uint64_t maxcode = 0;
    int total_bits = 0;
    for (int i = 0; i < npayload; ++i) {
        L.pay_min[i] = L.entries > 0 ? h[3 + 2 * i] : 0;
        L.pay_max[i] = L.entries > 0 ? h[4 + 2 * i] : 0;
        const uint64_t range = (uint64_t)L.pay_max[i] - (uint64_t)L.pay_min[i];
        L.pay_bits[i] = bits_for(range);
        if (total_bits + L.pay_bits[i] > 63) return SJQ_ERR_UNSUPPORTED;
        maxcode |= range << total_bits;
        total_bits += L.pay_bits[i];
    }
    // Narrowest code that leaves all-ones free as the miss marker; a table that holds every key of its range
    // (entries == slots) needs no marker below one byte, because there the range test alone decides a hit.
    const uint64_t span_if_any = (uint64_t)L.kmax - (uint64_t)L.kmin; // span - 1
    const bool every_key = L.entries > 0 && span_if_any + 1 == (uint64_t)L.entries;
    const int min_bits = (opts && opts->min_code_bits > 0) ? opts->min_code_bits : 2;
    if (min_bits != 2 && min_bits != 4 && min_bits != 8) return SJQ_ERR_INVALID_ARG;
    int code_bits = 0;
    if (npayload > 0) {
        if (min_bits <= 2 && (every_key ? maxcode <= 0x3u : maxcode < 0x3u)) code_bits = 2;
        else if (min_bits <= 4 && (every_key ? maxcode <= 0xFu : maxcode < 0xFu)) code_bits = 4;
        else if (maxcode < 0xFFu) code_bits = 8;
        else if (maxcode < 0xFFFFu) code_bits = 16;
        else if (maxcode < 0xFFFFFFFFu) code_bits = 32;
        else code_bits = 64;
    }
    const int force = opts ? opts->force_kind : SJQ_TABLE_AUTO;
    if (force != SJQ_TABLE_AUTO && force != SJQ_TABLE_FORCE_DIRECT && force != SJQ_TABLE_FORCE_HASH)
        return SJQ_ERR_INVALID_ARG;
    const int64_t max_direct = (opts && opts->max_direct_bytes > 0) ? opts->max_direct_bytes : (int64_t)64 << 20;
    // (the skewed 64-bit-key workload: 1.61 / 1.65 / 1.71 / 1.91 ms at load 33 / 40 / 50 / 60 %)
    const int load_pct = (opts && opts->hash_load_pct > 0) ? opts->hash_load_pct : 40;
    if (load_pct > 90) return SJQ_ERR_INVALID_ARG;

    const uint64_t span_m1 = (uint64_t)L.kmax - (uint64_t)L.kmin; // span - 1, no overflow
    bool direct_ok = span_m1 < ((uint64_t)1 << 40);
    size_t direct_bytes = 0;
    if (direct_ok) {
        const uint64_t span = span_m1 + 1;
        // one spare entry after the last slot, never set: a probe clamps its index there instead of testing the range
        direct_bytes = align_up((size_t)(((span + 1) * (uint64_t)(npayload == 0 ? 1 : code_bits) + 31) / 32 * 4), 16);
    }
    bool use_direct;
    if (force == SJQ_TABLE_FORCE_DIRECT) {
        if (!direct_ok || direct_bytes > ((size_t)1 << 36)) return SJQ_ERR_UNSUPPORTED;
        use_direct = true;
    } else if (force == SJQ_TABLE_FORCE_HASH) {
        use_direct = false;
    } else {
        use_direct = direct_ok && (int64_t)direct_bytes <= max_direct;
    }
    if (use_direct) {
        L.slots = (int64_t)(span_m1 + 1);
        L.code_bits = code_bits;
        L.kind = npayload == 0 ? SJQ_TABLE_DIRECT_BITMAP
                 : code_bits == 2 ? SJQ_TABLE_DIRECT_U2
                 : code_bits == 4 ? SJQ_TABLE_DIRECT_U4
                 : code_bits == 8 ? SJQ_TABLE_DIRECT_U8
                 : code_bits == 16 ? SJQ_TABLE_DIRECT_U16
                 : code_bits == 32 ? SJQ_TABLE_DIRECT_U32
                                   : SJQ_TABLE_DIRECT_U64;
        // a code array is 8 to 64 times the size of a bitmap over the same slots: keep both, so that a
        // filter stage probes the bitmap and only the survivors gather their payload from the codes
        if (npayload > 0) L.filter_bits = (int64_t)((span_m1 + 129) / 128 * 128); // at least one spare bit after the last slot
    } else {
        L.kind = L.key_dtype == SJQ_I64 ? SJQ_TABLE_HASH_I64 : SJQ_TABLE_HASH_I32;
        L.code_bits = npayload == 0 ? 0 : (code_bits <= 32 ? 32 : 64);
        const uint64_t k = (uint64_t)bucket_keys(L.key_dtype == SJQ_I64 ? 8 : 4, L.code_bits / 8);
        const uint64_t want = ((uint64_t)L.entries * 100u + (uint64_t)load_pct - 1) / (uint64_t)load_pct;
        const uint64_t buckets = std::max<uint64_t>((want + k - 1) / k, 2);
        L.slots = (int64_t)(buckets * k);
        // presence bitmap: 16 bits per entry (about 6 % false positives), at least 1024 bits, at most 2^32
        uint64_t fbits = 1024;
        while (fbits < (uint64_t)L.entries * 16 && fbits < ((uint64_t)1 << 32)) fbits <<= 1;
        L.filter_bits = (int64_t)fbits;
    }
    if (!layout_table_bytes(L, &L.table_bytes)) return SJQ_ERR_UNSUPPORTED;
    *layout = L;
    return SJQ_OK;
}

namespace sjq {
namespace {

// Check one table of a batch and describe its build and the fills before it.
sjq_status describe_build(const sjq_dim_desc &d, const sjq_dim_layout &L, void *table_mem, size_t table_bytes,
                          int32_t *status_dev, BuildTask *B, DimFilters *F, int *nfilters, FillParams *I, sjq_table *T)
{
    if (!table_mem || !status_dev) return SJQ_ERR_INVALID_ARG;
    if (!aligned16(table_mem)) return SJQ_ERR_ALIGN;
    *B = BuildTask{};
    sjq_status st = fill_rows(d, &B->rows, F, nfilters);
    if (st != SJQ_OK) return st;
    // The layout is the caller's: every size used below is recomputed from its shape fields, never taken
    // from its table_bytes, and a layout whose fields contradict one another is rejected here.
    size_t need_bytes = 0;
    if (L.npayload != d.npayload || L.key_dtype != d.cols[d.key_col].dtype || L.dim_rows != B->rows.n ||
        !layout_table_bytes(L, &need_bytes) || need_bytes != L.table_bytes)
        return SJQ_ERR_INVALID_ARG;
    for (int i = 0; i < d.npayload; ++i)
        if (L.pay_bits[i] < 0 || L.pay_bits[i] > 63) return SJQ_ERR_INVALID_ARG;
    if (table_bytes < need_bytes) return SJQ_ERR_BUFFER_SMALL;

    T->layout = L;
    T->base = static_cast<char *>(table_mem);
    T->slots = T->base + kTableHeaderBytes;
    T->filter = nullptr;
    T->launches = 0;
    T->magic = kTableMagic;

    B->kind = L.kind;
    B->code_bits = L.code_bits;
    B->kmin = L.kmin;
    B->span = (uint64_t)L.slots;
    for (int i = 0; i < SJQ_MAX_PAYLOADS; ++i) {
        B->pay_min[i] = L.pay_min[i];
        B->pay_max[i] = L.pay_max[i];
        B->pay_bits[i] = L.pay_bits[i];
    }
    B->header = reinterpret_cast<unsigned long long *>(T->base);
    B->status = status_dev;
    B->slots = T->slots;
    const bool direct = is_direct_kind(L.kind);
    B->usual = usual_payloads(B->rows) && (!direct || L.slots <= INT32_MAX) && L.pay_min[0] >= INT32_MIN &&
               L.pay_max[0] <= INT32_MAX && L.pay_min[0] <= L.pay_max[0];
    B->expect_full = direct && L.code_bits > 0 && L.code_bits < 8 && L.entries == L.slots ? (long long)L.entries : -1;

    uint4 pattern;
    if (direct) {
        T->slots_bytes = direct_array_bytes(L);
        const unsigned int fill = L.kind == SJQ_TABLE_DIRECT_BITMAP ? 0u : 0xFFFFFFFFu;
        pattern = make_uint4(fill, fill, fill, fill);
    } else {
        const int kb = L.key_dtype == SJQ_I64 ? 8 : 4, cb = L.code_bits / 8;
        B->bucket_k = bucket_keys(kb, cb);
        B->code_off = bucket_code_offset(kb, cb, B->bucket_k);
        B->buckets = (uint32_t)(L.slots / B->bucket_k);
        B->fmask = (uint32_t)(L.filter_bits - 1);
        T->slots_bytes = (size_t)B->buckets * kBucketBytes;
        // Every word of a bucket starts as the empty marker's pattern: both markers (the minimum of the key
        // type) are a repeated 0x80 00 .. 00 word, so the codes start as that pattern too and are overwritten
        // when their slot is claimed.
        pattern = L.key_dtype == SJQ_I64 ? make_uint4(0u, 0x80000000u, 0u, 0x80000000u)
                                         : make_uint4(0x80000000u, 0x80000000u, 0x80000000u, 0x80000000u);
    }
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    if (B->expect_full >= 0) I->task[I->ntasks++] = {reinterpret_cast<uint4 *>(T->base), kTableHeaderBytes / 16, zero, 0, 0};
    I->task[I->ntasks++] = {reinterpret_cast<uint4 *>(T->slots), (T->slots_bytes + 15) / 16, pattern, 0, 0};
    if (L.filter_bits) {
        T->filter = T->slots + align_up(T->slots_bytes, 256);
        B->filter = reinterpret_cast<unsigned int *>(T->filter);
        // (the layout pads the bitmap's region to 256 bytes)
        I->task[I->ntasks++] = {reinterpret_cast<uint4 *>(T->filter), ((size_t)(L.filter_bits / 8) + 15) / 16, zero, 0, 0};
    }
    return SJQ_OK;
}

// Launch a build kernel behind the fills: it waits for them on the device.
bool launch_behind(void (*kernel)(BuildParams), BuildParams &B, int threads, int blocks_per_sm, int sm_count, cudaStream_t stream)
{
    const uint32_t grid = share_blocks(B.ntasks, (int64_t)blocks_per_sm * sm_count, [&](int i) {
        return std::make_pair(&B.task[i].rows, (B.task[i].rows.n + 4 * threads - 1) / (4 * threads));
    });
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, B) == cudaSuccess;
}

template <int FORMS>
bool launch_hash_build(BuildParams &H, int sm_count, cudaStream_t stream)
{
    return launch_behind(hash_build_kernel<FORMS>, H, kHashThreads, kHashPerSm<FORMS>, sm_count, stream);
}

// Enqueue the fills and the builds of a batch: one launch for the direct tables, one for those with open addressing.
sjq_status build_launch(const sjq_dim_desc *dims, int ndims, const sjq_dim_layout *layouts, void *const *table_mem,
                        const size_t *table_bytes, int32_t *const *status_dev, bool clear_status, void *stream_,
                        sjq_table **tables)
{
    cudaStream_t stream = (cudaStream_t)stream_;
    BuildParams B, H;
    FillParams I{};
    int nfilters = 0;
    B.ntasks = H.ntasks = 0;
    sjq_status st = SJQ_OK;
    for (int i = 0; i < ndims && st == SJQ_OK; ++i) { // (the entries of `tables` are NULL before)
        tables[i] = new (std::nothrow) sjq_table();
        if (!tables[i]) {
            st = SJQ_ERR_INVALID_ARG;
            break;
        }
        BuildParams &to = is_hash_kind(layouts[i].kind) ? H : B;
        BuildTask &task = to.task[to.ntasks];
        st = describe_build(dims[i], layouts[i], table_mem[i], table_bytes[i], status_dev[i], &task, &B.filters,
                            &nfilters, &I, tables[i]);
        if (st != SJQ_OK) break;
        if (clear_status) I.clear_status[i] = status_dev[i];
        // (a layout that promises every key of its range is checked against a dimension without rows too)
        if (task.rows.n > 0 || task.expect_full >= 0) ++to.ntasks;
    }
    DeviceInfo dev;
    if (st == SJQ_OK) st = device_info(&dev);
    if (st == SJQ_OK) {
        const uint32_t fill_grid = share_blocks(I.ntasks, 8 * dev.sm_count, [&](int i) {
            return std::make_pair(&I.task[i], (int64_t)((I.task[i].units + kFillTile - 1) / kFillTile));
        });
        table_init_kernel<<<fill_grid, kFillThreads, 0, stream>>>(I);
        bool ok = cudaGetLastError() == cudaSuccess;
        int launches = 1;
        if (ok && B.ntasks) {
            ok = launch_behind(direct_build_kernel, B, kBuildThreads, 4, dev.sm_count, stream);
            ++launches;
        }
        if (ok && H.ntasks) {
            H.filters = B.filters;
            int64_t usual = 0, other = 0;
            for (int i = 0; i < H.ntasks; ++i) (H.task[i].usual ? usual : other) += H.task[i].rows.n;
            ok = other == 0     ? launch_hash_build<kFormUsual>(H, dev.sm_count, stream)
                 : usual > other ? launch_hash_build<kFormUsual | kFormOther>(H, dev.sm_count, stream)
                                 : launch_hash_build<kFormOther>(H, dev.sm_count, stream);
            ++launches;
        }
        tables[0]->launches = launches;
        if (!ok) {
            (void)cudaGetLastError();
            st = SJQ_ERR_CUDA;
        }
    }
    if (st != SJQ_OK)
        for (int i = 0; i < ndims; ++i) {
            delete tables[i];
            tables[i] = nullptr;
        }
    return st;
}

} // namespace
} // namespace sjq

extern "C" sjq_status sjq_dims_build(const sjq_dim_desc *dims, int ndims, const sjq_dim_layout *layouts,
                                     void *const *table_mem, const size_t *table_bytes, int32_t *const *status_dev,
                                     int32_t clear_status, void *stream, sjq_table **tables)
{
    if (!dims || ndims <= 0 || !layouts || !table_mem || !table_bytes || !status_dev || !tables) return SJQ_ERR_INVALID_ARG;
    for (int i = 0; i < ndims; ++i) tables[i] = nullptr;
    for (int first = 0; first < ndims;) {
        const int n = batch_of(dims, ndims, first);
        const sjq_status st = build_launch(dims + first, n, layouts + first, table_mem + first, table_bytes + first,
                                           status_dev + first, clear_status != 0, stream, tables + first);
        if (st != SJQ_OK) {
            for (int i = 0; i < ndims; ++i) {
                delete tables[i];
                tables[i] = nullptr;
            }
            return st;
        }
        first += n;
    }
    return SJQ_OK;
}

extern "C" sjq_status sjq_build_dim(const sjq_col *cols, int ncols, const sjq_pred *preds, int npreds, int key_col,
                                    const int *payload_cols, int npayload, const sjq_dim_layout *layout,
                                    void *table_mem, size_t table_bytes, int32_t *status_dev, void *stream,
                                    sjq_table **table)
{
    if (!layout || !table_mem || !status_dev || !table) return SJQ_ERR_INVALID_ARG;
    const sjq_dim_desc d{cols, ncols, preds, npreds, key_col, payload_cols, npayload, nullptr};
    sjq_table *made = nullptr;
    const sjq_status st = build_launch(&d, 1, layout, &table_mem, &table_bytes, &status_dev, false, stream, &made);
    if (st == SJQ_OK) *table = made;
    return st;
}

extern "C" sjq_status sjq_dim_layout_bytes(const sjq_dim_layout *layout, size_t *bytes)
{
    if (!layout || !bytes) return SJQ_ERR_INVALID_ARG;
    return layout_table_bytes(*layout, bytes) ? SJQ_OK : SJQ_ERR_INVALID_ARG;
}

extern "C" sjq_status sjq_table_info(const sjq_table *table, sjq_dim_layout *layout)
{
    if (!table || table->magic != kTableMagic || !layout) return SJQ_ERR_INVALID_ARG;
    *layout = table->layout;
    return SJQ_OK;
}

extern "C" int32_t sjq_table_kernel_launches(const sjq_table *table)
{
    return (table && table->magic == kTableMagic) ? table->launches : 0;
}

extern "C" void sjq_table_destroy(sjq_table *table)
{
    if (table && table->magic == kTableMagic) {
        table->magic = 0;
        delete table;
    }
}

extern "C" const char *sjq_strerror(sjq_status s)
{
    switch (s) {
    case SJQ_OK: return "ok";
    case SJQ_ERR_INVALID_ARG: return "invalid argument";
    case SJQ_ERR_UNSUPPORTED: return "unsupported query or table shape";
    case SJQ_ERR_ALIGN: return "device pointer not 16-byte aligned";
    case SJQ_ERR_CUDA: return "CUDA runtime error (no device or launch failure)";
    case SJQ_ERR_BUFFER_SMALL: return "caller-provided buffer too small";
    case SJQ_ERR_STATIC_LIMIT: return "request exceeds the built-in scratch of the no-allocation entry point";
    case SJQ_ERR_JIT: return "run-time specialisation unavailable (compiler, device sources or module load)";
    case SJQ_ERR_DUP_KEY: return "duplicate dimension key among rows passing the filter";
    case SJQ_ERR_TABLE_FULL: return "hash table full";
    case SJQ_ERR_GROUP_RANGE: return "group key outside [0, num_groups)";
    case SJQ_ERR_GROUP_OVERFLOW: return "more distinct groups than the hashed capacity";
    case SJQ_ERR_RESERVED_KEY: return "dimension key equals the reserved empty marker";
    case SJQ_ERR_LAYOUT_MISMATCH: return "dimension data does not match the planned layout";
    case SJQ_ERR_ASYNC_WAIT: return "a bounded wait for a bulk-asynchronous copy ran out (result still exact)";
    default: return "unknown status";
    }
}

extern "C" const char *sjq_version(void) { return "sjq 0.1 (sm_100a)"; }
