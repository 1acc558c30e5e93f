// Canonical order of a hashed result: ascending key.
//
// The global group table of Section 3.3 hands its groups back in table order, which depends on the hash function
// and on the capacity; two runs of the same query agree only as sets.  sjq_result_sort puts the list of
// (key, sum, count) triples into ascending signed key order on the device: a stable least-significant-digit radix
// sort of (key - smallest key, position) pairs, 8 bits a pass.
//
// The number of groups and the range of the keys are known on the device only, so nothing waits on the host: the
// host enqueues every pass that 64-bit keys could need, a first kernel finds smallest and largest key and whether
// the list is in order already, and the passes that the range does not need return at once (group keys are small
// numbers as a rule: 20 bits for a million groups, three passes; a list in order needs none).
//
// What bounds it: kernel latency.  A pass over a million pairs moves 24 MB, which the L2 holds, so its two kernels
// are short (5 to 15 us) and what they do one after the other counts.  Hence
//   - at most kSortBlocks blocks of 1024 threads (one per SM), each owning one contiguous piece of the list: the
//     digit counts are kSortBlocks x 256 words whatever the length, and every scatter block forms its own offsets
//     from them (a kernel of its own that scanned 256 counts per 1024 elements with one block took 461 us a pass
//     at a capacity of 2 million, 9/10 of the whole sort; the counts of 8 SMs' worth of loads take 2 us here);
//   - the measures travel once: they are copied aside by the first counting kernel and gathered by the last
//     scatter, which writes all three result arrays;
//   - each kernel is launched while its predecessor still runs and waits for it on the device (programmatic
//     dependent launch), so that a pass without work costs about a microsecond.
#include <algorithm>

#include "sjq_internal.h"

namespace sjq {
namespace {

constexpr int kSortThreads = 1024;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortRounds = 4;                         // elements per thread and tile
constexpr int kSortTile = kSortThreads * kSortRounds;
constexpr int kSortBlocks = 148;                       // one per SM
constexpr int kSortMinPiece = 2048;                    // elements a block takes before another one is put to work
constexpr int kSortPasses = 8;

struct SortRange {
    unsigned long long lo, hi; // smallest and largest key, sign bit flipped
    unsigned long long disorder; // a key larger than its successor was seen
    unsigned long long pad;
};

struct SortHeader {
    unsigned long long lo;
    int32_t passes; // digits the range needs; 0: nothing to do
    int32_t pad;
};

struct SortParams {
    const int64_t *n_groups; // device: number of entries
    int64_t capacity;
    int64_t *keys, *sums, *counts; // the list, sorted in place
    unsigned long long *k[2];      // keys less the smallest one, in turn
    unsigned int *p[2];            // positions in the list as it came, in turn
    int64_t *tsums, *tcounts;      // the measures as they came
    SortRange *ranges;             // one per block of the first kernel
    SortHeader *header;
    unsigned int *totals;          // [kSortPasses][256] elements per digit
    unsigned int *hist;            // [kSortBlocks][256] elements per block and digit of the current pass
    int32_t pass;
};

__device__ __forceinline__ unsigned long long flip(int64_t k) { return (unsigned long long)k ^ 0x8000000000000000ull; }

__device__ __forceinline__ int64_t sort_count(const SortParams &S)
{
    const int64_t n = *S.n_groups;
    return n < 0 ? 0 : (n > S.capacity ? S.capacity : n);
}

// The piece of the list that this block owns: [lo, hi), the same in every kernel of a sort.
__device__ __forceinline__ void sort_piece(int64_t n, int64_t *lo, int64_t *hi)
{
    int64_t blocks = (n + kSortMinPiece - 1) / kSortMinPiece;
    if (blocks > (int64_t)gridDim.x) blocks = gridDim.x;
    if (blocks < 1) blocks = 1;
    const int64_t per = (n + blocks - 1) / blocks;
    const int64_t a = (int64_t)blockIdx.x * per, b = a + per;
    *lo = a < n ? a : n;
    *hi = b < n ? b : n;
}

// Range of the keys and whether they are in order, one record per block.
__global__ void __launch_bounds__(kSortThreads) sort_range_kernel(const __grid_constant__ SortParams S)
{
    cudaTriggerProgrammaticLaunchCompletion();
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < kSortPasses * 256; i += kSortThreads) S.totals[i] = 0;
    int64_t lo, hi;
    const int64_t n = sort_count(S);
    sort_piece(n, &lo, &hi);
    unsigned long long kmin = ~0ull, kmax = 0ull, disorder = 0ull;
    for (int64_t i = lo + threadIdx.x; i < hi; i += kSortThreads) {
        const unsigned long long k = flip(S.keys[i]);
        kmin = k < kmin ? k : kmin;
        kmax = k > kmax ? k : kmax;
        if (i + 1 < n && flip(S.keys[i + 1]) < k) disorder = 1ull;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, kmin, o), b = __shfl_xor_sync(0xffffffffu, kmax, o);
        kmin = a < kmin ? a : kmin;
        kmax = b > kmax ? b : kmax;
    }
    __shared__ unsigned long long wlo[kSortWarps], whi[kSortWarps];
    const int any = __syncthreads_or((int)disorder);
    if ((threadIdx.x & 31) == 0) {
        wlo[threadIdx.x >> 5] = kmin;
        whi[threadIdx.x >> 5] = kmax;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kSortWarps; ++w) {
            kmin = wlo[w] < kmin ? wlo[w] : kmin;
            kmax = whi[w] > kmax ? whi[w] : kmax;
        }
        S.ranges[blockIdx.x] = SortRange{kmin, kmax, any ? 1ull : 0ull, 0ull};
    }
}

// What the ranges of all blocks say, formed by every block for itself in the first counting kernel (later kernels
// read the header that block 0 leaves).
__device__ __forceinline__ SortHeader sort_header(const SortParams &S)
{
    __shared__ SortHeader H;
    if (S.pass > 0) return *S.header;
    if (threadIdx.x < 32) {
        unsigned long long lo = ~0ull, hi = 0ull, disorder = 0ull;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) {
            const SortRange r = S.ranges[b];
            lo = r.lo < lo ? r.lo : lo;
            hi = r.hi > hi ? r.hi : hi;
            disorder |= r.disorder;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long a = __shfl_xor_sync(0xffffffffu, lo, o), b = __shfl_xor_sync(0xffffffffu, hi, o);
            lo = a < lo ? a : lo;
            hi = b > hi ? b : hi;
        }
        const bool sorted = __all_sync(0xffffffffu, disorder == 0ull);
        if (threadIdx.x == 0) {
            H.lo = lo;
            H.passes = sorted || hi <= lo ? 0 : (64 - __clzll((long long)(hi - lo)) + 7) / 8;
            if (blockIdx.x == 0) *S.header = H;
        }
    }
    __syncthreads();
    return H;
}

// Elements per digit of this block's piece.  Eight copies of the counters, by lane, keep the conflicts low where
// a digit takes few values (the top digit of a range).
__global__ void __launch_bounds__(kSortThreads) sort_hist_kernel(const __grid_constant__ SortParams S)
{
    constexpr int kCopies = 8;
    __shared__ unsigned int h[kCopies][256];
    cudaTriggerProgrammaticLaunchCompletion();
    for (int i = threadIdx.x; i < kCopies * 256; i += kSortThreads) (&h[0][0])[i] = 0;
    cudaGridDependencySynchronize();
    const SortHeader H = sort_header(S);
    if (S.pass >= H.passes) return;
    int64_t lo, hi;
    sort_piece(sort_count(S), &lo, &hi);
    if (lo >= hi && blockIdx.x > 0) return; // no piece: nobody reads this block's counts
    __syncthreads();
    unsigned int *const mine = h[threadIdx.x & (kCopies - 1)];
    const unsigned long long *const in = S.k[S.pass & 1];
    const int shift = 8 * S.pass;
    for (int64_t i = lo + threadIdx.x; i < hi; i += kSortThreads) {
        unsigned long long k;
        if (S.pass == 0) { // the list is copied aside on the way
            k = flip(S.keys[i]) - H.lo;
            S.k[0][i] = k;
            S.tsums[i] = S.sums[i];
            S.tcounts[i] = S.counts[i];
        } else {
            k = in[i];
        }
        atomicAdd(&mine[(unsigned int)(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        unsigned int c = 0;
        for (int j = 0; j < kCopies; ++j) c += h[j][threadIdx.x];
        S.hist[(size_t)blockIdx.x * 256 + threadIdx.x] = c;
        if (c) atomicAdd(&S.totals[S.pass * 256 + threadIdx.x], c);
    }
}

// Stable scatter of this block's piece, tile by tile.  A warp owns 128 consecutive elements of a tile and takes them
// 32 at a time; an element's position is the start of its digit, plus the elements with that digit in earlier
// blocks, earlier tiles, earlier warps of the tile and earlier lanes of the warp.
__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(const __grid_constant__ SortParams S)
{
    __shared__ unsigned int offset[256];               // next output position per digit
    __shared__ unsigned short wcount[kSortWarps][256]; // per warp: elements per digit, then those of earlier warps
    __shared__ unsigned int part[4][256];
    __shared__ unsigned int scan[8];
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    const SortHeader H = *S.header;
    if (S.pass >= H.passes) return;
    const bool last = S.pass == H.passes - 1;
    int64_t lo, hi;
    sort_piece(sort_count(S), &lo, &hi);
    if (lo >= hi) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int digit_of_thread = threadIdx.x & 255, quarter = threadIdx.x >> 8;
    {
        // elements of every digit in the blocks before this one, a quarter of the blocks per group of 256 threads
        const int b1 = (int)blockIdx.x;
        unsigned int sum = 0;
#pragma unroll 8
        for (int b = quarter; b < b1; b += 4) sum += S.hist[(size_t)b * 256 + digit_of_thread];
        part[quarter][digit_of_thread] = sum;
        // start of every digit: exclusive scan of the 256 totals
        unsigned int total = 0, incl = 0;
        if (threadIdx.x < 256) {
            total = S.totals[S.pass * 256 + threadIdx.x];
            incl = total;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) scan[warp] = incl;
        }
        __syncthreads();
        if (threadIdx.x < 256) {
            for (int w = 0; w < warp; ++w) incl += scan[w];
            offset[threadIdx.x] = incl - total + part[0][threadIdx.x] + part[1][threadIdx.x] + part[2][threadIdx.x] + part[3][threadIdx.x];
        }
    }
    const unsigned long long *const kin = S.k[S.pass & 1];
    const unsigned int *const pin = S.p[S.pass & 1];
    unsigned long long *const kout = S.k[(S.pass & 1) ^ 1];
    unsigned int *const pout = S.p[(S.pass & 1) ^ 1];
    const int shift = 8 * S.pass;
    for (int64_t base = lo; base < hi; base += kSortTile) {
        unsigned long long key[kSortRounds];
        unsigned int pos[kSortRounds];
        unsigned short rank[kSortRounds];
#pragma unroll
        for (int r = 0; r < kSortRounds; ++r) {
            const int64_t i = base + warp * (32 * kSortRounds) + r * 32 + lane;
            key[r] = 0;
            pos[r] = 0;
            if (i < hi) {
                key[r] = kin[i];
                pos[r] = S.pass ? pin[i] : (unsigned int)i;
            }
        }
        reinterpret_cast<uint4 *>(&wcount[0][0])[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
        static_assert(sizeof(wcount) == kSortThreads * sizeof(uint4), "one 16-byte store per thread clears the counters");
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSortRounds; ++r) {
            const bool valid = base + warp * (32 * kSortRounds) + r * 32 + lane < hi;
            const unsigned int digit = (unsigned int)(key[r] >> shift) & 255u;
            // lanes of the warp with the same digit; a lane without an element matches nobody
            const unsigned int peers = __match_any_sync(0xffffffffu, valid ? digit : 256u + (unsigned int)lane);
            const unsigned int before = __popc(peers & ((1u << lane) - 1u));
            const unsigned int seen = valid ? wcount[warp][digit] : 0u;
            __syncwarp();
            if (valid && before == 0) wcount[warp][digit] = (unsigned short)(seen + __popc(peers));
            __syncwarp();
            rank[r] = (unsigned short)(seen + before);
        }
        __syncthreads();
        // per digit: exclusive prefix over the 32 warps, eight warps per group of 256 threads
        unsigned int c[8], sum = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            c[j] = wcount[quarter * 8 + j][digit_of_thread];
            sum += c[j];
        }
        part[quarter][digit_of_thread] = sum;
        __syncthreads();
        unsigned int run = 0;
        for (int q = 0; q < quarter; ++q) run += part[q][digit_of_thread];
        const unsigned int tile_total = run + sum; // whole tile in the last group
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            wcount[quarter * 8 + j][digit_of_thread] = (unsigned short)run;
            run += c[j];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSortRounds; ++r) {
            if (base + warp * (32 * kSortRounds) + r * 32 + lane < hi) {
                const unsigned int digit = (unsigned int)(key[r] >> shift) & 255u;
                const unsigned int at = offset[digit] + wcount[warp][digit] + rank[r];
                if (last) {
                    S.keys[at] = (int64_t)((key[r] + H.lo) ^ 0x8000000000000000ull);
                    S.sums[at] = S.tsums[pos[r]];
                    S.counts[at] = S.tcounts[pos[r]];
                } else {
                    kout[at] = key[r];
                    pout[at] = pos[r];
                }
            }
        }
        __syncthreads();
        if (quarter == 3) offset[digit_of_thread] += tile_total;
        // (the next tile reads the offsets after two more barriers)
    }
}

size_t up256(size_t v) { return (v + 255) / 256 * 256; }

struct SortLayout {
    size_t k0, k1, p0, p1, ranges, header, totals, hist, tsums, tcounts, total;
    int nblocks;
};

SortLayout sort_layout(int64_t capacity)
{
    SortLayout L{};
    const size_t c = (size_t)std::max<int64_t>(capacity, 1);
    L.nblocks = (int)std::min<size_t>((c + kSortMinPiece - 1) / kSortMinPiece, (size_t)kSortBlocks);
    size_t at = 0;
    L.k0 = at, at += up256(c * 8);
    L.k1 = at, at += up256(c * 8);
    L.p0 = at, at += up256(c * 4);
    L.p1 = at, at += up256(c * 4);
    L.ranges = at, at += up256(sizeof(SortRange) * L.nblocks);
    L.header = at, at += 256;
    L.totals = at, at += (size_t)kSortPasses * 256 * 4;
    L.hist = at, at += (size_t)256 * L.nblocks * 4;
    L.tsums = at, at += up256(c * 8);
    L.tcounts = at, at += up256(c * 8);
    L.total = at;
    return L;
}

// Launch behind the previous kernel of the sort without waiting for it: every kernel but the first waits on the
// device (cudaGridDependencySynchronize) before it touches what its predecessors wrote.
bool launch_behind(void (*kernel)(SortParams), int grid, const SortParams &S, cudaStream_t stream)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kSortThreads);
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, S) == cudaSuccess;
}

} // namespace
} // namespace sjq

using namespace sjq;

extern "C" sjq_status sjq_result_sort_scratch_bytes(int64_t capacity, size_t *bytes)
{
    if (capacity <= 0 || capacity > ((int64_t)1 << 31) || !bytes) return SJQ_ERR_INVALID_ARG;
    *bytes = sort_layout(capacity).total;
    return SJQ_OK;
}

extern "C" sjq_status sjq_result_sort(int64_t *keys, int64_t *sums, int64_t *counts, const int64_t *n_groups,
                                      int64_t capacity, void *scratch, size_t scratch_bytes, void *stream_)
{
    if (!keys || !sums || !counts || !n_groups || !scratch || capacity <= 0 || capacity > ((int64_t)1 << 31))
        return SJQ_ERR_INVALID_ARG;
    if (!aligned16(scratch) || (reinterpret_cast<uintptr_t>(keys) & 7u) || (reinterpret_cast<uintptr_t>(sums) & 7u) ||
        (reinterpret_cast<uintptr_t>(counts) & 7u) || (reinterpret_cast<uintptr_t>(n_groups) & 7u))
        return SJQ_ERR_ALIGN;
    const SortLayout L = sort_layout(capacity);
    if (scratch_bytes < L.total) return SJQ_ERR_BUFFER_SMALL;
    DeviceInfo dev;
    sjq_status st = device_info(&dev);
    if (st != SJQ_OK) return st;
    cudaStream_t stream = (cudaStream_t)stream_;
    char *base = static_cast<char *>(scratch);
    SortParams S{};
    S.n_groups = n_groups;
    S.capacity = capacity;
    S.keys = keys, S.sums = sums, S.counts = counts;
    S.k[0] = reinterpret_cast<unsigned long long *>(base + L.k0);
    S.k[1] = reinterpret_cast<unsigned long long *>(base + L.k1);
    S.p[0] = reinterpret_cast<unsigned int *>(base + L.p0);
    S.p[1] = reinterpret_cast<unsigned int *>(base + L.p1);
    S.tsums = reinterpret_cast<int64_t *>(base + L.tsums);
    S.tcounts = reinterpret_cast<int64_t *>(base + L.tcounts);
    S.ranges = reinterpret_cast<SortRange *>(base + L.ranges);
    S.header = reinterpret_cast<SortHeader *>(base + L.header);
    S.totals = reinterpret_cast<unsigned int *>(base + L.totals);
    S.hist = reinterpret_cast<unsigned int *>(base + L.hist);
    sort_range_kernel<<<L.nblocks, kSortThreads, 0, stream>>>(S);
    bool ok = cudaGetLastError() == cudaSuccess;
    for (int pass = 0; pass < kSortPasses && ok; ++pass) {
        S.pass = pass;
        ok = launch_behind(sort_hist_kernel, L.nblocks, S, stream) && launch_behind(sort_scatter_kernel, L.nblocks, S, stream);
    }
    if (!ok) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    return SJQ_OK;
}
