// Canonical order of a hashed result: ascending key.
//
// The global group table of Section 3.3 hands its groups back in table order, which depends on the hash function
// and on the capacity; two runs of the same query agree only as sets.  sjq_result_sort puts the list of
// (key, sum, count) triples into ascending signed key order on the device, equal keys as they came.
//
// The number of groups is known on the device only, so nothing waits on the host: the host enqueues the same kernels
// whatever the list holds, each launched while its predecessor still runs and waiting for it on the device
// (programmatic dependent launch), and a first kernel also finds out whether the list is in order already, in which
// case the others return at once.
//
// What bounds it: kernel latency.  A million pairs are 24 MB, which the L2 holds, so a kernel takes 3 to 15 us and it
// is the number of kernels one after the other that counts.  Two ways, by the capacity of the list:
//   - up to kSampleMost entries a sample sort, four or five kernels: splitters from a sorted sample; the bucket of every
//     entry, counted; the entries into their buckets; every bucket sorted in shared memory (merge of eight lists of
//     200,000 with its sort: 200 us with the radix sort, 106 with this one);
//   - beyond, a stable least-significant-digit radix sort of (key - smallest key, position) pairs, 8 bits a pass,
//     two kernels each; passes that the range of the keys does not need return at once.  At most kSortBlocks blocks
//     own one contiguous piece of the list each, so that the digit counts are few and every scatter block forms its
//     own offsets from them.
// Both copy the measures aside once and gather them in the last kernel, which writes all three result arrays.
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

constexpr int64_t kSampleMost = (int64_t)1 << 20;
constexpr int kBuckets = 1024;      // at most; about 256 entries each in a shorter list
constexpr int kOversample = 4;      // samples per bucket
constexpr int kBinMost = 64;        // entries of a bin that are compared with one another

// The blocks that sort the buckets, by the length of the list, which only the device knows: where the capacity is
// large both kernels are launched and one of them returns at once.  A bucket larger than the room in shared memory is
// ranked entry by entry, so it must be rare.  Bucket sizes depend on the ranks of the sampled entries alone, not on
// how the keys are spread, and a bucket of four samples exceeds x times the average with the tail of a gamma
// distribution of order four.  Little: four blocks of 256 threads per SM; at its longest the average bucket is a
// fifth of the room and one list in 300 has a larger one.  Large: one block of 1024 per SM; the average is at most an
// eighth, one list in 10^7.  (A million unordered entries: 2,300 us with the little blocks, which had forty such
// buckets in every list, 131 with the large ones, 253 with the radix sort; 430,000 entries 65 and 88.  Six samples a
// bucket instead of four: ranking them costs every list beyond 131,072 entries 12 us.)
template <int THREADS, int PER_SM, int ROOM_BITS, int BIN_BITS>
struct BucketBlocks {
    static constexpr int kThreads = THREADS, kPerSm = PER_SM;
    static constexpr bool kLarge = PER_SM == 1;
    static constexpr int kRoomBits = ROOM_BITS, kRoom = 1 << ROOM_BITS; // entries of a bucket that shared memory holds
    static constexpr int kBinBits = BIN_BITS, kBins = 1 << BIN_BITS;    // bins of a bucket
    static constexpr size_t kShared = (size_t)kRoom * (8 + 8 + 2);      // keys, a second array of words, numbers
};
typedef BucketBlocks<256, 4, 11, 11> LittleBlocks;
typedef BucketBlocks<1024, 1, 13, 12> LargeBlocks;
constexpr int64_t kLittleMost = (int64_t)kBuckets * (LittleBlocks::kRoom / 5);

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
    // sample sort
    unsigned long long *split_key; // [kBuckets - 1] splitters, ascending by (key, position)
    unsigned int *split_pos;
    unsigned int *bucket_total;    // [kBuckets] entries per bucket
    unsigned int *bucket_base;     // [blocks][kBuckets] places of a block's entries within their buckets
    unsigned int *disorder;        // [blocks] a key larger than its successor was seen
    int32_t pieces;                // blocks of the first three kernels
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
            const int t = threadIdx.x;
            offset[t] = incl - total + part[0][t] + part[1][t] + part[2][t] + part[3][t];
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

// ------------------------------------------------------------------ sample sort
__host__ __device__ __forceinline__ int buckets_for(int64_t n)
{
    int nb = 1;
    while (nb < kBuckets && (int64_t)nb * 256 < n) nb <<= 1;
    return nb;
}

// Position of sample i of s in a list of n: anywhere in the i-th of s equal parts, so that no regular pattern in the
// list meets the samples; samples ascend in position.
__host__ __device__ __forceinline__ int64_t sample_at(int i, int s, int64_t n)
{
    const int64_t lo = (int64_t)i * n / s, hi = (int64_t)(i + 1) * n / s;
    unsigned int h = (unsigned int)i * 2654435761u + 0x9E3779B9u;
    h ^= h >> 15;
    h *= 2246822519u;
    h ^= h >> 13;
    return lo + (int64_t)(h % (unsigned int)(hi - lo));
}

__device__ __forceinline__ bool list_in_order(const SortParams &S)
{
    int any = 0;
    for (int b = threadIdx.x; b < S.pieces; b += blockDim.x) any |= (int)S.disorder[b];
    return __syncthreads_or(any) == 0;
}

// Is the list in order, and the splitters: every block holds the sample and ranks its share of it, one per warp.
__global__ void __launch_bounds__(kSortThreads) sample_split_kernel(const __grid_constant__ SortParams S)
{
    __shared__ unsigned long long sample[kBuckets * kOversample];
    cudaTriggerProgrammaticLaunchCompletion();
    const int64_t n = sort_count(S);
    const int nb = buckets_for(n), ns = nb > 1 ? nb * kOversample : 0;
    for (int i = threadIdx.x; i < ns; i += kSortThreads) sample[i] = flip(S.keys[sample_at(i, ns, n)]);
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < kBuckets; i += kSortThreads) S.bucket_total[i] = 0;
    int64_t lo, hi;
    sort_piece(n, &lo, &hi);
    int disorder = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += kSortThreads)
        if (i + 1 < n && S.keys[i + 1] < S.keys[i]) disorder = 1;
    disorder = __syncthreads_or(disorder);
    if (threadIdx.x == 0) S.disorder[blockIdx.x] = (unsigned int)disorder;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = blockIdx.x * kSortWarps + warp; i < ns; i += gridDim.x * kSortWarps) {
        const unsigned long long k = sample[i];
        unsigned int before = 0;
        for (int j = lane; j < ns; j += 32) before += (sample[j] < k) | ((sample[j] == k) & (j < i));
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane == 0 && before % kOversample == 0 && before > 0) {
            S.split_key[before / kOversample - 1] = k;
            S.split_pos[before / kOversample - 1] = (unsigned int)sample_at(i, ns, n);
        }
    }
}

// The bucket of every entry of this block's piece (the number of splitters not above it) and its place among the
// block's entries of that bucket; the block's places within the buckets; the measures copied aside.
__global__ void __launch_bounds__(kSortThreads) sample_count_kernel(const __grid_constant__ SortParams S)
{
    __shared__ unsigned long long split_key[kBuckets];
    __shared__ unsigned int split_pos[kBuckets], count[kBuckets];
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    if (list_in_order(S)) return;
    const int64_t n = sort_count(S);
    const int nb = buckets_for(n);
    for (int i = threadIdx.x; i < nb; i += kSortThreads) {
        count[i] = 0;
        if (i < nb - 1) {
            split_key[i] = S.split_key[i];
            split_pos[i] = S.split_pos[i];
        }
    }
    __syncthreads();
    int64_t lo, hi;
    sort_piece(n, &lo, &hi);
    for (int64_t i = lo + threadIdx.x; i < hi; i += kSortThreads) {
        const unsigned long long k = flip(S.keys[i]);
        S.tsums[i] = S.sums[i];
        S.tcounts[i] = S.counts[i];
        int b = 0;
        for (int step = nb >> 1; step > 0; step >>= 1) {
            const unsigned long long sk = split_key[b + step - 1];
            if (sk < k || (sk == k && split_pos[b + step - 1] <= (unsigned int)i)) b += step;
        }
        const unsigned int at = atomicAdd(&count[b], 1u);
        static_assert(kSampleMost / kSortBlocks < (1 << 13) && kBuckets <= (1 << 10), "a place and a bucket fit one word");
        S.p[0][i] = (unsigned int)b << 16 | at;
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += kSortThreads)
        S.bucket_base[(size_t)blockIdx.x * kBuckets + b] = count[b] ? atomicAdd(&S.bucket_total[b], count[b]) : 0u;
}

// First entry of every bucket: exclusive scan of the totals by the first kBuckets / 4 threads of a block.
__device__ __forceinline__ void bucket_starts(const SortParams &S, int nb, unsigned int *start, unsigned int *warp_sum)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    unsigned int incl = 0;
    if (t < kBuckets / 4) {
        if (4 * t < nb) v = reinterpret_cast<const uint4 *>(S.bucket_total)[t]; // (totals beyond nb are zero)
        incl = v.x + v.y + v.z + v.w;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) warp_sum[warp] = incl;
    }
    __syncthreads();
    if (t < kBuckets / 4) {
        for (int w = 0; w < warp; ++w) incl += warp_sum[w];
        start[4 * t + 3] = incl - v.w;
        start[4 * t + 2] = incl - v.w - v.z;
        start[4 * t + 1] = incl - v.w - v.z - v.y;
        start[4 * t] = incl - v.w - v.z - v.y - v.x;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kSortThreads) sample_scatter_kernel(const __grid_constant__ SortParams S)
{
    __shared__ unsigned int place[kBuckets], warp_sum[kBuckets / 128];
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    if (list_in_order(S)) return;
    const int64_t n = sort_count(S);
    const int nb = buckets_for(n);
    int64_t lo, hi;
    sort_piece(n, &lo, &hi);
    if (lo >= hi) return;
    bucket_starts(S, nb, place, warp_sum);
    for (int b = threadIdx.x; b < nb; b += kSortThreads) place[b] += S.bucket_base[(size_t)blockIdx.x * kBuckets + b];
    __syncthreads();
    for (int64_t i = lo + threadIdx.x; i < hi; i += kSortThreads) {
        const unsigned int w = S.p[0][i], at = place[w >> 16] + (w & 0xFFFFu);
        S.k[1][at] = flip(S.keys[i]);
        S.p[1][at] = (unsigned int)i;
    }
}

// Smallest and largest key of a block's bucket.
template <class B>
__device__ __forceinline__ void block_range(unsigned long long &kmin, unsigned long long &kmax, unsigned long long *least,
                                            unsigned long long *most)
{
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, kmin, o), y = __shfl_xor_sync(0xffffffffu, kmax, o);
        kmin = x < kmin ? x : kmin;
        kmax = y > kmax ? y : kmax;
    }
    if ((threadIdx.x & 31) == 0) least[threadIdx.x >> 5] = kmin, most[threadIdx.x >> 5] = kmax;
    __syncthreads();
    for (int w = 0; w < B::kThreads / 32; ++w) {
        kmin = least[w] < kmin ? least[w] : kmin;
        kmax = most[w] > kmax ? most[w] : kmax;
    }
}

// Sort R * B::kThreads values by a bitonic network; value r * B::kThreads + thread sits in v[r].  Partners in the
// same thread or warp meet in registers, the others in shared memory.
template <class B, int R>
__device__ __forceinline__ void bitonic(unsigned long long (&v)[R], unsigned long long *buf)
{
    const int tid = threadIdx.x;
    for (int k = 2; k <= R * B::kThreads; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= B::kThreads) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
#pragma unroll
                    for (int o = 1; o < R; o <<= 1) {
                        if (o * B::kThreads != j || (r & o)) continue;
                        const bool up = ((r * B::kThreads) & k) == 0;
                        const unsigned long long a = v[r], b = v[r | o], lo = a < b ? a : b, hi = a < b ? b : a;
                        v[r] = up ? lo : hi;
                        v[r | o] = up ? hi : lo;
                    }
                }
                continue;
            }
            unsigned long long other[R];
            if (j >= 32) {
                __syncthreads(); // what was read the last time
#pragma unroll
                for (int r = 0; r < R; ++r) buf[r * B::kThreads + tid] = v[r];
                __syncthreads();
#pragma unroll
                for (int r = 0; r < R; ++r) other[r] = buf[r * B::kThreads + (tid ^ j)];
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) other[r] = __shfl_xor_sync(0xffffffffu, v[r], j);
            }
            const bool low = (tid & j) == 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool up = ((r * B::kThreads + tid) & k) == 0, least = low == up;
                v[r] = (v[r] < other[r]) == least ? v[r] : other[r];
            }
        }
    }
}

// Order of a bucket's m <= R * B::kThreads entries: order[i] = the entry that comes i-th.  The values sorted are the
// top bits of the distance from the bucket's smallest key, then the entry's number: one word instead of key and
// position.  False when two neighbours agree in those bits.
template <class B, int R>
__device__ __forceinline__ bool order_bucket(const unsigned long long *key, int m, unsigned long long kmin, int shift,
                                             unsigned long long *buf, unsigned short *order)
{
    constexpr int kNumberBits = B::kRoomBits;
    unsigned long long v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = r * B::kThreads + (int)threadIdx.x;
        v[r] = e < m ? ((key[e] - kmin) >> shift) << kNumberBits | (unsigned long long)e : ~0ull;
    }
    bitonic<B, R>(v, buf);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) buf[r * B::kThreads + threadIdx.x] = v[r];
    __syncthreads();
    bool same = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = r * B::kThreads + (int)threadIdx.x;
        if (e >= m) continue;
        order[e] = (unsigned short)(v[r] & ((1u << kNumberBits) - 1u));
        same |= e + 1 < m && (buf[e + 1] ^ v[r]) >> kNumberBits == 0;
    }
    return __syncthreads_or(same) == 0;
}

// A bucket's m entries by one more distribution: bins of equal width over the bucket's range, as many as shared memory
// holds entries, so that most bins take one or none; an entry's place is its bin's start plus the smaller entries of
// its bin.  Half a dozen barriers where the network has one pair per step (lists of 400,000 entries: merge and sort
// 127 us with the network, 106 with the bins; three waves of the network's blocks took 43 of them).  Registers are
// kept to four blocks per SM: with five, measures spill and it takes 112.  R > 0: m <= R * B::kThreads, and a
// thread's entries stay in registers, keys and measures requested before the first wait; R = 0: any m <= B::kRoom,
// keys read again (from the L1) in each pass.  False, with nothing written, when a bin takes more than kBinMost
// entries (keys bunched within the bucket).
template <class B, int R>
__device__ __forceinline__ bool bin_bucket(const SortParams &S, unsigned int lo, int m, unsigned long long *key,
                                           unsigned int *bin, unsigned int *pos, unsigned short *number,
                                           unsigned long long *least, unsigned long long *most, unsigned int *warp_sum)
{
    constexpr int kBins = B::kBins, kPerThread = kBins / B::kThreads, kKept = R > 0 ? R : 1;
    static_assert(kPerThread % 4 == 0, "whole 128-bit words");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long k[kKept], kmin = ~0ull, kmax = 0ull;
    unsigned int p[kKept];
    int64_t sum[kKept], count[kKept];
    if (R > 0) {
#pragma unroll
        for (int r = 0; r < kKept; ++r) {
            const int e = r * B::kThreads + tid;
            if (e < m) k[r] = S.k[1][lo + e], p[r] = S.p[1][lo + e];
        }
#pragma unroll
        for (int r = 0; r < kKept; ++r)
            if (r * B::kThreads + tid < m) sum[r] = S.tsums[p[r]], count[r] = S.tcounts[p[r]];
    }
    auto entries = [&](auto &&f) { // f(slot, entry, its key) for every entry of this thread
        if (R > 0) {
#pragma unroll
            for (int r = 0; r < kKept; ++r)
                if (r * B::kThreads + tid < m) f(r, r * B::kThreads + tid, k[r]);
        } else {
#pragma unroll 1
            for (int e = tid; e < m; e += B::kThreads) f(0, e, S.k[1][lo + e]);
        }
    };
    uint4 *words = reinterpret_cast<uint4 *>(bin) + tid * (kPerThread / 4);
#pragma unroll
    for (int q = 0; q < kPerThread / 4; ++q) words[q] = make_uint4(0u, 0u, 0u, 0u);
    entries([&](int, int, unsigned long long x) {
        kmin = x < kmin ? x : kmin;
        kmax = x > kmax ? x : kmax;
    });
    block_range<B>(kmin, kmax, least, most);
    const int bits = 64 - __clzll((long long)(kmax - kmin)), shift = bits > B::kBinBits ? bits - B::kBinBits : 0;
    entries([&](int, int e, unsigned long long x) {
        number[e] = (unsigned short)atomicAdd(&bin[(x - kmin) >> shift], 1u);
    });
    __syncthreads();
    unsigned int mine = 0, largest = 0;
#pragma unroll
    for (int q = 0; q < kPerThread / 4; ++q) {
        const uint4 w = words[q];
        mine += w.x + w.y + w.z + w.w;
        largest = max(max(max(largest, w.x), max(w.y, w.z)), w.w);
    }
    unsigned int first = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int u = __shfl_up_sync(0xffffffffu, first, o);
        if (lane >= o) first += u;
    }
    if (lane == 31) warp_sum[warp] = first;
    if (__syncthreads_or(largest > (unsigned int)kBinMost)) return false;
    first -= mine;
    for (int w = 0; w < warp; ++w) first += warp_sum[w];
#pragma unroll
    for (int q = 0; q < kPerThread / 4; ++q) {
        const uint4 w = words[q];
        words[q] = make_uint4(first, first + w.x, first + w.x + w.y, first + w.x + w.y + w.z);
        first += w.x + w.y + w.z + w.w;
    }
    __syncthreads();
    entries([&](int r, int e, unsigned long long x) {
        const unsigned int i = bin[(x - kmin) >> shift] + number[e];
        key[i] = x;
        pos[i] = R > 0 ? p[r] : S.p[1][lo + e];
    });
    __syncthreads();
    entries([&](int r, int e, unsigned long long x) {
        const unsigned int d = (unsigned int)((x - kmin) >> shift), i0 = bin[d];
        const unsigned int i1 = d + 1 < (unsigned int)kBins ? bin[d + 1] : (unsigned int)m;
        const unsigned int from = R > 0 ? p[r] : pos[i0 + number[e]];
        unsigned int place = lo + i0;
        for (unsigned int i = i0; i < i1; ++i) place += (key[i] < x) | ((key[i] == x) & (pos[i] < from));
        S.keys[place] = (int64_t)(x ^ 0x8000000000000000ull);
        S.sums[place] = R > 0 ? sum[r] : S.tsums[from];
        S.counts[place] = R > 0 ? count[r] : S.tcounts[from];
    });
    return true;
}

// Sort the buckets, a block each: by bins, or by the network where the keys are bunched.  Where bunched keys are equal,
// or so far apart that the top bits do not tell them apart, or a bucket is larger than shared memory (an unlucky
// sample), its entries are ranked one by one against the whole bucket.
template <class B>
__global__ void __launch_bounds__(B::kThreads, B::kPerSm) sample_bucket_kernel(const __grid_constant__ SortParams S)
{
    extern __shared__ __align__(16) unsigned long long key[]; // B::kShared bytes
    unsigned long long *const buf = key + B::kRoom;
    unsigned short *const order = reinterpret_cast<unsigned short *>(buf + B::kRoom);
    __shared__ unsigned int start[kBuckets], warp_sum[B::kThreads / 32];
    __shared__ unsigned long long least[B::kThreads / 32], most[B::kThreads / 32];
    static_assert(B::kThreads >= kBuckets / 4, "bucket_starts takes so many threads");
    static_assert(8 * (size_t)B::kRoom >= 4 * (size_t)(B::kBins + B::kRoom), "bins and positions fit beside the keys");
    cudaGridDependencySynchronize();
    const int64_t n = sort_count(S);
    const bool ordered = list_in_order(S);
    if (ordered || B::kLarge != (n > kLittleMost)) return;
    const int nb = buckets_for(n);
    bucket_starts(S, nb, start, warp_sum);
    auto store = [&](unsigned int at, unsigned long long k, unsigned int p) {
        S.keys[at] = (int64_t)(k ^ 0x8000000000000000ull);
        S.sums[at] = S.tsums[p];
        S.counts[at] = S.tcounts[p];
    };
    for (int b = blockIdx.x; b < nb; b += gridDim.x) {
        const unsigned int lo = start[b], m = S.bucket_total[b];
        if (m == 0) continue;
        bool done = false;
        unsigned int *const bin = reinterpret_cast<unsigned int *>(buf), *const pos = bin + B::kBins;
        __syncthreads(); // the bucket before has been written out
        if (m <= B::kThreads) done = bin_bucket<B, 1>(S, lo, (int)m, key, bin, pos, order, least, most, warp_sum);
        else if (m <= 2 * B::kThreads) done = bin_bucket<B, 2>(S, lo, (int)m, key, bin, pos, order, least, most, warp_sum);
        else if (m <= (unsigned int)B::kRoom)
            done = bin_bucket<B, 0>(S, lo, (int)m, key, bin, pos, order, least, most, warp_sum);
        if (done) continue;
        if (m <= (unsigned int)B::kRoom) {
            __syncthreads(); // the bins have been read
            unsigned long long kmin = ~0ull, kmax = 0ull;
            for (int e = threadIdx.x; e < (int)m; e += B::kThreads) {
                const unsigned long long k = S.k[1][lo + e];
                key[e] = k;
                kmin = k < kmin ? k : kmin;
                kmax = k > kmax ? k : kmax;
            }
            block_range<B>(kmin, kmax, least, most);
            // (a distance of all ones would meet the padding: one bit less than the entry's number leaves)
            constexpr int kDistance = 63 - B::kRoomBits;
            const int bits = 64 - __clzll((long long)(kmax - kmin)), shift = bits > kDistance ? bits - kDistance : 0;
            if (m <= B::kThreads) done = order_bucket<B, 1>(key, (int)m, kmin, shift, buf, order);
            else if (m <= 2 * B::kThreads) done = order_bucket<B, 2>(key, (int)m, kmin, shift, buf, order);
            else if (m <= 4 * B::kThreads) done = order_bucket<B, 4>(key, (int)m, kmin, shift, buf, order);
            else done = order_bucket<B, 8>(key, (int)m, kmin, shift, buf, order);
            if (done)
                for (int e = threadIdx.x; e < (int)m; e += B::kThreads) store(lo + e, key[order[e]], S.p[1][lo + order[e]]);
        }
        if (done) continue;
        for (unsigned int e = threadIdx.x; e < m; e += B::kThreads) {
            const unsigned long long k = S.k[1][lo + e];
            const unsigned int p = S.p[1][lo + e];
            unsigned int before = 0;
            for (unsigned int j = 0; j < m; ++j) {
                const unsigned long long o = S.k[1][lo + j];
                before += (o < k) | ((o == k) & (S.p[1][lo + j] < p));
            }
            store(lo + before, k, p);
        }
    }
}

size_t up256(size_t v) { return (v + 255) / 256 * 256; }

struct SortLayout {
    size_t k0, k1, p0, p1, ranges, header, totals, hist, tsums, tcounts, split_key, split_pos, bucket_total, disorder, total;
    int nblocks;
    bool sample;
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
    L.hist = at, at += (size_t)kBuckets * L.nblocks * 4; // (the radix sort's 256 counts per block, or bucket_base)
    L.split_key = at, at += (size_t)kBuckets * 8;
    L.split_pos = at, at += (size_t)kBuckets * 4;
    L.bucket_total = at, at += (size_t)kBuckets * 4;
    L.disorder = at, at += up256((size_t)kSortBlocks * 4);
    L.sample = capacity <= kSampleMost;
    L.tsums = at, at += up256(c * 8);
    L.tcounts = at, at += up256(c * 8);
    L.total = at;
    return L;
}

// Launch behind the previous kernel of the sort without waiting for it: every kernel but the first waits on the
// device (cudaGridDependencySynchronize) before it touches what its predecessors wrote.
bool launch_behind(void (*kernel)(SortParams), int grid, int threads, const SortParams &S, cudaStream_t stream,
                   size_t shared = 0)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = shared;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, S) == cudaSuccess;
}

template <class B>
bool launch_buckets(int64_t most, const SortParams &S, cudaStream_t stream)
{
    void (*const kernel)(SortParams) = sample_bucket_kernel<B>;
    if (B::kShared > ((size_t)40 << 10) &&
        cudaFuncSetAttribute(reinterpret_cast<const void *>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)B::kShared) != cudaSuccess)
        return false;
    const int64_t buckets = std::min<int64_t>((S.capacity + 127) / 128, most);
    return launch_behind(kernel, (int)buckets, B::kThreads, S, stream, B::kShared);
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
    S.split_key = reinterpret_cast<unsigned long long *>(base + L.split_key);
    S.split_pos = reinterpret_cast<unsigned int *>(base + L.split_pos);
    S.bucket_total = reinterpret_cast<unsigned int *>(base + L.bucket_total);
    S.bucket_base = S.hist;
    S.disorder = reinterpret_cast<unsigned int *>(base + L.disorder);
    S.pieces = L.nblocks;
    bool ok;
    if (L.sample) {
        sample_split_kernel<<<L.nblocks, kSortThreads, 0, stream>>>(S);
        ok = cudaGetLastError() == cudaSuccess && launch_behind(sample_count_kernel, L.nblocks, kSortThreads, S, stream) &&
             launch_behind(sample_scatter_kernel, L.nblocks, kSortThreads, S, stream) &&
             launch_buckets<LittleBlocks>(kBuckets, S, stream) &&
             (capacity <= kLittleMost || launch_buckets<LargeBlocks>(kSortBlocks, S, stream));
    } else {
        sort_range_kernel<<<L.nblocks, kSortThreads, 0, stream>>>(S);
        ok = cudaGetLastError() == cudaSuccess;
        for (int pass = 0; pass < kSortPasses && ok; ++pass) {
            S.pass = pass;
            ok = launch_behind(sort_hist_kernel, L.nblocks, kSortThreads, S, stream) &&
                 launch_behind(sort_scatter_kernel, L.nblocks, kSortThreads, S, stream);
        }
    }
    if (!ok) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    return SJQ_OK;
}

// The sampler as the kernels use it, for tests on the host (not part of the interface): the positions sampled in a list
// of n entries (`positions` NULL: none are written); returns their number.  `room`: entries of a bucket that shared
// memory holds; `little`, `most`: the longest lists of the two forms of the sample sort.
extern "C" int32_t sjq_result_sort_samples(int64_t n, int64_t *positions, int32_t *per_bucket, int32_t *room,
                                           int64_t *little, int64_t *most)
{
    const int nb = buckets_for(n), ns = nb > 1 ? nb * kOversample : 0;
    for (int i = 0; positions && i < ns; ++i) positions[i] = sample_at(i, ns, n);
    *per_bucket = kOversample;
    *room = n <= kLittleMost ? LittleBlocks::kRoom : LargeBlocks::kRoom;
    *little = kLittleMost;
    *most = kSampleMost;
    return ns;
}
