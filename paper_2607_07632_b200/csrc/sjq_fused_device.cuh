// The fused probe kernel: one pass over the fact table.
//
// Execution model.  A machine-sized grid of persistent blocks strides over
// tiles of the fact table (Section 3.2 of the paper, "grid-stride persistent
// threads").  Every warp runs a small push pipeline of its own:
//
//  level 0   (dense) every thread owns kSlots groups of four consecutive
//            rows, so one 128-bit load brings four values of the first
//            column and a warp reads 512 contiguous bytes; the first stage
//            keeps one bit per row.  The sixteen loads and probes of a thread
//            are independent, which keeps enough bytes in flight to cover
//            HBM latency.
//  level l   the survivors of level l-1 are compacted (popcount + warp scan)
//            into queue l of the warp in shared memory; whenever a queue
//            holds a full batch (kRows per lane) the warp runs the next filter
//            stage on it, loading that stage's column with one 4-byte load per
//            surviving row only (lazy loading, Section 3.2: a later column is
//            never read for an eliminated row), and pushes the survivors on.
//  last      the final level gathers the group-key payloads and the measure
//            columns of the survivors into register accumulators and runs the
//            terminal.
//
// A probe is a range-checked single load from a direct-mapped table (global or
// staged in shared memory) or a bounded lock-step linear probe of an
// open-addressing table (Section 3.3).  The terminal is a register accumulator
// with one atomic per block, a shared-memory privatised group table flushed
// with one atomic per touched group per block, global atomics, or a global
// group hash table (Section 3.3 "Shared-memory privatized group-by").
#ifndef SJQ_FUSED_DEVICE_CUH
#define SJQ_FUSED_DEVICE_CUH

#include "sjq_run.cuh"

// Two ways to build this code.  Ahead of time the query's shape is data: stage descriptors sit in
// shared memory and every stage is dispatched by a uniform switch.  With SJQ_JIT the file is
// compiled at run time for one query shape (the analogue of the paper's composition-based fusion,
// Section 4.2): "sjq_jit_shape.h", generated by the host, defines the shape as constants, the stage
// loops unroll, the switches fold and only the stage bodies the query uses remain.  Values that
// depend on the data (key ranges, thresholds, table sizes, pointers) stay kernel parameters.
#if defined(SJQ_JIT)
#include "sjq_jit_shape.h"
#define SJQ_PV(f) (SJQ_JIT_##f)
#define SJQ_STAGE(s) jit_stage(P, (s))
#define SJQ_UNROLL_STAGES _Pragma("unroll")
#else
#define SJQ_PV(f) (P.f)
#define SJQ_STAGE(s) st[(s)]
#define SJQ_UNROLL_STAGES
#endif

#ifndef SJQ_LB_THREADS
#define SJQ_LB_THREADS 384
#define SJQ_LB_BLOCKS 2
#endif

namespace sjq {

namespace {

// The parameter block as the functions below see it: a compiled kernel's stages are parameters like the rest, the
// interpreting kernels pass theirs along as a copy in shared memory.
#if defined(SJQ_JIT)
typedef RunParams RunArg;
#else
typedef RunCore RunArg;
#endif

// 256-bit global loads exist from CUDA 12.9 on (the compiler that builds this file, ahead of time or at run time)
#if (__CUDACC_VER_MAJOR__ > 12) || (__CUDACC_VER_MAJOR__ == 12 && __CUDACC_VER_MINOR__ >= 9)
#define SJQ_HAVE_LOAD256 1
#else
#define SJQ_HAVE_LOAD256 0
#endif
constexpr bool kLoad256 = SJQ_HAVE_LOAD256 != 0;

// Four consecutive values of a column.  `aligned`: the column starts on a 32-byte boundary.
template <typename T>
struct Vec4;
template <>
struct Vec4<int32_t> {
    static __device__ __forceinline__ void load(const int32_t *p, int32_t *v, bool)
    {
        // read once: leave the L1 to the dimension tables
        asm volatile("ld.global.nc.L1::no_allocate.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                     : "l"(p));
    }
};
template <>
struct Vec4<int64_t> {
    static __device__ __forceinline__ void load(const int64_t *p, int64_t *v, bool aligned)
    {
        // One 256-bit load: two 128-bit loads of neighbouring lanes would each touch every sector of the 1024 bytes,
        // and the L1 passes one sector per cycle (the skewed 64-bit-key workload, bound by it, 300 M rows, both loads
        // in turn three times: 1800 -> 1690, 1832 -> 1717 and 1781 -> 1680 us; asked once of the interpreting kernel,
        // 10 M rows: 274 and 273).
#if SJQ_HAVE_LOAD256
        if (aligned) {
            asm volatile("ld.global.nc.L1::no_allocate.v4.b64 {%0, %1, %2, %3}, [%4];"
                         : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3])
                         : "l"(p));
            return;
        }
#endif
        asm volatile("ld.global.nc.L1::no_allocate.v2.b64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "l"(p));
        asm volatile("ld.global.nc.L1::no_allocate.v2.b64 {%0, %1}, [%2];" : "=l"(v[2]), "=l"(v[3]) : "l"(p + 2));
    }
};

// One value of a later column for one surviving row.  The load asks L2 to fetch no more than 64
// bytes around it: with the default, a lone survivor pulled in up to 256 bytes of a column that
// nothing else would use (measured on the four-join workload: 16.8 -> 13.4 bytes of DRAM traffic per
// fact row).
// ... and it does not claim an L1 line: the value is used once, the L1 is for the dimension tables.
__device__ __forceinline__ int32_t ld_sparse(const int32_t *p)
{
    int32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::64B.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int64_t ld_sparse(const int64_t *p)
{
    int64_t v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::64B.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

template <typename T>
struct Index {
    typedef uint64_t type;
};
template <>
struct Index<int32_t> {
    typedef uint32_t type;
};

// ------------------------------------------------------------------ stage bodies
// Each body takes the values v[0..NR) of the rows whose bit is set in m and
// returns the mask of rows that pass.  Values of rows outside m are ignored.

template <typename T, int NR>
__device__ __forceinline__ uint32_t body_pred_range(const DStage &S, const T (&v)[NR], uint32_t m)
{
    uint32_t pass = 0;
    if (sizeof(T) == 4) {
        if (!S.never) {
#pragma unroll
            for (int i = 0; i < NR; ++i)
                pass |= (uint32_t)(((uint32_t)v[i] - (uint32_t)S.lo32) <= S.width32) << i;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NR; ++i) pass |= (uint32_t)(((int64_t)v[i] >= S.lo) & ((int64_t)v[i] <= S.hi)) << i;
    }
    if (S.neg) pass = ~pass;
    return m & pass;
}

template <typename T, int NR>
__device__ __forceinline__ uint32_t body_pred_set(const RunArg &P, const DStage &S, const T (&v)[NR], uint32_t m)
{
    uint32_t pass = 0;
    for (int k = 0; k < S.nset; ++k) {
        const int64_t lit = P.sets[S.set_idx][k];
#pragma unroll
        for (int i = 0; i < NR; ++i) pass |= (uint32_t)((int64_t)v[i] == lit) << i;
    }
    return m & pass;
}

// A word of a direct-mapped table, `at` words from its start: from the copy in shared memory, from global memory, or, where
// the copy is the first part of a larger table (kTabPart), from either.
struct TablePlaces {
    const unsigned char *global, *shared;
    uint32_t held; // bytes of the copy
};
template <int WHERE, typename W, typename I>
__device__ __forceinline__ W table_word(const TablePlaces &T, I at)
{
    if (WHERE == kTabShared || (WHERE == kTabPart && at < (I)(T.held / sizeof(W)))) return reinterpret_cast<const W *>(T.shared)[at];
    return __ldg(reinterpret_cast<const W *>(T.global) + at);
}

template <typename T, int OP, int WHERE, int NR, bool WANT, typename C>
__device__ __forceinline__ uint32_t body_direct(const DStage &S, const unsigned char *smem, const T (&v)[NR],
                                                uint32_t m, C (&code)[NR])
{
    // (formed once: an ahead-of-time kernel would read the descriptor at every row, four joins asked once 252 -> 262 us)
    const TablePlaces places{WHERE == kTabShared ? nullptr : static_cast<const unsigned char *>(S.tab),
                         WHERE == kTabGlobal ? nullptr : smem + S.smem_off, WHERE == kTabPart ? S.tab_bytes : 0u};
    // A key outside the table's range is a miss, never an out-of-range access: its index is clamped to the
    // spare entry after the last slot, which is never set (one min instead of a range test and a mask).
    typename Index<T>::type idx[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        if (sizeof(T) == 4) {
            const uint32_t d = (uint32_t)v[i] - (uint32_t)S.kmin32;
            idx[i] = d < S.clamp32 ? d : S.clamp32;
        } else {
            const uint64_t d = (uint64_t)v[i] - (uint64_t)S.kmin;
            idx[i] = d <= S.last ? d : S.last + 1;
        }
    }
    uint32_t hit = 0;
    if constexpr (OP == OP_DIRECT_BITMAP) {
        uint32_t w[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            w[i] = 0;
            if ((m >> i) & 1u) w[i] = table_word<WHERE, uint32_t>(places, idx[i] >> 5);
        }
        // rotate the wanted bit of the word straight into position i of the mask (the funnel shift takes its
        // amount modulo 32): subtract, rotate, and-or
#pragma unroll
        for (int i = 0; i < NR; ++i) hit |= __funnelshift_r(w[i], w[i], (uint32_t)idx[i] - (uint32_t)i) & (1u << i);
        return m & hit;
    } else if constexpr (OP == OP_DIRECT_U4 || OP == OP_DIRECT_U2) {
        // sub-byte codes: eight (sixteen) to a 32-bit word.  All ones is the miss marker, except in a table
        // that holds every key of its range: there the range test (the clamp) alone decides.
        constexpr int BITS = OP == OP_DIRECT_U4 ? 4 : 2;
        constexpr uint32_t PER = 32 / BITS, MASK = (1u << BITS) - 1u;
        uint32_t w[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            w[i] = ~0u;
            if ((m >> i) & 1u) w[i] = table_word<WHERE, uint32_t>(places, idx[i] / PER);
        }
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const uint32_t c = (w[i] >> (((uint32_t)idx[i] % PER) * BITS)) & MASK;
            bool ok;
            if (S.full) ok = sizeof(T) == 4 ? (uint32_t)idx[i] != S.clamp32 : (uint64_t)idx[i] <= S.last;
            else ok = c != MASK;
            hit |= (uint32_t)ok << i;
            if (WANT) code[i] = c;
        }
        return m & hit;
    } else {
        // (codes stay in the caller's word: a compiled kernel, whose words have 64 bits, takes 86.3 us with 32-bit ones
        // here and 84.4 without, two joins, 60 M rows)
        C c[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            c[i] = (C)~0ULL;
            if ((m >> i) & 1u) {
                if (OP == OP_DIRECT_U8) c[i] = table_word<WHERE, uint8_t>(places, idx[i]);
                else if (OP == OP_DIRECT_U16) c[i] = table_word<WHERE, uint16_t>(places, idx[i]);
                else if (OP == OP_DIRECT_U32) c[i] = table_word<WHERE, uint32_t>(places, idx[i]);
                else c[i] = (C)table_word<WHERE, uint64_t>(places, idx[i]);
            }
        }
        const C miss = OP == OP_DIRECT_U8 ? (C)0xFFull : OP == OP_DIRECT_U16 ? (C)0xFFFFull
                       : OP == OP_DIRECT_U32 ? (C)0xFFFFFFFFull : (C)~0ULL;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            hit |= (uint32_t)(c[i] != miss) << i;
            if (WANT) code[i] = c[i];
        }
        return m & hit;
    }
}

// Hot-key table of an open-addressing join, held in shared memory: 0 = the key is not held, 1 = it is in the
// dimension table (*code receives its payload code), 2 = it is absent.  The table is direct-mapped and read-only
// during the run; entry kHotSlots is its header (first word: keys held; zero = skip the look-ups).
__device__ __forceinline__ bool hot_in_use(const DStage &S, const unsigned char *smem)
{
    return S.hot && *reinterpret_cast<const uint32_t *>(smem + S.hot_off + (uint32_t)kHotSlots * 16u) != 0u;
}
__device__ __forceinline__ uint32_t hot_lookup(const DStage &S, const unsigned char *smem, uint64_t key, uint32_t *code)
{
    const uint4 e = *reinterpret_cast<const uint4 *>(smem + S.hot_off + ((hot_hash(key) & (uint32_t)(kHotSlots - 1)) << 4));
    *code = e.z;
    return (e.x == (uint32_t)key && e.y == (uint32_t)(key >> 32)) ? e.w : 0u;
}

// Open addressing over 32-byte buckets (K keys, then their K codes): a key's linear probe starts at its
// home bucket, a lookup loads one whole bucket per step (two 128-bit loads: only the key part when the
// codes are not wanted), compares every key in it, and stops at a match or at the first bucket with a
// free slot.  A hit finds its code in the words already loaded: one sector per probe step.  The rows of a
// chunk advance in lock step so that their loads overlap; bounded by the bucket count.
template <typename T, int CB, int NR, bool WANT, typename C>
__device__ __forceinline__ uint32_t body_hash(const DStage &S, const unsigned char *smem, const T (&v)[NR], uint32_t m,
                                              C (&code)[NR])
{
    constexpr int KB = (int)sizeof(T);
    constexpr int K = bucket_keys(KB, CB);
    constexpr int CODE_WORD = bucket_code_offset(KB, CB, K) / 4;
    constexpr int PIECES = (WANT && CB) ? kBucketBytes / 16 : (K * KB + 15) / 16; // 16-byte pieces to read
    constexpr int CH = NR < 2 ? NR : 2;                                            // rows advancing together
    const T empty = sizeof(T) == 4 ? (T)kEmptyKey32 : (T)kEmptyKey64;
    const uint4 *table = static_cast<const uint4 *>(S.tab);
    const uint32_t nb = (uint32_t)S.last; // number of buckets
    uint32_t hit = 0;
#pragma unroll
    for (int i = 0; i < NR; ++i) code[i] = 0;
    if (CB != 8 && hot_in_use(S, smem)) {
        // rows whose key the hot table holds are answered from shared memory and leave the probe
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            if ((m >> i) & 1u) {
                uint32_t c;
                const uint32_t state = hot_lookup(S, smem, (uint64_t)(int64_t)v[i], &c);
                if (state != 0u) m &= ~(1u << i);
                if (state == 1u) {
                    hit |= 1u << i;
                    if (WANT) code[i] = c;
                }
            }
        }
    }
#pragma unroll
    for (int base = 0; base < NR; base += CH) {
        uint32_t bucket[CH];
        uint32_t pending = 0;
#pragma unroll
        for (int i = 0; i < CH; ++i) {
            bucket[i] = home_bucket((uint64_t)(int64_t)v[base + i], nb);
            pending |= (uint32_t)(((m >> (base + i)) & 1u) && v[base + i] != empty) << i; // the marker is never a key
        }
        for (uint32_t it = 0; pending != 0 && it < nb; ++it) {
            uint32_t u[CH][PIECES * 4];
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                if (kLoad256 && PIECES == 2 && S.wide) {
                    // the whole bucket in one 256-bit load: a random load costs the L1 the same whether it brings 16
                    // or 32 bytes (measured: 250-280 G buckets/s against 129-135 G with two 128-bit loads)
#pragma unroll
                    for (int q = 0; q < 8; ++q) u[i][q] = 0u;
#if SJQ_HAVE_LOAD256
                    if ((pending >> i) & 1u)
                        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                                     : "=r"(u[i][0]), "=r"(u[i][1]), "=r"(u[i][2]), "=r"(u[i][3]), "=r"(u[i][4]),
                                       "=r"(u[i][5]), "=r"(u[i][6]), "=r"(u[i][7])
                                     : "l"(table + (size_t)bucket[i] * (kBucketBytes / 16)));
#endif
                } else {
#pragma unroll
                    for (int q = 0; q < PIECES; ++q) {
                        uint4 w = make_uint4(0u, 0u, 0u, 0u);
                        if ((pending >> i) & 1u) w = __ldg(table + (size_t)bucket[i] * (kBucketBytes / 16) + q);
                        u[i][4 * q] = w.x, u[i][4 * q + 1] = w.y, u[i][4 * q + 2] = w.z, u[i][4 * q + 3] = w.w;
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                if ((pending >> i) & 1u) {
                    bool found = false, has_free = false;
                    C c = 0;
#pragma unroll
                    for (int j = 0; j < K; ++j) {
                        T kj;
                        if (sizeof(T) == 4) kj = (T)u[i][j];
                        else kj = (T)(((uint64_t)u[i][2 * j + 1] << 32) | u[i][2 * j]);
                        if (kj == v[base + i]) {
                            found = true;
                            if (WANT && CB == 4) c = u[i][CODE_WORD + j];
                            if (WANT && CB == 8) c = (C)(((uint64_t)u[i][CODE_WORD + 2 * j + 1] << 32) | u[i][CODE_WORD + 2 * j]);
                        }
                        has_free |= kj == empty;
                    }
                    if (found) {
                        hit |= 1u << (base + i);
                        if (WANT) code[base + i] = c;
                        pending &= ~(1u << i);
                    } else if (has_free) {
                        pending &= ~(1u << i);
                    } else {
                        bucket[i] = bucket[i] + 1 == nb ? 0 : bucket[i] + 1;
                    }
                }
            }
        }
    }
    return hit;
}

// Presence bitmap of an open-addressing table: one bit per hash value; a clear bit proves the key
// absent, a set bit sends the row on to the exact probe.
template <typename T, int NR>
__device__ __forceinline__ uint32_t body_hashbits(const DStage &S, const unsigned char *smem, const T (&v)[NR],
                                                  uint32_t m)
{
    const uint32_t *bits = static_cast<const uint32_t *>(S.tab);
    const uint32_t fmask = (uint32_t)S.hmask;
    uint32_t known = 0; // rows the hot table answers: present ones pass without touching the bitmap
    if (hot_in_use(S, smem)) {
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            if ((m >> i) & 1u) {
                uint32_t c;
                const uint32_t state = hot_lookup(S, smem, (uint64_t)(int64_t)v[i], &c);
                if (state != 0u) m &= ~(1u << i);
                if (state == 1u) known |= 1u << i;
            }
        }
    }
    uint32_t w[NR], idx[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        idx[i] = filter_hash((uint64_t)(int64_t)v[i]) & fmask;
        w[i] = 0;
        if ((m >> i) & 1u) w[i] = __ldg(bits + (idx[i] >> 5));
    }
    uint32_t hit = 0;
#pragma unroll
    for (int i = 0; i < NR; ++i) hit |= __funnelshift_r(w[i], w[i], idx[i] - (uint32_t)i) & (1u << i);
    hit &= m;
    return hit | known;
}

// C: the word codes are held in.  With 32 bits there are no 64-bit codes; the tables of 32-bit keys are direct, those of
// 64-bit keys (HASH) open-addressing, and nothing else filters on a 64-bit column.
template <typename T, int NR, bool WANT, bool HASH, typename C>
__device__ __forceinline__ uint32_t run_stage(const RunArg &P, const DStage &S, const unsigned char *smem,
                                              const T (&v)[NR], uint32_t m, C (&code)[NR])
{
    constexpr bool kWide = sizeof(C) == 8;
    if constexpr (!kWide && sizeof(T) == 8) {
        if (S.op == OP_HASHBITS) return body_hashbits<T, NR>(S, smem, v, m);
        if (S.op != OP_HASH64) return m; // OP_LOAD
        return S.code_bits == 0 ? body_hash<T, 0, NR, WANT>(S, smem, v, m, code) : body_hash<T, 4, NR, WANT>(S, smem, v, m, code);
    }
#if defined(SJQ_JIT)
    if (S.in_smem == kTabPart) {
        switch (S.op) {
        case OP_DIRECT_BITMAP: return body_direct<T, OP_DIRECT_BITMAP, kTabPart, NR, WANT>(S, smem, v, m, code);
        case OP_DIRECT_U2: return body_direct<T, OP_DIRECT_U2, kTabPart, NR, WANT>(S, smem, v, m, code);
        case OP_DIRECT_U4: return body_direct<T, OP_DIRECT_U4, kTabPart, NR, WANT>(S, smem, v, m, code);
        default: return body_direct<T, OP_DIRECT_U8, kTabPart, NR, WANT>(S, smem, v, m, code); // (no wider codes)
        }
    }
#endif
    switch (S.op * 2 + S.in_smem) {
    case OP_PRED_RANGE * 2: return body_pred_range<T, NR>(S, v, m);
    case OP_PRED_SET * 2: return body_pred_set<T, NR>(P, S, v, m);
    case OP_DIRECT_BITMAP * 2: return body_direct<T, OP_DIRECT_BITMAP, kTabGlobal, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_BITMAP * 2 + 1: return body_direct<T, OP_DIRECT_BITMAP, kTabShared, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U8 * 2: return body_direct<T, OP_DIRECT_U8, kTabGlobal, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U8 * 2 + 1: return body_direct<T, OP_DIRECT_U8, kTabShared, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U16 * 2: return body_direct<T, OP_DIRECT_U16, kTabGlobal, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U16 * 2 + 1: return body_direct<T, OP_DIRECT_U16, kTabShared, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U32 * 2: return body_direct<T, OP_DIRECT_U32, kTabGlobal, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U32 * 2 + 1: return body_direct<T, OP_DIRECT_U32, kTabShared, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U64 * 2: return !kWide ? m : body_direct<T, OP_DIRECT_U64, kTabGlobal, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U64 * 2 + 1: return !kWide ? m : body_direct<T, OP_DIRECT_U64, kTabShared, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U4 * 2: return body_direct<T, OP_DIRECT_U4, kTabGlobal, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U4 * 2 + 1: return body_direct<T, OP_DIRECT_U4, kTabShared, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U2 * 2: return body_direct<T, OP_DIRECT_U2, kTabGlobal, NR, WANT>(S, smem, v, m, code);
    case OP_DIRECT_U2 * 2 + 1: return body_direct<T, OP_DIRECT_U2, kTabShared, NR, WANT>(S, smem, v, m, code);
    case OP_HASHBITS * 2: return HASH && kWide ? body_hashbits<T, NR>(S, smem, v, m) : 0u; // comes with an exact probe stage
    case OP_HASH32 * 2:
    case OP_HASH64 * 2:
        if constexpr (HASH && kWide) {
            if (S.code_bits == 0) return body_hash<T, 0, NR, WANT>(S, smem, v, m, code);
            if (S.code_bits == 32) return body_hash<T, 4, NR, WANT>(S, smem, v, m, code);
            return body_hash<T, 8, NR, WANT>(S, smem, v, m, code);
        }
        return 0; // kernels built without the hash probe are never given such a stage
    default: return m; // OP_LOAD
    }
}

// ------------------------------------------------------------------ accumulators

// Feed a batch's values into the accumulators.  Every test on the stage's
// recipe is uniform and sits outside the row loop; a row contributes iff its
// bit is set in m.  acc32: every multiplier of the stage and every value it
// can see fits in 32 bits, so a contribution is one widening multiply-add.
template <int NR, typename V>
__device__ __forceinline__ void add_scaled(int64_t (&dst)[NR], int64_t mult, const V (&val)[NR], uint32_t m)
{
#pragma unroll
    for (int k = 0; k < NR; ++k)
        if ((m >> k) & 1u) dst[k] += mult * (int64_t)val[k];
}
template <int NR>
__device__ __forceinline__ void add_scaled32(int64_t (&dst)[NR], int32_t mult, const int32_t (&val)[NR], uint32_t m)
{
#pragma unroll
    for (int k = 0; k < NR; ++k)
        if ((m >> k) & 1u) dst[k] += (int64_t)mult * val[k]; // one widening multiply-add
}

template <bool MUL, typename T, int NR, typename C>
__device__ __forceinline__ void accumulate(const DStage &S, const T (&v)[NR], const C (&code)[NR], uint32_t m,
                                           int64_t (&key)[NR], int64_t (&X)[NR], int64_t (&Y)[NR])
{
    const uint32_t acc = S.acc;
    if (sizeof(C) == 4 || (S.acc32 && sizeof(T) == 4)) {
        if (acc & 0x7u) {
            int32_t r[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) r[k] = (int32_t)v[k];
            if (acc & 1u) add_scaled32<NR>(key, S.mult32[0], r, m);
            if (acc & 2u) add_scaled32<NR>(X, S.mult32[1], r, m);
            if (MUL && (acc & 4u)) add_scaled32<NR>(Y, S.mult32[2], r, m);
        }
        if (acc & 0x38u) {
            const uint32_t mask0 = (uint32_t)S.pmask0;
            const int32_t min0 = (int32_t)S.pmin0;
            int32_t p0[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) p0[k] = (int32_t)((uint32_t)code[k] & mask0) + min0;
            if (acc & 8u) add_scaled32<NR>(key, S.mult32[3], p0, m);
            if (acc & 16u) add_scaled32<NR>(X, S.mult32[4], p0, m);
            if (MUL && (acc & 32u)) add_scaled32<NR>(Y, S.mult32[5], p0, m);
        }
        if (acc & 0x1C0u) {
            const uint32_t sh = S.pbits0;
            const int32_t min1 = (int32_t)S.pmin1;
            int32_t p1[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) p1[k] = (int32_t)((uint32_t)code[k] >> sh) + min1;
            if (acc & 64u) add_scaled32<NR>(key, S.mult32[6], p1, m);
            if (acc & 128u) add_scaled32<NR>(X, S.mult32[7], p1, m);
            if (MUL && (acc & 256u)) add_scaled32<NR>(Y, S.mult32[8], p1, m);
        }
        return;
    }
    if (acc & 0x7u) {
        if (acc & 1u) add_scaled<NR>(key, S.mult[0], v, m);
        if (acc & 2u) add_scaled<NR>(X, S.mult[1], v, m);
        if (MUL && (acc & 4u)) add_scaled<NR>(Y, S.mult[2], v, m);
    }
    if (acc & 0x38u) {
        const uint64_t mask0 = S.pmask0;
        const int64_t min0 = S.pmin0;
        int64_t p0[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) p0[k] = (int64_t)(code[k] & mask0) + min0;
        if (acc & 8u) add_scaled<NR>(key, S.mult[3], p0, m);
        if (acc & 16u) add_scaled<NR>(X, S.mult[4], p0, m);
        if (MUL && (acc & 32u)) add_scaled<NR>(Y, S.mult[5], p0, m);
    }
    if (acc & 0x1C0u) {
        const uint32_t sh = S.pbits0;
        const int64_t min1 = S.pmin1;
        int64_t p1[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) p1[k] = (int64_t)(code[k] >> sh) + min1;
        if (acc & 64u) add_scaled<NR>(key, S.mult[6], p1, m);
        if (acc & 128u) add_scaled<NR>(X, S.mult[7], p1, m);
        if (MUL && (acc & 256u)) add_scaled<NR>(Y, S.mult[8], p1, m);
    }
}

// Insert-or-find in the global group table (open addressing, linear probe, bounded): the cell of group g, or ~0 when
// the table is full (status set).  The reserved empty marker as a key uses the side slot after the last regular slot.
__device__ __forceinline__ uint64_t group_cell(int64_t *gkeys, uint64_t gmask, int32_t *status, int64_t g)
{
    if (g == kEmptyKey64) return gmask + 1;
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(gkeys);
    uint64_t slot = hash64((uint64_t)g) & gmask;
    for (uint64_t it = 0; it <= gmask; ++it) {
        unsigned long long cur = *reinterpret_cast<volatile unsigned long long *>(&keys[slot]);
        if (cur == (unsigned long long)g) return slot;
        if (cur == (unsigned long long)kEmptyKey64) {
            cur = atomicCAS(&keys[slot], (unsigned long long)kEmptyKey64, (unsigned long long)g);
            if (cur == (unsigned long long)kEmptyKey64 || cur == (unsigned long long)g) return slot;
        }
        slot = (slot + 1) & gmask;
    }
    set_status(status, SJQ_ERR_GROUP_OVERFLOW);
    return ~0ull;
}

// Add (val, cnt) to the {sum, count} cells of one row per lane; `on`: the lane has a row.  All 32 lanes call it.
// Two neighbouring lanes share a row, one adds its sum and the other its count, so that both adds leave in one
// 32-byte sector: sixteen rows per instruction, half the sectors of a lane adding first the one, then the other.
// L2 performs about 192 G sector additions per second whatever a sector holds (200 M random rows on a million groups:
// 2.08 ms with two adds per lane, 1.04 in pairs; on a thousand contended groups 8.3 and 4.2), and the L1 passes one
// sector per cycle.
template <bool ONE>
__device__ __forceinline__ void add_pairs(unsigned long long *cells, uint32_t cell, uint64_t val, uint64_t cnt, bool on)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t rows = __ballot_sync(0xffffffffu, on);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        if (((rows >> (16 * half)) & 0xFFFFu) == 0u) continue;
        const int src = (int)(lane >> 1) + 16 * half;
        const uint32_t c = __shfl_sync(0xffffffffu, cell, src);
        unsigned long long v = __shfl_sync(0xffffffffu, (unsigned long long)val, src);
        const unsigned long long k = ONE ? 1ull : __shfl_sync(0xffffffffu, (unsigned long long)cnt, src);
        if (lane & 1u) v = k;
        if ((rows >> src) & 1u) atomicAdd(cells + 2 * (uint64_t)c + (lane & 1u), v);
    }
}

// 64-bit add into shared memory as two native 32-bit atomics: the low word's
// returned old value tells this thread whether its own add carried, so every
// carry is propagated exactly once and the 64-bit total is exact.
// The low and the high words of the cells are two arrays of their own (`hi_off` words apart), so that the
// low words of consecutive groups fall into consecutive banks; as halves of 64-bit cells they used every
// second bank only.
__device__ __forceinline__ void smem_add64(unsigned int *lo_word, uint32_t hi_off, uint64_t val)
{
    const unsigned int lo = (unsigned int)val;
    unsigned int hi = (unsigned int)(val >> 32);
    const unsigned int old = atomicAdd(lo_word, lo);
    hi += (unsigned int)((old + lo) < old);
    if (hi) atomicAdd(lo_word + hi_off, hi);
}
// Shared group table: [sum low words | sum high words | count low words | count high words], each `ng` words.
__device__ __forceinline__ uint64_t smem_cell(const unsigned int *words, uint64_t ng, uint64_t g)
{
    return ((uint64_t)words[ng + g] << 32) | words[g];
}

// A row's group key is out of range.  A pass that clears its results itself notes it in shared memory and tells it at the
// end, when the status word is known to be clear; so do all ahead-of-time kernels whose blocks keep sums of their own,
// which do not know at compile time whether they will clear.
__shared__ uint32_t range_seen;
template <int AGG>
__device__ __forceinline__ constexpr bool range_noted()
{
#if defined(SJQ_JIT)
    return (AGG == AGG_SCALAR || AGG == AGG_SMEM) && SJQ_JIT_may_clear != 0;
#else
    return AGG == AGG_SCALAR || AGG == AGG_SMEM;
#endif
}
template <bool NOTED>
__device__ __forceinline__ void note_range(const RunArg &P)
{
    if (NOTED) range_seen = 1u;
    else set_status(P.status, SJQ_ERR_GROUP_RANGE);
}

// The terminal on a batch: group keys of all rows first (their divisions overlap), then the
// aggregation; every test on the query shape is uniform and outside the row loops.
// FUSED: called by the fused kernel, where every lane of the warp arrives here (with or without rows), so that lanes may
// work on each other's rows.
template <int AGG, bool MUL, int NR, bool FUSED = true>
__device__ __forceinline__ void terminal(const RunArg &P, unsigned char *smem, const int64_t (&key)[NR],
                                         const int64_t (&X)[NR], const int64_t (&Y)[NR], uint32_t m, int64_t &lsum,
                                         int64_t &lcnt)
{
    const bool pairs = FUSED && (AGG == AGG_GLOBAL || AGG == AGG_HASH) && SJQ_PV(pairs) != 0;
    if (pairs ? !__any_sync(0xffffffffu, m != 0u) : m == 0u) return;
    int64_t val[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) val[k] = MUL ? X[k] * Y[k] : X[k];
    int64_t g[NR];
    if (AGG != AGG_SCALAR || SJQ_PV(has_key)) {
        const int64_t modulo = SJQ_PV(modulo);
        if (modulo == 0) {
#pragma unroll
            for (int k = 0; k < NR; ++k) g[k] = key[k];
        } else if (SJQ_PV(modmask)) {
            const int64_t mask = (int64_t)SJQ_PV(modmask);
#pragma unroll
            for (int k = 0; k < NR; ++k) g[k] = key[k] >= 0 ? (key[k] & mask) : (key[k] % modulo);
        } else if (SJQ_PV(mod32)) {
            const uint32_t d = (uint32_t)modulo;
#pragma unroll
            for (int k = 0; k < NR; ++k)
                g[k] = (uint64_t)key[k] <= 0xFFFFFFFFull ? (int64_t)((uint32_t)key[k] % d) : (key[k] % modulo);
        } else {
#pragma unroll
            for (int k = 0; k < NR; ++k) g[k] = key[k] % modulo;
        }
    }
    if (P.post_offset != 0) { // data-dependent (key range): a parameter, not part of a compiled shape
#pragma unroll
        for (int k = 0; k < NR; ++k) g[k] += P.post_offset;
    }
    if (AGG == AGG_SCALAR) {
        if (SJQ_PV(has_key)) {
#pragma unroll
            for (int k = 0; k < NR; ++k)
                if (((m >> k) & 1u) && g[k] != 0) {
                    note_range<FUSED && range_noted<AGG>()>(P);
                    m &= ~(1u << k);
                }
        }
#pragma unroll
        for (int k = 0; k < NR; ++k)
            if ((m >> k) & 1u) lsum += val[k];
        lcnt += __popc(m);
        return;
    }
    if (AGG == AGG_HASH) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            uint64_t cell = ~0ull;
            if ((m >> k) & 1u) cell = group_cell(P.gkeys, P.gmask, P.status, g[k]);
            if (pairs) {
                add_pairs<true>(reinterpret_cast<unsigned long long *>(P.sums), (uint32_t)cell, (uint64_t)val[k], 1ull, cell != ~0ull);
            } else if (cell != ~0ull) {
                atomicAdd(reinterpret_cast<unsigned long long *>(P.sums) + 2 * cell, (unsigned long long)val[k]);
                atomicAdd(reinterpret_cast<unsigned long long *>(P.counts) + 2 * cell, 1ull);
            }
        }
        return;
    }
    const uint64_t ng = (uint64_t)P.num_groups;
#pragma unroll
    for (int k = 0; k < NR; ++k)
        if (((m >> k) & 1u) && (uint64_t)g[k] >= ng) {
            note_range<FUSED && range_noted<AGG>()>(P);
            m &= ~(1u << k);
        }
    const bool want_count = SJQ_PV(want_count) != 0;
    const uint32_t shift = SJQ_PV(cell_shift); // 1: sums and counts alternate in one array
    if (AGG == AGG_GLOBAL && pairs) {
#pragma unroll
        for (int k = 0; k < NR; ++k)
            add_pairs<true>(reinterpret_cast<unsigned long long *>(P.sums), (uint32_t)g[k], (uint64_t)val[k], 1ull, (m >> k) & 1u);
        return;
    }
    if (SJQ_PV(warp_agg)) {
        // Warp-level pre-aggregation: the lanes of a warp holding the same group key are found with one match
        // instruction, their values are added inside the warp, and one lane per distinct key issues the
        // atomics.  Worth it when a few groups take most rows (the lanes of a warp would otherwise serialise on
        // the same counter); costs about a dozen instructions per row when every lane has its own key.
        unsigned int *ss = reinterpret_cast<unsigned int *>(smem + P.smem_groups);
        unsigned long long *sums = reinterpret_cast<unsigned long long *>(P.sums);
        unsigned long long *counts = reinterpret_cast<unsigned long long *>(P.counts);
        const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const bool on = (m >> k) & 1u;
            const unsigned active = __activemask();
            // a lane without a row takes a key no group can have (group keys are below num_groups)
            const unsigned long long kk = on ? (unsigned long long)g[k] : (0x8000000000000000ull | lane);
            const unsigned peers = __match_any_sync(active, kk);
            // exact 64-bit sum over at most 32 lanes, in three pieces that cannot overflow 32 bits
            const uint64_t v = on ? (uint64_t)val[k] : 0ull;
            const uint64_t s0 = __reduce_add_sync(peers, (unsigned)(v & 0x3FFFFFu));
            const uint64_t s1 = __reduce_add_sync(peers, (unsigned)((v >> 22) & 0x3FFFFFu));
            const uint64_t s2 = __reduce_add_sync(peers, (unsigned)(v >> 44));
            if (on && lane == (uint32_t)(__ffs(peers) - 1)) {
                const uint64_t total = s0 + (s1 << 22) + (s2 << 44);
                const uint64_t cnt = (uint64_t)__popc(peers);
                if (AGG == AGG_SMEM) {
                    smem_add64(ss + g[k], (uint32_t)ng, total);
                    if (want_count) smem_add64(ss + 2 * ng + g[k], (uint32_t)ng, cnt);
                } else {
                    atomicAdd(sums + (g[k] << shift), (unsigned long long)total);
                    if (want_count) atomicAdd(counts + (g[k] << shift), (unsigned long long)cnt);
                }
            }
        }
        return;
    }
    if (AGG == AGG_SMEM) {
        unsigned int *ss = reinterpret_cast<unsigned int *>(smem + P.smem_groups);
#pragma unroll
        for (int k = 0; k < NR; ++k)
            if ((m >> k) & 1u) smem_add64(ss + g[k], (uint32_t)ng, (uint64_t)val[k]);
        if (want_count) {
            // a block sees fewer than 2^32 rows (count32): its count of a group cannot carry, and an add whose
            // result nobody reads is a reduction the lane does not wait for
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                if ((m >> k) & 1u) {
                    if (SJQ_PV(count32)) atomicAdd(ss + 2 * ng + g[k], 1u);
                    else smem_add64(ss + 2 * ng + g[k], (uint32_t)ng, 1ull);
                }
            }
        }
    } else {
        unsigned long long *gs = reinterpret_cast<unsigned long long *>(P.sums);
#pragma unroll
        for (int k = 0; k < NR; ++k)
            if ((m >> k) & 1u) atomicAdd(gs + (g[k] << shift), (unsigned long long)val[k]);
        if (want_count) {
            unsigned long long *gc = reinterpret_cast<unsigned long long *>(P.counts);
#pragma unroll
            for (int k = 0; k < NR; ++k)
                if ((m >> k) & 1u) atomicAdd(gc + (g[k] << shift), 1ull);
        }
    }
}

// ------------------------------------------------------------------ row batches
// A batch is up to kRows rows per lane, named by 32-bit offsets from a base
// row that is uniform over the warp (so a column address costs one multiply-
// add per row).  CONTIG: the lane owns four consecutive rows (one 128-bit
// load); otherwise the rows are survivors popped from a queue (one 4- or
// 8-byte load each).

template <typename T, bool CONTIG, int NR>
__device__ __forceinline__ void load_rows(const DStage &S, int64_t base, const uint32_t (&off)[NR], uint32_t valid,
                                          uint32_t need, T (&v)[NR])
{
    const T *c = static_cast<const T *>(S.col) + base;
    static_assert(!CONTIG || NR == 4, "a thread-owned group is four consecutive rows");
    if (CONTIG && valid == 0xFu) {
        Vec4<T>::load(c + off[0], v, S.col32);
        return;
    }
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        v[k] = 0;
        if ((need >> k) & 1u) v[k] = ld_sparse(c + off[k]);
    }
}

// NARROW kernels: every code of the query has 32 bits, and every fact column but the keys of open-addressing tables.
template <bool NARROW>
struct CodeWord {
    typedef uint64_t type;
};
template <>
struct CodeWord<true> {
    typedef uint32_t type;
};

// One pure filter stage on a batch: returns the mask of rows that pass.
template <bool HASH, bool NARROW, int NR>
__device__ __forceinline__ uint32_t filter_rows(const RunArg &P, const DStage &S, const unsigned char *smem,
                                                int64_t base, const uint32_t (&off)[NR], uint32_t valid)
{
    typename CodeWord<NARROW>::type unused[NR];
    if constexpr (!NARROW || HASH) {
        if (S.is64) {
            int64_t v[NR];
            load_rows<int64_t, false, NR>(S, base, off, valid, valid, v);
            return run_stage<int64_t, NR, false, HASH>(P, S, smem, v, valid, unused);
        }
    }
    int32_t v[NR];
    load_rows<int32_t, false, NR>(S, base, off, valid, valid, v);
    return run_stage<int32_t, NR, false, HASH>(P, S, smem, v, valid, unused);
}

// Stages [first, nstages) with accumulators, then the terminal.  The column of
// the next stage is requested before the current stage's probe is resolved, so
// a stage costs one memory latency, not two.
template <int AGG, bool MUL, bool CONTIG, bool HASH, bool NARROW, int NR>
__device__ __forceinline__ void final_rows(const RunArg &P, const DStage *st, unsigned char *smem, int first,
                                           int64_t base, const uint32_t (&off)[NR], uint32_t valid, int64_t &lsum,
                                           int64_t &lcnt)
{
    uint32_t m = valid;
    int64_t key[NR], X[NR], Y[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        key[k] = P.key_offset;
        X[k] = 0;
        Y[k] = 0;
    }
    int32_t vnext[NR];
    bool have_next = false;
    SJQ_UNROLL_STAGES
    for (int s = first; s < SJQ_PV(nstages); ++s) {
        const DStage &S = SJQ_STAGE(s);
        const uint32_t need = SJQ_PV(eager) ? valid : m;
        if (!need) break;
        const uint32_t simple = S.simple;
        if (simple) { // a plain int32 column feeding one accumulator: no probe, no recipe to interpret
            int32_t v[NR];
            if (have_next) {
#pragma unroll
                for (int k = 0; k < NR; ++k) v[k] = vnext[k];
            } else {
                load_rows<int32_t, CONTIG, NR>(S, base, off, valid, need, v);
            }
            have_next = (s + 1 < SJQ_PV(nstages)) && ((NARROW && !HASH) || !SJQ_STAGE(s + 1).is64);
            if (have_next) load_rows<int32_t, CONTIG, NR>(SJQ_STAGE(s + 1), base, off, valid, need, vnext);
            const int32_t mult = S.mult32[simple - 1];
            if (simple == 2) add_scaled32<NR>(X, mult, v, m);
            else if (simple == 1) add_scaled32<NR>(key, mult, v, m);
            else if (MUL) add_scaled32<NR>(Y, mult, v, m);
            continue;
        }
        typename CodeWord<NARROW>::type code[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) code[k] = 0;
        if constexpr (!NARROW || HASH) {
            if (S.is64) {
                int64_t v[NR];
                load_rows<int64_t, CONTIG, NR>(S, base, off, valid, need, v);
                have_next = false;
                m = run_stage<int64_t, NR, true, HASH>(P, S, smem, v, m, code);
                if (S.acc) accumulate<MUL, int64_t, NR>(S, v, code, m, key, X, Y);
                continue;
            }
        }
        int32_t v[NR];
        if (have_next) {
#pragma unroll
            for (int k = 0; k < NR; ++k) v[k] = vnext[k];
        } else {
            load_rows<int32_t, CONTIG, NR>(S, base, off, valid, need, v);
        }
        have_next = (s + 1 < SJQ_PV(nstages)) && ((NARROW && !HASH) || !SJQ_STAGE(s + 1).is64);
        if (have_next) load_rows<int32_t, CONTIG, NR>(SJQ_STAGE(s + 1), base, off, valid, need, vnext);
        m = run_stage<int32_t, NR, true, HASH>(P, S, smem, v, m, code);
        if (S.acc) accumulate<MUL, int32_t, NR>(S, v, code, m, key, X, Y);
    }
    terminal<AGG, MUL, NR>(P, smem, key, X, Y, m, lsum, lcnt);
}

#if defined(SJQ_JIT)
// The final level of a kernel compiled for the query, fed from a queue.  The planner has scheduled
// every column load: a column is requested as soon as the mask it depends on is known (on entry, or
// right after the last stage before it that drops rows), at most kLoadsInFlight columns ahead, so the
// level costs about one memory latency per run of stages that drop nothing instead of one per stage.
// CONTIG: the rows are a thread's own four consecutive rows (no queues at all: the plan for queries most of
// whose rows survive, where every column is read whole anyway): one 128-bit load per column, issued up
// front, four columns deep.
template <int AGG, bool MUL, bool HASH, bool CONTIG, int NR>
__device__ __forceinline__ void final_rows_scheduled(const RunArg &P, unsigned char *smem, int first, int64_t base,
                                                     const uint32_t (&off)[NR], uint32_t valid, int64_t &lsum,
                                                     int64_t &lcnt)
{
    constexpr int kLoadsInFlight = CONTIG ? 4 : 3;
    uint32_t m = valid;
    int64_t key[NR], X[NR], Y[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        key[k] = P.key_offset;
        X[k] = 0;
        Y[k] = 0;
    }
    int32_t buf[kLoadsInFlight][NR]; // column of stage t waits in buf[(t - first) % kLoadsInFlight]
#pragma unroll
    for (int t = first; t < SJQ_PV(nstages); ++t) {
        const DStage &T = SJQ_STAGE(t);
        if (T.issue_after < first && !T.is64)
            load_rows<int32_t, CONTIG, NR>(T, base, off, valid, valid, buf[(t - first) % kLoadsInFlight]);
    }
#pragma unroll
    for (int s = first; s < SJQ_PV(nstages); ++s) {
        const DStage &S = SJQ_STAGE(s);
        if (!(SJQ_PV(eager) ? valid : m)) break;
        const uint32_t simple = S.simple;
        if (simple) {
            const int32_t mult = S.mult32[simple - 1];
            if (simple == 2) add_scaled32<NR>(X, mult, buf[(s - first) % kLoadsInFlight], m);
            else if (simple == 1) add_scaled32<NR>(key, mult, buf[(s - first) % kLoadsInFlight], m);
            else if (MUL) add_scaled32<NR>(Y, mult, buf[(s - first) % kLoadsInFlight], m);
        } else {
            uint64_t code[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) code[k] = 0;
            if (S.is64) {
                int64_t v[NR];
                load_rows<int64_t, CONTIG, NR>(S, base, off, valid, SJQ_PV(eager) ? valid : m, v);
                m = run_stage<int64_t, NR, true, HASH>(P, S, smem, v, m, code);
                if (S.acc) accumulate<MUL, int64_t, NR>(S, v, code, m, key, X, Y);
            } else {
                m = run_stage<int32_t, NR, true, HASH>(P, S, smem, buf[(s - first) % kLoadsInFlight], m, code);
                if (S.acc) accumulate<MUL, int32_t, NR>(S, buf[(s - first) % kLoadsInFlight], code, m, key, X, Y);
            }
        }
        const uint32_t need = SJQ_PV(eager) ? valid : m;
#pragma unroll
        for (int t = s + 1; t <= s + kLoadsInFlight; ++t) {
            if (t < SJQ_PV(nstages)) {
                const DStage &T = SJQ_STAGE(t);
                if (T.issue_after == s && !T.is64)
                    load_rows<int32_t, CONTIG, NR>(T, base, off, valid, need, buf[(t - first) % kLoadsInFlight]);
            }
        }
    }
    terminal<AGG, MUL, NR>(P, smem, key, X, Y, m, lsum, lcnt);
}
#endif

// ------------------------------------------------------------------ level 0
// One filter stage on the thread's own kSlots groups of four consecutive rows
// of a tile: the column is loaded for a group only while one of its rows is
// alive.  FULL: the whole tile lies inside the table (no bounds masks).
// `staged` != nullptr: the tile's values of this column were copied into shared memory by a bulk-asynchronous
// copy (in table order); the thread reads its four values of each slice from there.
template <typename T, bool FULL, bool HASH, bool NARROW>
__device__ __forceinline__ uint32_t dense_stage(const RunArg &P, const DStage &S, const unsigned char *smem,
                                                int64_t row0, int32_t slot_stride, uint32_t valid, uint32_t alive,
                                                const unsigned char *staged = nullptr)
{
    T v[kDenseRows];
    const T *c = static_cast<const T *>(S.col) + row0;
#pragma unroll
    for (int u = 0; u < kSlots; ++u) {
#pragma unroll
        for (int r = 0; r < 4; ++r) v[4 * u + r] = 0;
        if (FULL && staged != nullptr) {
            const T *sp = reinterpret_cast<const T *>(staged) + u * slot_stride + 4 * threadIdx.x;
            if (sizeof(T) == 4) {
                const uint4 w = *reinterpret_cast<const uint4 *>(sp);
                v[4 * u] = (T)(int32_t)w.x, v[4 * u + 1] = (T)(int32_t)w.y, v[4 * u + 2] = (T)(int32_t)w.z, v[4 * u + 3] = (T)(int32_t)w.w;
            } else {
                const uint4 a = *reinterpret_cast<const uint4 *>(sp), b = *(reinterpret_cast<const uint4 *>(sp) + 1);
                v[4 * u] = (T)(((uint64_t)a.y << 32) | a.x), v[4 * u + 1] = (T)(((uint64_t)a.w << 32) | a.z);
                v[4 * u + 2] = (T)(((uint64_t)b.y << 32) | b.x), v[4 * u + 3] = (T)(((uint64_t)b.w << 32) | b.z);
            }
        } else if ((alive >> (4 * u)) & 0xFu) {
            if (FULL) {
                Vec4<T>::load(c + u * slot_stride, &v[4 * u], S.col32);
            } else {
                const uint32_t nv = (valid >> (4 * u)) & 0xFu;
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if ((nv >> r) & 1u) v[4 * u + r] = __ldcs(c + u * slot_stride + r);
            }
        }
    }
    typename CodeWord<NARROW>::type unused[kDenseRows];
    return run_stage<T, kDenseRows, false, HASH>(P, S, smem, v, alive, unused);
}

template <bool FULL, bool HASH, bool NARROW>
__device__ __forceinline__ uint32_t level0(const RunArg &P, const DStage *st, const unsigned char *smem,
                                           int64_t row0, int32_t slot_stride, uint32_t valid,
                                           const unsigned char *staged = nullptr)
{
    uint32_t alive = valid;
    SJQ_UNROLL_STAGES
    for (int s = 0; s < SJQ_PV(nd0); ++s) {
        if (!alive) break;
        const DStage &S = SJQ_STAGE(s);
        const unsigned char *from = s == 0 ? staged : nullptr; // only the first column is staged
        if constexpr (!NARROW || HASH) {
            if (S.is64) {
                alive = dense_stage<int64_t, FULL, HASH, NARROW>(P, S, smem, row0, slot_stride, valid, alive, from);
                continue;
            }
        }
        alive = dense_stage<int32_t, FULL, HASH, NARROW>(P, S, smem, row0, slot_stride, valid, alive, from);
    }
    return alive;
}

// ------------------------------------------------------------------ bulk-asynchronous staging of the first column
// A block's tile of the first column (block size x 4 x kSlots consecutive values, 12 to 64 KB: copies below
// 4 KB ran at a third of the bandwidth) is brought into shared memory by one cp.async.bulk global -> shared
// copy that completes on an mbarrier (no tensor map, no cluster multicast, this GPU's memory only); three tiles
// are in flight per block.  The warps stay independent: each waits for a tile at its own pace, reads its
// slice, and counts itself off; the warp that counts last refills the buffer with the tile three steps ahead.
// Every wait is bounded: if one runs out the warp records SJQ_ERR_ASYNC_WAIT, reads this and every later tile
// with plain loads (the result stays exact; the other warps of the block follow when their refills stop
// coming) and, before it leaves, gives the copies still in flight a last bounded wait.
constexpr int kBulkStages = 3;
// polls of an mbarrier before a wait gives up: a copy lands within microseconds (a handful of polls); each poll may
// itself block for a hardware-defined slice, so the bound is kept well under a second in the worst case
constexpr int kBulkSpins = 1 << 16;
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bulk_issue(uint32_t bar, uint32_t dst, const void *src, uint32_t bytes)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); // earlier reads of the buffer precede the copy
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool bulk_wait(uint32_t bar, uint32_t parity, int spins)
{
    uint32_t done = 0;
    for (int spin = 0; spin < spins && !done; ++spin)
        asm volatile("{ .reg .pred q; mbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2; selp.u32 %0, 1, 0, q; }"
                     : "=r"(done)
                     : "r"(bar), "r"(parity)
                     : "memory");
    return done != 0;
}

// ------------------------------------------------------------------ per-warp queues
// Queue l of a warp (a ring of 32-bit row offsets in shared memory) holds the
// rows that passed stages 0 .. nd0+l-1.  The level fed by queue l runs filter
// stage nd0+l and pushes to queue l+1, or, for the last queue, runs the
// remaining stages and the terminal.  Heads and counts live in registers and are
// selected without indexing so that they never spill to local memory.
struct QueueState {
    uint32_t h0, h1, h2, c0, c1, c2;
    __device__ __forceinline__ uint32_t head(int l) const { return l == 0 ? h0 : (l == 1 ? h1 : h2); }
    __device__ __forceinline__ uint32_t count(int l) const { return l == 0 ? c0 : (l == 1 ? c1 : c2); }
    __device__ __forceinline__ void set_head(int l, uint32_t v)
    {
        h0 = l == 0 ? v : h0;
        h1 = l == 1 ? v : h1;
        h2 = l == 2 ? v : h2;
    }
    __device__ __forceinline__ void set_count(int l, uint32_t v)
    {
        c0 = l == 0 ? v : c0;
        c1 = l == 1 ? v : c1;
        c2 = l == 2 ? v : c2;
    }
};

// Slot of ring position `pos` in a queue of `cap` entries.  A lane pushes its survivors to consecutive
// positions, so when most rows survive the lanes of one store are 4 or 8 positions apart and would share 4 or
// 8 banks; folding bits 5-7 of the position into bits 0-2 spreads such a store over all 32 banks, and 32
// consecutive positions (a pop) still map to 32 different banks.
// Only kernels compiled for a query do it, and only when the planner asks (fold = 7: many rows survive
// level 0); the interpreted kernels have no registers to spare for it.
__device__ __forceinline__ uint32_t queue_slot(uint32_t pos, uint32_t cap, uint32_t fold)
{
    const uint32_t p = pos & (cap - 1);
#if defined(SJQ_JIT)
    return p ^ ((p >> 5) & fold);
#else
    return p;
#endif
}

__device__ __forceinline__ uint32_t queue_cap(int l) { return l == 0 ? (uint32_t)kQueue0Cap : (uint32_t)kQueueCap; }
__device__ __forceinline__ uint32_t queue_base(int l)
{
    return l == 0 ? 0u : (uint32_t)(kQueue0Cap + (l - 1) * kQueueCap);
}

// ------------------------------------------------------------------ results cleared by the pass itself
// A clear kernel in front of the pass costs a small query a fifth of its time: a launch on the host and a kernel boundary
// on the device.  With words to meet at (P.sync) the first few blocks of the pass clear the results while the others
// begin; a block's sums are its own (registers, a shared group table), and it looks at the flags at its end, before it
// adds them to the results (a pass that adds its rows one by one to a global table would have to look before its first row:
// 300 thousand rows, skewed keys, 4096 groups 23.4 us with the clear kernel and 26.9 so).  A flag is up when it holds the
// number of this very call, so that the words may hold anything before the first one; the last block to finish takes all
// flags down, so that a captured call can be replayed.  The blocks that clear wait for nobody before their flags are up
// and are the first of the grid, so the others never wait for a block that waits for them.
// Every wait is bounded all the same.  A block whose wait ran out does not add its sums, which the late clear might wipe,
// and arrives as late; the last block to arrive, behind every clear, turns that into the status.  The word that counts the
// arrivals names the call too.  Block 0 raises it to that name, which leaves alone what blocks that were late before it
// have counted there under the same name; a block that does not find the name (the words held something larger before
// their first use) puts it there and counts again.  So every block is counted once, the last one is known, and it leaves
// the words at rest.
// (100 thousand rows, filter and sum, interpreted, calls back to back: 9.7 -> 7.6 us, the host's launch.  On the device, in a
// captured call, 5.6 us with a clear kernel, which starts beside the call before, and 5.1 so; compiled 3.2 and 3.6.  What
// counts there is the chain behind the block that clears: no fence but the flag's release, no fence before the arrival, no
// answer waited for: 4.3 us with them.)
constexpr int kClearSpins = 1 << 20;
constexpr uint64_t kClearArrivals = (1ull << 20) - 1, kClearLate = 1ull << 20; // the rest of the word: the call
constexpr int kClearCall = 21;
// What hardly ever runs stays out of the way of what does (524,288 rows, filter and sum, compiled: 5.45 us with it in line,
// 5.04 so).
__device__ __noinline__ void clear_sleep(int ms)
{
    while (ms-- > 0) __nanosleep(1000000u);
}
// Counts a block that was late, or that did not find the call's name; returns the word before.
__device__ __noinline__ uint64_t clear_count_again(unsigned long long *arrivals, uint64_t call, uint64_t found, uint64_t late)
{
    for (;;) { // (a try fails because another block has arrived: bounded by the grid)
        const uint64_t word = (((found ^ call) >> kClearCall) == 0 ? found : call) | late;
        const uint64_t now = atomicCAS(arrivals, (unsigned long long)found, (unsigned long long)(word + 1));
        if (now == found) return word;
        found = now;
    }
}
__device__ __forceinline__ void clear_share(const RunArg &P)
{
    const int64_t step = (int64_t)P.clear_blocks * blockDim.x;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (P.clear_late_ms && blockIdx.x == 0) clear_sleep(P.clear_late_ms);
    for (int64_t i = first; i < P.clear_cells / 2; i += step) {
        reinterpret_cast<longlong2 *>(P.sums)[i] = make_longlong2(0, 0);
        if (P.clear_counts) reinterpret_cast<longlong2 *>(P.clear_counts)[i] = make_longlong2(0, 0);
    }
    if (first == 0) {
        if (P.clear_cells & 1) {
            P.sums[P.clear_cells - 1] = 0;
            if (P.clear_counts) P.clear_counts[P.clear_cells - 1] = 0;
        }
        *P.status = 0;
        // (no answer is waited for, as a compare-and-swap's would be)
        atomicMax(reinterpret_cast<unsigned long long *>(P.sync), (unsigned long long)(P.epoch << kClearCall));
    }
}
// (thread 0, behind a barrier of the block: a release carries the stores of all its threads)
__device__ __forceinline__ void clear_told(const RunArg &P)
{
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(P.sync + 1 + blockIdx.x), "l"(P.epoch) : "memory");
}
// (thread 0, before a barrier of the block)  Whether all flags are up.
__device__ __forceinline__ bool clear_wait(const RunArg &P)
{
    int spins = kClearSpins;
    for (int b = 0; b < P.clear_blocks; ++b) {
        uint64_t seen = 0;
        for (; spins > 0 && seen != P.epoch; --spins)
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(P.sync + 1 + b) : "memory");
        if (seen != P.epoch) return false;
    }
    return true;
}
// (thread 0, behind its wait for the clear; the sums need not have arrived, and block 0's status has, behind its flag)
__device__ __forceinline__ void clear_over(const RunArg &P, bool late)
{
    unsigned long long *const arrivals = reinterpret_cast<unsigned long long *>(P.sync);
    const uint64_t call = P.epoch << kClearCall;
    uint64_t word = late ? 0 : atomicAdd(arrivals, 1ull);
    if (late || ((word ^ call) >> kClearCall) != 0) word = clear_count_again(arrivals, call, word, late ? kClearLate : 0);
    if ((word & kClearArrivals) != gridDim.x - 1) return;
    if (word & kClearLate) {
        __threadfence();
        set_status(P.status, SJQ_ERR_ASYNC_WAIT);
    }
    for (int b = 0; b <= P.clear_blocks; ++b) P.sync[b] = 0;
}

// The scalar terminal's tail (Section 3.2: one atomic per block instead of one per matching row): warp
// shuffle reduce, block reduce through shared memory, one global atomic per block.  False (thread 0) if the block waited for
// the clear in vain and its sums were not added.
__device__ __forceinline__ bool scalar_block_reduce(const RunArg &P, int64_t lsum, int64_t lcnt, bool self_clear = false)
{
    bool cleared = true;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        lcnt += __shfl_xor_sync(0xffffffffu, lcnt, o);
    }
    __shared__ int64_t part[64];
    if (lane == 0) {
        part[warp] = lsum;
        part[32 + warp] = lcnt;
    }
    __syncthreads();
    if (warp == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        lsum = lane < nw ? part[lane] : 0;
        lcnt = lane < nw ? part[32 + lane] : 0;
        for (int o = 16; o > 0; o >>= 1) {
            lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
            lcnt += __shfl_xor_sync(0xffffffffu, lcnt, o);
        }
        if (lane == 0 && self_clear) cleared = clear_wait(P);
        if (lane == 0 && lcnt != 0 && cleared) {
            atomicAdd(reinterpret_cast<unsigned long long *>(P.sums), (unsigned long long)lsum);
            if (P.counts) atomicAdd(reinterpret_cast<unsigned long long *>(P.counts), (unsigned long long)lcnt);
        }
    }
    return cleared;
}

// `given`: the stage descriptors of the parameter block.
// DIRECT: no queues, every stage runs on thread-owned rows.
template <int AGG, bool MUL, bool HASH, bool DIRECT, bool NARROW>
__device__ __forceinline__ void fused_body(const RunArg &P, const DStage *given, unsigned char *smem)
{
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;

    // (only in kernels for few rows: the registers that it takes cost a pass over many rows up to 30 %, and the clear kernel
    // costs that one next to nothing, since the pass starts behind it)
    const bool self_clear = (AGG == AGG_SCALAR || AGG == AGG_SMEM) && DIRECT && SJQ_PV(may_clear) && P.sync;
    if (self_clear) {
        // launched while the kernel before it still runs (four joins, 400 thousand rows, interpreted: 12.4 -> 10.5 us)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if ((int)blockIdx.x < P.clear_blocks) clear_share(P);
    }

    // Stage descriptors and small direct tables -> shared memory (once per block).
    DStage *st = reinterpret_cast<DStage *>(smem + P.smem_stages);
#if !defined(SJQ_JIT)
    {
        const uint32_t words = (uint32_t)(P.nstages * sizeof(DStage) / 8);
        const uint64_t *src = reinterpret_cast<const uint64_t *>(given);
        uint64_t *dst = reinterpret_cast<uint64_t *>(st);
        for (uint32_t i = tid; i < words; i += blockDim.x) dst[i] = src[i];
    }
#endif
    SJQ_UNROLL_STAGES
    for (int s = 0; s < SJQ_PV(nstages); ++s) {
#if defined(SJQ_JIT)
        const DStage &S = SJQ_STAGE(s);
#else
        const DStage &S = given[s];
#endif
        if (S.in_smem) {
            const uint4 *src = static_cast<const uint4 *>(S.tab);
            uint4 *dst = reinterpret_cast<uint4 *>(smem + S.smem_off);
            for (uint32_t i = tid; i < S.tab_bytes / 16; i += blockDim.x) dst[i] = __ldg(src + i);
        }
        if (HASH && S.hot == 1) { // the bitmap stage copies the join's hot-key table; its exact probe reads the same copy
            // (plain loads: the table was written by the kernels enqueued just before this one)
            const uint4 *src = static_cast<const uint4 *>(S.hot_tab);
            uint4 *dst = reinterpret_cast<uint4 *>(smem + S.hot_off);
            for (uint32_t i = tid; i < (uint32_t)kHotSlots + 1u; i += blockDim.x) dst[i] = src[i];
        }
    }
    if (AGG == AGG_SMEM) {
        unsigned long long *ss = reinterpret_cast<unsigned long long *>(smem + P.smem_groups);
        const int64_t cells = P.num_groups * (SJQ_PV(want_count) ? 2 : 1);
        for (int64_t i = tid; i < cells; i += blockDim.x) ss[i] = 0ull;
    }
    if (range_noted<AGG>() && tid == 0) range_seen = 0u;
    __syncthreads();
    if (self_clear && tid == 0 && (int)blockIdx.x < P.clear_blocks) clear_told(P);
    // launched behind the kernel that clears the results: nothing above touches them, everything below may
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // (the listing of a hashed result, or the clear of the next pass, is launched while this kernel runs and waits for its
    // end on the device)
    asm volatile("griddepcontrol.launch_dependents;");

    int64_t lsum = 0, lcnt = 0;

    if constexpr (DIRECT) {
        // No queue: every stage runs on the thread's own four consecutive rows.
        const int64_t tile_rows = (int64_t)blockDim.x * kDirectRows;
        const int64_t ntiles = (P.n + tile_rows - 1) / tile_rows;
        uint32_t off[kDirectRows];
#pragma unroll
        for (int k = 0; k < kDirectRows; ++k) off[k] = (uint32_t)(4 * tid + k);
        for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const int64_t base = tile * tile_rows;
            const int64_t rem = P.n - base - 4 * (int64_t)tid;
            const uint32_t valid = rem >= 4 ? 0xFu : (rem > 0 ? ((1u << (int)rem) - 1u) : 0u);
#if defined(SJQ_JIT)
            final_rows_scheduled<AGG, MUL, HASH, true, kDirectRows>(P, smem, 0, base, off, valid, lsum, lcnt);
#else
            final_rows<AGG, MUL, true, HASH, NARROW, kDirectRows>(P, st, smem, 0, base, off, valid, lsum, lcnt);
#endif
        }
    } else {
        const int nq = SJQ_PV(nq);
        uint32_t *const qmem = reinterpret_cast<uint32_t *>(smem + P.smem_queue) +
                               warp * (kQueue0Cap + (nq - 1) * kQueueCap);
        QueueState Q{0, 0, 0, 0, 0, 0};
        const bool wide = P.n > 0xFFFFFFFFll; // offsets are tile-relative and the queues are flushed per tile
#if defined(SJQ_JIT)
        constexpr bool kBulk = SJQ_JIT_l0_bulk != 0;
#else
        constexpr bool kBulk = false;
#endif
        const int32_t slot_stride = (int32_t)blockDim.x * 4;
        const int32_t tile_rows = slot_stride * kSlots;
        const uint32_t ntiles = (uint32_t)((P.n + tile_rows - 1) / tile_rows); // host checks n / tile_rows < 2^31
        int64_t qbase = 0;
        uint32_t tile = blockIdx.x;
        bool flushing = false;

        // bulk-asynchronous staging of the first column (compiled kernels the planner chose it for)
        const uint32_t l0_elem = SJQ_STAGE(0).is64 ? 8u : 4u;
        const uint32_t tile_bytes = (uint32_t)tile_rows * l0_elem;
        unsigned char *const l0_buf = smem + P.smem_l0;
        unsigned long long *const l0_bar = reinterpret_cast<unsigned long long *>(l0_buf + (size_t)kBulkStages * tile_bytes);
        unsigned int *const l0_done = reinterpret_cast<unsigned int *>(l0_bar + kBulkStages); // warps done with a buffer
        bool bulk_ok = kBulk;
        uint32_t bstage = 0, bphase = 0;
        auto tile_full = [&](uint32_t t) { return t < ntiles && (int64_t)t * tile_rows + tile_rows <= P.n; };
        auto issue_tile = [&](uint32_t t, uint32_t stage) {
#if defined(SJQ_JIT)
            if (SJQ_JIT_l0_bulk == 2) return; // test form: no copy is ever issued, so every wait runs out
#endif
            const char *src = static_cast<const char *>(SJQ_STAGE(0).col) + (int64_t)t * tile_rows * l0_elem;
            bulk_issue(smem_addr(&l0_bar[stage]), smem_addr(l0_buf + (size_t)stage * tile_bytes), src, tile_bytes);
        };
        if (kBulk) {
            if (tid == 0) {
                for (int b = 0; b < kBulkStages; ++b) {
                    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&l0_bar[b])));
                    l0_done[b] = 0;
                }
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
                for (uint32_t b = 0; b < (uint32_t)kBulkStages; ++b)
                    if (tile_full(tile + b * gridDim.x)) issue_tile(tile + b * gridDim.x, b);
            }
            __syncthreads(); // the barriers exist before any warp waits on one
        }

        // One loop, one call site per piece of work: pick the deepest queue holding a full
        // batch (so that a push never meets a full queue); else filter the next tile and push
        // its survivors; at the end drain what is left.
        for (;;) {
            int l = (nq >= 3 && Q.c2 >= (uint32_t)kBatch) ? 2
                    : (nq >= 2 && Q.c1 >= (uint32_t)kBatch) ? 1
                    : (Q.c0 >= (uint32_t)kBatch)            ? 0
                                                            : -1;
            uint32_t nb = kBatch;
            if (l < 0) {
                if (flushing) {
                    l = Q.c0 ? 0 : (Q.c1 ? 1 : (Q.c2 ? 2 : -1));
                    if (l < 0) {
                        flushing = false;
                        if (tile >= ntiles) break;
                        continue;
                    }
                    nb = Q.count(l) < (uint32_t)kBatch ? Q.count(l) : (uint32_t)kBatch;
                } else if (tile < ntiles) {
                    // level 0: the first stage on the thread's own rows of the next tile
                    const int64_t tile_base = (int64_t)tile * tile_rows;
                    const int64_t row0 = tile_base + 4 * tid;
                    if (wide) qbase = tile_base;
                    if (!kBulk) { // ask L2 for the first column of the tile this block filters after the next one
                        const int64_t nrow = row0 + (int64_t)gridDim.x * tile_rows * 2;
                        if (nrow + tile_rows <= P.n) {
                            const DStage &S0 = SJQ_STAGE(0);
                            const char *pc = static_cast<const char *>(S0.col) + nrow * (S0.is64 ? 8 : 4);
#pragma unroll
                            for (int k = 0; k < kSlots; ++k)
                                asm volatile("prefetch.global.L2 [%0];" ::"l"(pc + (int64_t)k * slot_stride * (S0.is64 ? 8 : 4)));
                        }
                    }
                    uint32_t alive;
                    if (tile_base + tile_rows <= P.n) {
                        const unsigned char *staged = nullptr;
                        if (kBulk && bulk_ok) {
                            if (__all_sync(0xffffffffu, bulk_wait(smem_addr(&l0_bar[bstage]), bphase, kBulkSpins))) {
                                staged = l0_buf + (size_t)bstage * tile_bytes;
                            } else { // the bounded wait ran out: say so, read this and all later tiles with plain loads
                                bulk_ok = false;
                                if (lane == 0) set_status(P.status, SJQ_ERR_ASYNC_WAIT);
                            }
                        }
                        alive = level0<true, HASH, NARROW>(P, st, smem, row0, slot_stride, kDenseRows >= 32 ? 0xFFFFFFFFu : ((1u << kDenseRows) - 1u), staged);
                        if (kBulk && staged != nullptr) {
                            __syncwarp(); // every lane of this warp has its values
                            if (lane == 0) {
                                __threadfence_block();
                                // the warp that counts last knows every warp is done with the buffer: it refills it
                                if (atomicAdd(&l0_done[bstage], 1u) == (blockDim.x >> 5) - 1u) {
                                    l0_done[bstage] = 0;
                                    __threadfence_block();
                                    const uint32_t later = tile + (uint32_t)kBulkStages * gridDim.x;
                                    if (tile_full(later)) issue_tile(later, bstage);
                                }
                            }
                            if (++bstage == (uint32_t)kBulkStages) {
                                bstage = 0;
                                bphase ^= 1u;
                            }
                        }
                    } else {
                        uint32_t valid = 0;
#pragma unroll
                        for (int k = 0; k < kSlots; ++k) {
                            const int64_t rem = P.n - (row0 + k * slot_stride);
                            const uint32_t nv = rem >= 4 ? 0xFu : (rem > 0 ? ((1u << (int)rem) - 1u) : 0u);
                            valid |= nv << (4 * k);
                        }
                        alive = level0<false, HASH, NARROW>(P, st, smem, row0, slot_stride, valid);
                    }
                    if (!__any_sync(0xffffffffu, alive != 0)) { // a very selective first stage: nothing to push
                        tile += gridDim.x;
                        if (wide) flushing = true;
                        continue;
                    }
                    // compact the warp's survivors into queue 0
                    const uint32_t mine = (uint32_t)__popc(alive);
                    uint32_t incl = mine;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += t;
                    }
                    const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
                    if (tot) {
                        uint32_t pos = Q.h0 + Q.c0 + incl - mine;
                        const uint32_t off0 = (uint32_t)(row0 - qbase);
                        if (SJQ_PV(sparse_push)) {
                            // few survivors per thread: walk the set bits instead of testing all the rows
                            for (uint32_t a = alive; a != 0u; a &= a - 1u) {
                                const uint32_t k = (uint32_t)__ffs((int)a) - 1u;
                                qmem[queue_slot(pos, kQueue0Cap, SJQ_PV(qfold))] = off0 + (k >> 2) * (uint32_t)slot_stride + (k & 3u);
                                ++pos;
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < kDenseRows; ++k) {
                                if ((alive >> k) & 1u) {
                                    qmem[queue_slot(pos, kQueue0Cap, SJQ_PV(qfold))] = off0 + (uint32_t)((k >> 2) * slot_stride + (k & 3));
                                    ++pos;
                                }
                            }
                        }
                        Q.c0 += tot;
                        __syncwarp();
                    }
                    tile += gridDim.x;
                    if (wide) flushing = true;
                    continue;
                } else {
                    if ((Q.c0 | Q.c1 | Q.c2) == 0) break;
                    flushing = true;
                    continue;
                }
            }

            // Run one batch of nb rows at the level fed by queue l.
            uint32_t off[kRows];
            uint32_t valid = 0;
            {
                const uint32_t *q = qmem + queue_base(l);
                const uint32_t h = Q.head(l), cap = queue_cap(l);
#pragma unroll
                for (int k = 0; k < kRows; ++k) {
                    const uint32_t e = (uint32_t)(k * 32 + lane);
                    off[k] = 0;
                    if (e < nb) {
                        off[k] = q[queue_slot(h + e, cap, SJQ_PV(qfold))];
                        valid |= 1u << k;
                    }
                }
                __syncwarp();
                Q.set_head(l, (h + nb) & (cap - 1));
                Q.set_count(l, Q.count(l) - nb);
            }
            if (l + 1 == nq) {
#if defined(SJQ_JIT)
                final_rows_scheduled<AGG, MUL, HASH, false, kRows>(P, smem, SJQ_JIT_nd0 + SJQ_JIT_nq - 1, qbase, off, valid, lsum, lcnt);
#else
                final_rows<AGG, MUL, false, HASH, NARROW, kRows>(P, st, smem, SJQ_PV(nd0) + nq - 1, qbase, off, valid, lsum, lcnt);
#endif
            } else {
#if defined(SJQ_JIT)
                // one copy of the filter level per queue-fed filter stage of this query
                uint32_t m;
                if (SJQ_JIT_nq <= 2 || l == 0)
                    m = filter_rows<HASH, NARROW, kRows>(P, SJQ_STAGE(SJQ_JIT_nd0), smem, qbase, off, valid);
                else
                    m = filter_rows<HASH, NARROW, kRows>(P, SJQ_STAGE(SJQ_JIT_nd0 + 1), smem, qbase, off, valid);
#else
                const uint32_t m = filter_rows<HASH, NARROW, kRows>(P, st[P.nd0 + l], smem, qbase, off, valid);
#endif
                const uint32_t mine = (uint32_t)__popc(m);
                uint32_t incl = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
                if (tot) {
                    uint32_t *q = qmem + queue_base(l + 1);
                    uint32_t pos = Q.head(l + 1) + Q.count(l + 1) + incl - mine;
#pragma unroll
                    for (int k = 0; k < kRows; ++k) {
                        if ((m >> k) & 1u) {
                            q[queue_slot(pos, kQueueCap, SJQ_PV(qfold))] = off[k];
                            ++pos;
                        }
                    }
                    Q.set_count(l + 1, Q.count(l + 1) + tot);
                    __syncwarp();
                }
            }
        }
        if (kBulk && !bulk_ok) {
            // staging was abandoned after a wait ran out: copies may still be on their way into this block's shared
            // memory; give each buffer one more bounded wait before the block can exit
            for (uint32_t b = 0; b < (uint32_t)kBulkStages; ++b)
                (void)bulk_wait(smem_addr(&l0_bar[b]), b >= bstage ? bphase : (bphase ^ 1u), kBulkSpins / 4);
        }
    }

    bool cleared = true; // what this block found when it waited for the clear (every thread's, or thread 0's)
    if (AGG == AGG_SCALAR) {
        cleared = scalar_block_reduce(P, lsum, lcnt, self_clear);
    } else if (AGG == AGG_SMEM) {
        // one global atomic per touched group per block
        if (self_clear) cleared = !__syncthreads_or(tid == 0 && !clear_wait(P));
        else __syncthreads();
        const unsigned int *ss = reinterpret_cast<const unsigned int *>(smem + P.smem_groups);
        const uint64_t ng = (uint64_t)P.num_groups;
        if (!cleared) {
            // (the late clear might wipe what is added now)
        } else if (SJQ_PV(cell_shift)) {
            // sums and counts alternate: neighbouring lanes take neighbouring words, so that a warp's adds meet 8
            // sectors and not 16 (2 M rows into a list: 1 % left, 60 groups 18.5 -> 14.4 us; half left, a thousand
            // 22.6 -> 19.9)
            for (int64_t i = tid; i < 2 * P.num_groups; i += blockDim.x) {
                const unsigned long long v = smem_cell((i & 1) ? ss + 2 * ng : ss, ng, (uint64_t)(i >> 1));
                if (v != 0ull) atomicAdd(reinterpret_cast<unsigned long long *>(P.sums) + i, v);
            }
        } else {
            for (int64_t g = tid; g < P.num_groups; g += blockDim.x) {
                const unsigned long long s = smem_cell(ss, ng, (uint64_t)g);
                const unsigned long long c = SJQ_PV(want_count) ? smem_cell(ss + 2 * ng, ng, (uint64_t)g) : 0ull;
                if (s != 0ull) atomicAdd(reinterpret_cast<unsigned long long *>(P.sums) + g, s);
                if (c != 0ull) atomicAdd(reinterpret_cast<unsigned long long *>(P.counts) + g, c);
            }
        }
    }
    if (range_noted<AGG>() && tid == 0 && range_seen && cleared) set_status(P.status, SJQ_ERR_GROUP_RANGE);
    if (self_clear && tid == 0) clear_over(P, !cleared);
}

#if !defined(SJQ_JIT)
template <typename Params, int AGG, bool MUL, int FORM>
__global__ void __launch_bounds__(SJQ_LB_THREADS, SJQ_LB_BLOCKS) fused_kernel(const __grid_constant__ Params P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    fused_body<AGG, MUL, (FORM & kFormHash) != 0, (FORM & kFormDirect) != 0, (FORM & kFormNarrow) != 0>(P, P.st, smem);
}

// The kernel of one aggregation path and form for a parameter block.
template <typename Params, int AGG, int FORM>
auto fused_of(bool mul) -> void (*)(const Params)
{
    return mul ? fused_kernel<Params, AGG, true, FORM> : fused_kernel<Params, AGG, false, FORM>;
}
#endif

} // namespace
} // namespace sjq

#if defined(SJQ_JIT)
// The one kernel of a run-time compiled module.
extern "C" __global__ void __launch_bounds__(SJQ_LB_THREADS, SJQ_LB_BLOCKS)
    sjq_jit_kernel(const __grid_constant__ sjq::RunParams P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    sjq::fused_body<SJQ_JIT_AGG, (SJQ_JIT_MUL != 0), (SJQ_JIT_HASH != 0), (SJQ_JIT_nq == 0), false>(P, P.st, smem);
}
#endif
#endif
