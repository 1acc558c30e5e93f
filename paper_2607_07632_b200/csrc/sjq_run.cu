// Host side of sjq_run: validation, the plan (evaluation order, which tables
// are staged in shared memory, which aggregation path), and the launches.
//
// The order rule follows the paper's observation that bytes moved, not
// arithmetic, decide the run time (Section 3.2): evaluate first what removes
// the most rows per byte read, so that later columns are loaded for few rows.
// The aggregation rule follows Section 3.3: privatise the group table in
// shared memory only when it fits and many survivors contend on it; keep the
// global table when few rows survive or the groups are many.  The rows-per-
// thread choice of Section 4.3.1 ("asymmetric batching") is the fixed four
// rows per 128-bit load here; occupancy supplies the memory-level parallelism.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstring>
#include <vector>

#include "sjq_run.cuh"

// Block size the ahead-of-time kernels are built for (their launch bound); a build for experiments may set another.
#ifndef SJQ_LB_THREADS
#define SJQ_LB_THREADS 384
#endif
#define SJQ_LB_THREADS_MAX SJQ_LB_THREADS

namespace sjq {

sjq_status fused_occupancy(int agg, bool mul, int form, int nstages, int block, size_t smem, int *ctas_per_sm);
sjq_status jit_prepare(const RunParams &P, int agg, bool mul, bool hash, int block, int lb_blocks, size_t smem,
                       int *ctas_per_sm, const void **kernel);
sjq_status jit_launch(const void *kernel, const RunParams &P, int grid, int block, size_t smem, bool behind,
                      cudaStream_t stream);
sjq_status fused_launch(int agg, bool mul, int form, int grid, int block, size_t smem, bool behind,
                        const RunParams &P, cudaStream_t stream);
sjq_status clear_launch(int64_t *sums, int64_t *counts, int64_t cells, int64_t *gkeys, int64_t gslots,
                        int64_t *n_groups, int32_t *status, int at_once, int sm_count, cudaStream_t stream);
sjq_status compact_launch(const int64_t *gkeys, const int64_t *cells, int64_t gslots, bool indexed,
                          int64_t dense_base, unsigned int *block_counts, int64_t *keys, int64_t *sums,
                          int64_t *counts, int64_t capacity, int64_t *n_groups, int32_t *status, int sm_count,
                          int beside, cudaStream_t stream, int *launches);

int host_stats_release();
size_t unfused_scratch_bytes(int64_t n, int gathering_joins);
sjq_status unfused_launch(const RunParams &P, int nfilter, int agg, bool mul, bool has_hash, void *scratch,
                          size_t scratch_bytes, int sm_count, cudaStream_t stream, int *launches);
sjq_status sample_launch(const sjq_col *fact, const DPred *preds, int npreds, int64_t n, unsigned long long *counts,
                         cudaStream_t stream);
sjq_status hot_launch(const void *col, bool is64, int64_t n, const sjq_table *T, void *scratch, cudaStream_t stream,
                      const void **hot_table, int *launches);
sjq_status merge_launch(const int64_t *keys, const int64_t *sums, const int64_t *counts, int64_t n, int64_t *gkeys,
                        int64_t *cells, uint64_t gmask, int32_t *status, int sm_count, cudaStream_t stream);

namespace {

// A list with room for everything the planner can put in it: the planning of a run allocates nothing.
template <typename T, int N>
struct Short {
    T items[N];
    int count = 0;

    Short() {}
    Short(int n, const T &v) : count(n)
    {
        for (int i = 0; i < n; ++i) items[i] = v;
    }
    void push_back(const T &v) { items[count++] = v; }
    void resize(int n) { count = n; }
    int size() const { return count; }
    T &operator[](int i) { return items[i]; }
    const T &operator[](int i) const { return items[i]; }
    T *begin() { return items; }
    T *end() { return items + count; }
    const T *begin() const { return items; }
    const T *end() const { return items + count; }
};

struct StageSpec {
    int kind;     // ST_PRED / ST_PROBE / ST_LOAD
    int index;    // predicate or join index (-1 for loads)
    int col;      // fact column
    double sel;   // estimated fraction of rows passing
    int width;    // bytes of a value of the column
    double cost;  // picoseconds per row evaluated, the column's bytes apart
    int prefilter; // 1: only the presence bitmap of a hashed join; 2: the exact probe that follows one
};
constexpr int kMaxFilters = SJQ_MAX_PREDS + 2 * SJQ_MAX_JOINS; // (a hashed join is two)
typedef Short<StageSpec, kMaxFilters> Specs;
typedef Short<int, kMaxFilters> Order;

// share of the rows surviving all filters from which a compiled kernel drops the survivor queues
constexpr double kDirectSurvival = 0.35;       // register accumulators
constexpr double kDirectSurvivalGrouped = 0.75; // group tables

double pred_selectivity(const sjq_pred &p)
{
    switch (p.op) {
    case SJQ_EQ: return 0.1;
    case SJQ_NE: return 0.9;
    case SJQ_IN: return std::min(0.5, 0.1 * std::max(1, p.nset));
    case SJQ_BETWEEN: return 0.25;
    default: return 0.4;
    }
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

uint64_t hashed_slots(int64_t capacity)
{
    uint64_t want = (uint64_t)std::max<int64_t>(capacity, 8) * 2;
    uint64_t slots = 16;
    while (slots < want) slots <<= 1;
    return slots;
}

bool valid_term(const sjq_term &t, int nfact, const sjq_join *joins, int njoins)
{
    if (t.src == SJQ_SRC_FACT) return t.a >= 0 && t.a < nfact;
    if (t.src == SJQ_SRC_PAYLOAD)
        return t.a >= 0 && t.a < njoins && t.b >= 0 && t.b < joins[t.a].table->layout.npayload;
    return false;
}

// A map staged in part (see there): from so many rows on, so much of it, in so much dynamic shared memory (a carve-out of 196
// KB less what the system and the kernel's own arrays take); and the rows from which chains are longer.
constexpr int64_t kPartRows = (int64_t)1 << 24;
constexpr size_t kPartBytes = (size_t)192 << 10;
constexpr size_t kPartCarveOut = ((size_t)196 << 10) - 1024 - 640;
constexpr int64_t kLongChainRows = (int64_t)1 << 26;

// What a filter stage costs, in picoseconds per fact row on the whole chip (148 SMs, 1.9 GHz, 6.5 TB/s).
constexpr double kPsByte = 0.154;  // a byte of DRAM traffic
constexpr double kPsIssue = 0.3;   // evaluating a row (about ten instructions)
constexpr double kPsShared = 0.4;  // a probe of a table staged in shared memory (random banks)
constexpr double kPsGlobal = 3.4;  // a probe of a global table: 32 random lines take the L1 32 cycles, whatever hits
constexpr double kPsFar = 10.0;    // ... of a table that the L2 cannot hold
constexpr size_t kStageBytes = (size_t)32 << 10; // tables up to this size are copied into shared memory
constexpr size_t kNearL2 = (size_t)64 << 20;

// DRAM delivers 64-byte pieces: one of a column is read iff one of its rows is still alive.
double column_ps(int width, double reach)
{
    double dead = 1.0 - std::min(1.0, reach);
    for (int rows = 64 / width; rows > 1; rows >>= 1) dead *= dead;
    return kPsByte * width * (1.0 - dead);
}

// The order of the filter stages with the least estimated time: the sum over the stages of the column's bytes
// (once per column, at the share of rows that reach it) and of the probes.  The share depends only on which stages
// came before, so the best order is found over subsets (up to 8 stages; one at a time, cheapest per row dropped
// first, beyond).  Exact probes behind a presence bitmap go last: they run at the final level.
// (Ranking by (1 - selectivity) / cost with one cost for every table below 200 KB left city x brand to chance: two
// joins that keep one row in 25, one probing 25 KB in shared memory, the other 175 KB through the L1, which is
// 0.67 or 3.3 ms for 600 M rows with the one or the other first.)
// `column(spec, reach)`: what reading a stage's column for the rows that reach it costs.
template <typename Column>
Order cheapest_order(const Specs &specs, Column column)
{
    constexpr int kExhaustive = 8;
    const int n = (int)specs.size();
    int early[kMaxFilters], m = 0;
    Order order;
    for (int i = 0; i < n; ++i)
        if (specs[i].prefilter != 2) early[m++] = i;
    auto cost = [&](int i, double reach, bool column_read) {
        return (column_read ? 0.0 : column(specs[i], reach)) + reach * specs[i].cost;
    };
    if (m <= kExhaustive) {
        struct Best { double ps, reach; int last; } best[1 << kExhaustive];
        unsigned same_col[kExhaustive]; // the stages that read the column of stage i
        for (int i = 0; i < m; ++i) {
            same_col[i] = 0;
            for (int j = 0; j < m; ++j) same_col[i] |= (unsigned)(specs[early[j]].col == specs[early[i]].col) << j;
        }
        const unsigned all = (1u << m) - 1u;
        for (unsigned set = 0; set <= all; ++set) best[set] = Best{set ? 1e300 : 0.0, 1.0, -1};
        for (unsigned set = 0; set < all; ++set) {
            for (int i = 0; i < m; ++i) {
                if (set >> i & 1u) continue;
                const double ps = best[set].ps + cost(early[i], best[set].reach, (same_col[i] & set) != 0);
                Best &to = best[set | 1u << i];
                if (ps < to.ps) to = Best{ps, best[set].reach * specs[early[i]].sel, i};
            }
        }
        for (unsigned set = all; set; set ^= 1u << best[set].last) order.push_back(early[best[set].last]);
        std::reverse(order.begin(), order.end());
    } else {
        double reach = 1.0;
        Short<char, kMaxFilters> used(n, 0);
        for (int k = 0; k < m; ++k) {
            int pick = -1;
            double least = 0.0;
            for (int e = 0; e < m; ++e) {
                const int i = early[e];
                if (used[i]) continue;
                bool column_read = false;
                for (int j : order) column_read |= specs[j].col == specs[i].col;
                const double per_drop = cost(i, reach, column_read) / std::max(1e-9, 1.0 - specs[i].sel);
                if (pick < 0 || per_drop < least) pick = i, least = per_drop;
            }
            used[pick] = 1;
            order.push_back(pick);
            reach *= specs[pick].sel;
        }
    }
    for (int i = 0; i < n; ++i)
        if (specs[i].prefilter == 2) order.push_back(i);
    return order;
}

// The filter stages of a query (its predicates and joins; a hashed join with a presence bitmap is two
// stages) with estimated selectivities and costs, and the order they are evaluated in: the caller's, or
// the cheapest.
sjq_status order_stages(const sjq_col *fact, const sjq_pred *preds, int npreds, const sjq_join *joins, int njoins,
                        const sjq_run_opts &opts, Specs *specs_out, Order *order_out)
{
    Specs &specs = *specs_out;
    Order &order = *order_out;
    // a measured pass fraction (parts per million) replaces the estimate where the caller supplies one
    auto hinted = [&](int i, double estimate) {
        const int32_t ppm = opts.pass_ppm[i];
        return ppm > 0 ? std::min(1.0, ppm / 1e6) : estimate;
    };
    for (int p = 0; p < npreds; ++p)
        specs.push_back({ST_PRED, p, preds[p].col, hinted(p, pred_selectivity(preds[p])),
                         fact[preds[p].col].dtype == SJQ_I64 ? 8 : 4, kPsIssue, 0});
    for (int j = 0; j < njoins; ++j) {
        const sjq_table *T = joins[j].table;
        const sjq_dim_layout &L = T->layout;
        const int width = L.key_dtype == SJQ_I64 ? 8 : 4;
        const double sel = hinted(npreds + j, L.dim_rows > 0 ? (double)L.entries / (double)L.dim_rows : 0.0);
        // bytes a filter stage on this table touches: the presence bitmap when a direct table has one
        const bool direct = is_direct_kind(L.kind);
        const size_t tb = !direct ? L.table_bytes
                          : (L.filter_bits > 0 && T->filter && !opts.no_filter_bitmap) ? (size_t)(L.filter_bits / 8)
                                                                                      : T->slots_bytes;
        const size_t staged_up_to = opts.smem_tables == 0 ? kStageBytes
                                    : opts.smem_tables == 1 ? 0
                                    : opts.smem_tables >= 1024 ? (size_t)opts.smem_tables
                                                               : (size_t)128 << 10;
        const double probe = direct && tb <= staged_up_to ? kPsShared : tb <= kNearL2 ? kPsGlobal : kPsFar;
        if (is_hash_kind(L.kind) && T->filter && L.filter_bits > 0) {
            // a hashed join is two stages: its presence bitmap (cheap, passes the hits and ~1/16 of the
            // misses) early, the exact probe (expensive) on what is left
            const double fp = std::min(1.0, (double)L.entries / (double)L.filter_bits);
            const double pass = std::min(1.0, sel + (1.0 - sel) * fp);
            specs.push_back({ST_PROBE, j, joins[j].fk_col, pass, width, kPsGlobal + kPsIssue, 1});
            specs.push_back({ST_PROBE, j, joins[j].fk_col, pass > 0 ? std::min(1.0, sel / pass) : 1.0, width,
                             probe + kPsIssue, 2});
            continue;
        }
        specs.push_back({ST_PROBE, j, joins[j].fk_col, std::min(1.0, sel), width, probe + kPsIssue, 0});
    }
    const int nfilter = (int)specs.size();
    if (opts.norder) {
        // the caller orders predicates and joins; a hashed join's bitmap and exact probe stay adjacent
        Short<char, SJQ_MAX_PREDS + SJQ_MAX_JOINS> seen(npreds + njoins, 0);
        for (int i = 0; i < npreds + njoins; ++i) {
            const int o = opts.order[i];
            if (o < 0 || o >= npreds + njoins || seen[o]) return SJQ_ERR_INVALID_ARG;
            seen[o] = 1;
            for (int k = 0; k < nfilter; ++k) {
                const bool match = o < npreds ? (specs[k].kind == ST_PRED && specs[k].index == o)
                                              : (specs[k].kind == ST_PROBE && specs[k].index == o - npreds);
                if (match) order.push_back(k);
            }
        }
    } else {
        order = cheapest_order(specs, [](const StageSpec &sp, double reach) { return column_ps(sp.width, reach); });
    }

    return SJQ_OK;
}

} // namespace
} // namespace sjq

using namespace sjq;

extern "C" sjq_status sjq_unfused_scratch_bytes(int64_t rows, int njoins, size_t *bytes)
{
    if (rows < 0 || njoins < 0 || njoins > SJQ_MAX_JOINS || !bytes) return SJQ_ERR_INVALID_ARG;
    *bytes = unfused_scratch_bytes(rows, njoins);
    return SJQ_OK;
}

extern "C" sjq_status sjq_run_workspace_bytes(const sjq_result_spec *spec, size_t *bytes)
{
    if (!spec || !bytes) return SJQ_ERR_INVALID_ARG;
    *bytes = 0;
    if (spec->mode == SJQ_HASHED) {
        if (spec->capacity <= 0) return SJQ_ERR_INVALID_ARG;
        *bytes = align_up((size_t)(hashed_slots(spec->capacity) + 1) * 8, 256) * 3;
    } else if (spec->mode != SJQ_SCALAR && spec->mode != SJQ_DENSE) {
        return SJQ_ERR_INVALID_ARG;
    }
    return SJQ_OK;
}

// ---------------------------------------------------------------------------
// Measured predicate selectivities.
namespace {

int32_t ppm_of(int64_t passed, int64_t sampled)
{
    if (sampled <= 0) return 0; // nothing sampled: no hint
    const int64_t ppm = (passed * 1000000 + sampled / 2) / sampled;
    return (int32_t)std::min<int64_t>(std::max<int64_t>(ppm, 1), 1000000);
}

} // namespace

extern "C" sjq_status sjq_pred_sample_begin(const sjq_col *fact, int nfact, const sjq_pred *preds, int npreds,
                                            void *scratch_dev, int64_t *host_counts, void *stream_)
{
    if (!fact || nfact <= 0 || nfact > 64 || npreds < 0 || npreds > SJQ_MAX_PREDS || (npreds && !preds) ||
        !scratch_dev || !host_counts)
        return SJQ_ERR_INVALID_ARG;
    if (!aligned16(scratch_dev)) return SJQ_ERR_ALIGN;
    const int64_t n = fact[0].n;
    DPred d[SJQ_MAX_PREDS];
    for (int c = 0; c < nfact; ++c) {
        if (fact[c].n != n || n < 0 || (fact[c].dtype != SJQ_I32 && fact[c].dtype != SJQ_I64) ||
            (n > 0 && !fact[c].data))
            return SJQ_ERR_INVALID_ARG;
        if (!aligned16(fact[c].data)) return SJQ_ERR_ALIGN;
    }
    for (int p = 0; p < npreds; ++p) {
        if (preds[p].col < 0 || preds[p].col >= nfact) return SJQ_ERR_INVALID_ARG;
        if (!canon_pred(preds[p], fact[preds[p].col].dtype, &d[p])) return SJQ_ERR_INVALID_ARG;
    }
    cudaStream_t stream = (cudaStream_t)stream_;
    unsigned long long *counts = static_cast<unsigned long long *>(scratch_dev);
    sjq_status st = sample_launch(fact, d, npreds, n, counts, stream);
    if (st != SJQ_OK) return st;
    if (cudaMemcpyAsync(host_counts, counts, (SJQ_MAX_PREDS + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, stream) !=
        cudaSuccess) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    return SJQ_OK;
}

extern "C" sjq_status sjq_pred_sample_end(const int64_t *host_counts, int npreds, int32_t *pass_ppm)
{
    if (!host_counts || npreds < 0 || npreds > SJQ_MAX_PREDS || (npreds && !pass_ppm)) return SJQ_ERR_INVALID_ARG;
    for (int p = 0; p < npreds; ++p) pass_ppm[p] = ppm_of(host_counts[1 + p], host_counts[0]);
    return SJQ_OK;
}

extern "C" sjq_status sjq_pred_sample(const sjq_col *fact, int nfact, const sjq_pred *preds, int npreds,
                                      void *scratch_dev, void *stream_, int32_t *pass_ppm)
{
    int64_t h[SJQ_MAX_PREDS + 1];
    sjq_status st = sjq_pred_sample_begin(fact, nfact, preds, npreds, scratch_dev, h, stream_);
    if (st != SJQ_OK) return st;
    if (cudaStreamSynchronize((cudaStream_t)stream_) != cudaSuccess) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    return sjq_pred_sample_end(h, npreds, pass_ppm);
}

namespace {

// A number that no other call has: the flags of a pass that clears its results hold it.
uint64_t next_epoch()
{
    static std::atomic<uint64_t> last{(uint64_t)std::chrono::steady_clock::now().time_since_epoch().count() << 20};
    return ++last | 1ull << 63;
}

// What a run is part of: by default of nothing, its columns are in device memory and its options are the caller's.
struct RunContext {
    // the order of the filters, if the options give one, is the caller's own and not one that this library chose for a
    // run from host memory
    bool callers_order = true;
    // some columns are read in place from host memory
    bool in_place = false;
    // rows to plan for where they are not the call's own: a last chunk is planned as the others, so that a compiled
    // kernel is not compiled again for it
    int64_t rows = -1;
};

} // namespace

static sjq_status run_planned(const sjq_col *fact, int nfact, const sjq_pred *preds, int npreds,
                              const sjq_join *joins, int njoins, const sjq_key_expr *key, const sjq_agg_expr *agg,
                              const sjq_result_spec *spec, const sjq_result *out, const sjq_run_opts *opts_,
                              const RunContext &context, void *stream_, sjq_run_info *info)
{
    // ------------------------------------------------------------ validation
    if (!fact || nfact <= 0 || nfact > 64 || npreds < 0 || npreds > SJQ_MAX_PREDS || (npreds && !preds) ||
        njoins < 0 || njoins > SJQ_MAX_JOINS || (njoins && !joins) || !agg || !spec || !out || !out->status ||
        !out->sums)
        return SJQ_ERR_INVALID_ARG;
    sjq_run_opts opts{};
    if (opts_) opts = *opts_;
    const int64_t n = fact[0].n;
    if (n < 0) return SJQ_ERR_INVALID_ARG;
    for (int c = 0; c < nfact; ++c) {
        if (fact[c].n != n || (fact[c].dtype != SJQ_I32 && fact[c].dtype != SJQ_I64)) return SJQ_ERR_INVALID_ARG;
        if (n > 0 && !fact[c].data) return SJQ_ERR_INVALID_ARG;
        if (!aligned16(fact[c].data)) return SJQ_ERR_ALIGN;
    }
    if (spec->mode != SJQ_SCALAR && spec->mode != SJQ_DENSE && spec->mode != SJQ_HASHED) return SJQ_ERR_INVALID_ARG;
    if ((spec->mode == SJQ_SCALAR) != (key == nullptr)) return SJQ_ERR_INVALID_ARG;
    if (spec->mode == SJQ_DENSE && spec->num_groups <= 0) return SJQ_ERR_INVALID_ARG;
    if (spec->mode == SJQ_HASHED &&
        (spec->capacity <= 0 || !out->keys || !out->counts || !out->n_groups || !out->workspace))
        return SJQ_ERR_INVALID_ARG;
    if (agg->want_count && !out->counts) return SJQ_ERR_INVALID_ARG;
    if (agg->op < SJQ_AGG_COL || agg->op > SJQ_AGG_ADD) return SJQ_ERR_INVALID_ARG;
    if (!aligned16(out->sums) || !aligned16(out->counts) || !aligned16(out->keys) || !aligned16(out->workspace) ||
        (reinterpret_cast<uintptr_t>(out->status) & 3u) || (reinterpret_cast<uintptr_t>(out->n_groups) & 7u))
        return SJQ_ERR_ALIGN;
    for (int j = 0; j < njoins; ++j) {
        const sjq_table *T = joins[j].table;
        if (!T || T->magic != kTableMagic || joins[j].fk_col < 0 || joins[j].fk_col >= nfact)
            return SJQ_ERR_INVALID_ARG;
        if (fact[joins[j].fk_col].dtype != T->layout.key_dtype) return SJQ_ERR_UNSUPPORTED;
    }
    for (int p = 0; p < npreds; ++p)
        if (preds[p].col < 0 || preds[p].col >= nfact) return SJQ_ERR_INVALID_ARG;
    if (key) {
        if (key->nterms < 0 || key->nterms > SJQ_MAX_KEY_TERMS) return SJQ_ERR_INVALID_ARG;
        for (int t = 0; t < key->nterms; ++t)
            if (!valid_term(key->t[t], nfact, joins, njoins)) return SJQ_ERR_INVALID_ARG;
    }
    if (!valid_term(agg->x, nfact, joins, njoins)) return SJQ_ERR_INVALID_ARG;
    if (agg->op != SJQ_AGG_COL && !valid_term(agg->y, nfact, joins, njoins)) return SJQ_ERR_INVALID_ARG;
    // the ahead-of-time kernels are bounded at SJQ_LB_THREADS_MAX; a specialised kernel is compiled for its block size
    if (opts.block_threads && (opts.block_threads < 128 || opts.block_threads % 32 ||
                               opts.block_threads > (opts.specialise ? 1024 : SJQ_LB_THREADS_MAX)))
        return SJQ_ERR_INVALID_ARG;
    if (opts.rows_per_lane != 0 && opts.rows_per_lane != 4 && !(opts.rows_per_lane == 8 && opts.specialise))
        return SJQ_ERR_INVALID_ARG;
    if (opts.dense_slots != 0 && opts.dense_slots != 2 && !(opts.dense_slots == 4 && opts.specialise))
        return SJQ_ERR_INVALID_ARG;
    if (opts.norder && opts.norder != npreds + njoins) return SJQ_ERR_INVALID_ARG;
    if (opts.hot_keys < 0 || opts.hot_keys > 2) return SJQ_ERR_INVALID_ARG;
    if (opts.hot_scratch && !aligned16(opts.hot_scratch)) return SJQ_ERR_ALIGN;
    if (reinterpret_cast<uintptr_t>(opts.sync) & 7u) return SJQ_ERR_ALIGN;

    DeviceInfo dev;
    sjq_status st = device_info(&dev);
    if (st != SJQ_OK) return st;
    cudaStream_t stream = (cudaStream_t)stream_;

    // ------------------------------------------------------------ stage list
    Specs specs;
    Order order;
    if ((st = order_stages(fact, preds, npreds, joins, njoins, opts, &specs, &order)) != SJQ_OK) return st;
    const int nfilter = (int)specs.size();

    // ------------------------------------------------------------ accumulators
    // Every term adds mult * value to one accumulator; fold the expressions
    // into per-source multipliers: src_mult[source][dest].
    struct Contribution { int src, a, b, dest; int64_t mult; };
    Short<Contribution, SJQ_MAX_KEY_TERMS + 2> contrib;
    auto add_term = [&](const sjq_term &t, int dest, int64_t sign) {
        contrib.push_back({t.src, t.a, t.b, dest, (int64_t)((uint64_t)t.mult * (uint64_t)sign)});
    };
    // a key taken modulo 1 is 0 whatever its terms are: they are neither loaded nor gathered
    if (key && key->modulo != 1)
        for (int t = 0; t < key->nterms; ++t) add_term(key->t[t], kAccKey, 1);
    const bool mul = agg->op == SJQ_AGG_MUL;
    add_term(agg->x, kAccX, 1);
    if (agg->op == SJQ_AGG_MUL) add_term(agg->y, kAccY, 1);
    if (agg->op == SJQ_AGG_SUB) add_term(agg->y, kAccX, -1);
    if (agg->op == SJQ_AGG_ADD) add_term(agg->y, kAccX, 1);

    RunParams P;
    std::memset(static_cast<RunCore *>(&P), 0, sizeof(RunCore)); // (stages are cleared as they are filled)
    P.n = n;
    int ns = 0;
    int nsets = 0;
    Short<int, SJQ_MAX_JOINS> stage_of_join(njoins, -1);
    Short<int, 64> stage_of_col(nfact, -1);
    Short<int, kMaxStages> stage_label;
    auto fill_stage = [&](DStage &S, const StageSpec &sp) -> sjq_status {
        std::memset(&S, 0, sizeof(S));
        S.kind = (uint8_t)sp.kind;
        S.col = fact[sp.col].data;
        S.is64 = (uint8_t)(fact[sp.col].dtype == SJQ_I64);
        S.col32 = S.is64 && (reinterpret_cast<uintptr_t>(S.col) & 31u) == 0;
        S.op = OP_LOAD;
        if (sp.kind == ST_PRED) {
            DPred d;
            if (!canon_pred(preds[sp.index], fact[sp.col].dtype, &d)) return SJQ_ERR_INVALID_ARG;
            if (d.nset) {
                S.op = OP_PRED_SET;
                S.nset = d.nset;
                S.set_idx = (uint8_t)nsets;
                for (int k = 0; k < d.nset; ++k) P.sets[nsets][k] = d.set[k];
                ++nsets;
            } else {
                S.op = OP_PRED_RANGE;
                S.lo = d.lo;
                S.hi = d.hi;
                S.neg = d.neg;
                S.never = d.never;
                S.lo32 = d.lo32;
                S.width32 = d.never ? 0u : (uint32_t)d.hi32 - (uint32_t)d.lo32;
            }
        } else if (sp.kind == ST_PROBE) {
            const sjq_table *T = joins[sp.index].table;
            const sjq_dim_layout &L = T->layout;
            if (L.slots > ((int64_t)1 << 31) && is_hash_kind(L.kind)) return SJQ_ERR_UNSUPPORTED;
            S.op = (uint8_t)(L.kind == SJQ_TABLE_DIRECT_BITMAP ? OP_DIRECT_BITMAP
                             : L.kind == SJQ_TABLE_DIRECT_U8   ? OP_DIRECT_U8
                             : L.kind == SJQ_TABLE_DIRECT_U16  ? OP_DIRECT_U16
                             : L.kind == SJQ_TABLE_DIRECT_U32  ? OP_DIRECT_U32
                             : L.kind == SJQ_TABLE_DIRECT_U64  ? OP_DIRECT_U64
                             : L.kind == SJQ_TABLE_DIRECT_U4   ? OP_DIRECT_U4
                             : L.kind == SJQ_TABLE_DIRECT_U2   ? OP_DIRECT_U2
                             : L.kind == SJQ_TABLE_HASH_I32    ? OP_HASH32
                                                               : OP_HASH64);
            S.tab = T->slots;
            S.kmin = L.kmin;
            S.last = (uint64_t)L.slots - 1;
            S.full = (uint8_t)(L.code_bits > 0 && L.code_bits < 8 && L.entries == L.slots);
            if (is_hash_kind(L.kind)) {
                S.last = (uint64_t)(T->slots_bytes / kBucketBytes); // bucket count
                S.wide = (uint8_t)((reinterpret_cast<uintptr_t>(T->slots) & 31u) == 0);
                if (sp.prefilter == 1) {
                    S.op = OP_HASHBITS;
                    S.tab = T->filter;
                }
            }
            S.kmin32 = (int32_t)L.kmin;
            S.last32 = (uint32_t)std::min<uint64_t>((uint64_t)L.slots - 1, 0xFFFFFFFFull);
            // with 2^32 slots or more every 32-bit index is in range and nothing is clamped
            S.clamp32 = (uint32_t)std::min<uint64_t>((uint64_t)L.slots, 0xFFFFFFFFull);
            S.hmask = sp.prefilter == 1 ? (uint64_t)L.filter_bits - 1 : 0;
            S.pmin0 = L.pay_min[0];
            S.pmin1 = L.pay_min[1];
            S.pbits0 = (uint8_t)L.pay_bits[0];
            S.pmask0 = L.pay_bits[0] >= 64 ? ~0ULL : ((1ULL << L.pay_bits[0]) - 1ULL);
            S.code_bits = (uint8_t)L.code_bits;
            S.tab_bytes = (uint32_t)std::min<size_t>(T->slots_bytes, 0xFFFFFFF0u);
        }
        return SJQ_OK;
    };
    for (int i = 0; i < nfilter; ++i) {
        const StageSpec &sp = specs[order[i]];
        if (ns >= kMaxStages) return SJQ_ERR_UNSUPPORTED;
        if ((st = fill_stage(P.st[ns], sp)) != SJQ_OK) return st;
        if (sp.kind == ST_PROBE && sp.prefilter != 1) stage_of_join[sp.index] = ns;
        if (stage_of_col[sp.col] < 0) stage_of_col[sp.col] = ns;
        stage_label.push_back(sp.kind == ST_PRED ? sp.index : npreds + sp.index);
        ++ns;
    }
    P.want_count = agg->want_count ? 1 : 0;
    P.status = out->status;
    if (key) {
        P.key_offset = key->offset;
        P.modulo = key->modulo;
        if (key->modulo > 0 && (key->modulo & (key->modulo - 1)) == 0) P.modmask = (uint64_t)key->modulo - 1;
        P.mod32 = key->modulo > 0 && key->modulo <= 0xFFFFFFFFLL;
    }

    // ------------------------------------------------------------ dense / sparse split
    // Fraction of rows reaching each filter stage, from the estimates.
    Short<double, kMaxFilters + 1> reach(nfilter + 1, 1.0);
    for (int s = 0; s < nfilter; ++s) reach[s + 1] = reach[s] * specs[order[s]].sel;
    const int64_t plan_rows = context.rows >= 0 ? context.rows : n;
    const double survivors = (double)plan_rows * reach[nfilter];
    // Level 0 runs, on thread-owned rows, the leading filter stages that still see a fair share of
    // the rows (a dense stage costs about the same per table row whatever survives, a queue-fed
    // level costs per surviving row, several times more: measured break-even between 20 % and 30 %).
    // Up to kMaxQueues - 1 later filter stages run as queue-fed levels; the rest at the final level.
    // Eager loading and compaction = never use no queue at all.
    int nd0 = 0, nfq = 0;
    // Most rows surviving every filter (by the measured fractions): each column is read for nearly every
    // 32-byte sector anyway, so queues would only add shared-memory traffic and turn 128-bit loads into 4-byte
    // ones.  A kernel compiled for the query then keeps thread-owned rows throughout and requests its columns
    // up front.
    // (A group-by terminal works on whatever lanes still hold a row, so with a shared-memory or global group
    // table compacted survivors keep paying until nearly all rows survive: measured on the selectivity sweep at
    // 50 %, one group 1.78 -> 1.44 ms without queues, a thousand groups 2.13 -> 2.32 ms.)
    const bool register_terminal = spec->mode == SJQ_SCALAR || (spec->mode == SJQ_DENSE && spec->num_groups == 1);
    const bool mostly_survive = opts.specialise && opts.compaction == 0 &&
                                reach[nfilter] >= (register_terminal ? kDirectSurvival : kDirectSurvivalGrouped);
    // Few rows: the kernel's time is a chain of memory latencies, one per queue level, and without queues it is one in
    // all (compiled, 400 thousand rows: city x city 12.5 -> 8.7 us, city x brand 14.6 -> 12.6, the others alike;
    // interpreted: four joins 16.6 -> 12.5, two joins 14.5 -> 10.5, filter and sum 12.5 -> 10.4; at 800 thousand rows
    // some gain and some lose).  Not where a column is read in place from host memory: a kernel without queues requests
    // columns before it knows which rows need them, four rows at a time, and would bring most of it over the bus.
    // Nor where the caller sets an option that only a kernel with queues can carry out.
    const bool asks_for_queues = opts.rows_per_lane || opts.dense_slots || opts.l0_bulk == 1 || opts.l0_bulk == 3;
    const bool few_rows = plan_rows <= (int64_t)1 << 19 && opts.compaction == 0 && !context.in_place && !asks_for_queues;
    const bool direct = few_rows || opts.eager_loads || opts.compaction == 1 || nfilter == 0 || opts.unfused || mostly_survive;
    if (!direct) {
        nd0 = 1;
        if (opts.compaction != 2) {
            const double dense_reach = 0.3;
            while (nd0 < nfilter && specs[order[nd0]].sel < 0.9 && reach[nd0] > dense_reach &&
                   specs[order[nd0]].prefilter != 2)
                ++nd0;
            // A queue of its own pays for a filter that still sees more than about one row in eight; a later one is
            // better taken at the final level, whose columns a compiled kernel requests together (600 M rows: four
            // joins, the third filter reached by 6 % of the rows, 1286 us with a queue for it and 1223 without, but
            // 1295 without one for the second, reached by 20 %; filter and sum, 4 %: 1280 and 1109; two joins, 4 %:
            // 783 and 735).  The interpreting kernel loads its columns one after the other and is better off with
            // queues (four joins, 60 M rows: 175 us against 290 without any), and beyond the few rows above an order
            // that the caller lays down is carried out with a level for every filter.
            const double queue_reach = opts.specialise && !(opts.norder && context.callers_order) ? 0.12 : 0.002;
            while (nd0 + nfq < nfilter && nfq < kMaxQueues - 1 && specs[order[nd0 + nfq]].sel < 0.9 &&
                   reach[nd0 + nfq] > queue_reach && specs[order[nd0 + nfq]].prefilter != 2)
                ++nfq;
        }
    }
    const int ndense = nd0 + nfq; // stages that only filter (no accumulators)
    P.nd0 = nd0;
    P.nq = direct ? 0 : nfq + 1;
    P.rows = opts.rows_per_lane ? opts.rows_per_lane : 4;
    // Few survivors of level 0 leave a compiled kernel room for sixteen rows per thread: twice the loads in flight for
    // the column that every row reads (200 M rows: two joins, 4 % left, 282 -> 250 us; city x brand, 4 %, 261 -> 220;
    // the sweep into a thousand groups at 1, 3, 6, 10 %, 210 -> 201, 297 -> 290, 354 -> 348, 412 -> 406).  With more
    // left the first queue, twice as large, costs more than it gives (14 % 447 -> 447, 20 % 477 -> 485; four joins,
    // 20 %, 409 -> 438), with next to none the lane's longer test of its rows does (0.1 % 127 -> 131).
    const bool few_left = opts.specialise && P.nq && reach[nd0] < 0.15;
    const bool sixteen = opts.dense_slots == 4 || (opts.dense_slots == 0 && few_left && reach[nd0] >= 0.005 && reach[nd0] < 0.12);
    P.slots = opts.specialise && sixteen ? 4 : 2;
    // a third or more of the rows reaching the first queue: pushes are dense enough for bank conflicts to matter
    P.qfold = (opts.specialise && P.nq && reach[nd0] >= 0.3) ? 7u : 0u;
    // fewer than about one row in seven surviving level 0: pushing by walking the set bits of a thread's mask beats
    // testing its eight rows one by one (city x brand 0.72 -> 0.68 ms, city x city 0.72 -> 0.71; at one in five,
    // the four-join workload, it loses: 1.19 -> 1.21 ms)
    P.sparse_push = few_left ? 1 : 0;

    // Sources of the accumulators.  A dense stage cannot feed an accumulator
    // (it only keeps a bit per row), so a value it would supply is gathered
    // again for the survivors by a sparse copy of the stage.
    Short<int, kMaxStages> gather_of_stage(ns, -1);
    for (const Contribution &c : contrib) {
        int s, src;
        if (c.src == SJQ_SRC_FACT) {
            if (stage_of_col[c.a] < 0) { // a column nobody filters on: plain load stage at the end
                if (ns >= kMaxStages) return SJQ_ERR_UNSUPPORTED;
                StageSpec sp{ST_LOAD, -1, c.a, 1.0, 4, 0.0, 0};
                fill_stage(P.st[ns], sp);
                stage_of_col[c.a] = ns;
                stage_label.push_back(-1);
                gather_of_stage.push_back(-1);
                ++ns;
            }
            s = stage_of_col[c.a];
            src = 0;
        } else {
            s = stage_of_join[c.a];
            src = 1 + c.b;
        }
        if (s < ndense) {
            if (gather_of_stage[s] < 0) {
                if (ns >= kMaxStages) return SJQ_ERR_UNSUPPORTED;
                P.st[ns] = P.st[s];
                gather_of_stage[s] = ns;
                stage_label.push_back(stage_label[s]);
                gather_of_stage.push_back(-1);
                ++ns;
            }
            s = gather_of_stage[s];
        }
        DStage &S = P.st[s];
        const int slot = 3 * src + c.dest;
        S.mult[slot] = (int64_t)((uint64_t)S.mult[slot] + (uint64_t)c.mult);
        S.acc |= (uint16_t)(1u << slot);
    }
    // a gathered copy that only needs the raw value need not filter again
    for (int s = ndense; s < ns; ++s) {
        DStage &S = P.st[s];
        bool is_copy = false;
        for (int d = 0; d < ndense; ++d) is_copy |= gather_of_stage[d] == s;
        if (is_copy && (S.acc & ~0x7u) == 0) {
            S.kind = ST_LOAD;
            S.op = OP_LOAD;
        }
    }
    // A filter stage on a direct table with payloads probes the table's presence bitmap (an eighth to a
    // sixty-fourth of the code array, so far more of it stays in L1/L2); the payload is gathered from the
    // codes by the sparse copy, for the survivors only.
    Short<char, kMaxStages> via_bitmap(ns, 0);
    if (!opts.no_filter_bitmap) {
        for (int s = 0; s < ndense; ++s) {
            DStage &S = P.st[s];
            if (S.kind != ST_PROBE || !is_code_op(S.op)) continue;
            const sjq_table *T = joins[specs[order[s]].index].table;
            if (!T->filter || T->layout.filter_bits <= 0) continue;
            S.op = OP_DIRECT_BITMAP;
            S.tab = T->filter;
            S.tab_bytes = (uint32_t)std::min<size_t>((size_t)(T->layout.filter_bits / 8), 0xFFFFFFF0u);
            via_bitmap[s] = 1;
        }
    }
    // 32-bit fast path of the accumulators: int32 column, multipliers and payload ranges within int32
    for (int s2 = 0; s2 < ns; ++s2) {
        DStage &S = P.st[s2];
        bool ok = !S.is64 || (S.acc & 0x7u) == 0; // (a payload's contribution does not depend on the key's width)
        for (int i = 0; i < 9; ++i) {
            ok = ok && S.mult[i] >= INT32_MIN && S.mult[i] <= INT32_MAX;
            S.mult32[i] = (int32_t)S.mult[i];
        }
        if (S.kind == ST_PROBE) {
            const int64_t hi0 = S.pmin0 + (int64_t)std::min<uint64_t>(S.pmask0, (uint64_t)INT32_MAX);
            ok = ok && S.code_bits <= 32 && S.pmin0 >= INT32_MIN && hi0 <= INT32_MAX && S.pmask0 <= 0x7FFFFFFFull;
            if (S.acc & 0x1C0u) {
                const int bits1 = (int)S.code_bits - (int)S.pbits0;
                ok = ok && bits1 < 31 && S.pmin1 >= INT32_MIN && S.pmin1 + ((int64_t)1 << std::max(bits1, 0)) <= INT32_MAX;
            }
        }
        S.acc32 = ok ? 1 : 0;
        S.simple = 0;
        if (ok && S.op == OP_LOAD && (S.acc == 1u || S.acc == 2u || S.acc == 4u))
            S.simple = (uint8_t)(1 + (S.acc == 1u ? 0 : S.acc == 2u ? 1 : 2));
    }
    P.nstages = ns;
    P.eager = opts.eager_loads ? 1 : 0;
    P.count32 = n < ((int64_t)1 << 32) ? 1 : 0;
    // Load schedule of the final level (used by kernels compiled for the query): a column is requested
    // once the last stage before it that is expected to drop rows has produced its mask, and at most
    // three columns ahead of the stage being processed.
    // Without queues a thread keeps its four consecutive rows and loads them with one 128-bit load, which is
    // skipped only when all four are dead: waiting for a mask pays only behind a stage that keeps less than
    // about one row in six; everything else is requested up front, four columns deep.
    {
        const int first = ndense, depth = P.nq ? 3 : 4;
        const double drop_below = P.nq ? 0.9 : 0.16;
        int last_barrier = first - 1;
        for (int t = first; t < ns; ++t) {
            P.st[t].issue_after = (int8_t)std::max(std::max(last_barrier, t - depth), first - 1);
            const bool drops = t < nfilter && specs[order[t]].sel < drop_below;
            if (drops) last_barrier = t;
        }
    }

    // A hashed result whose key is taken modulo M can only hold keys in (-M, M): when 2M - 1 cells fit the
    // workspace arrays the group table is indexed directly by key + M - 1 (no key array, no hashing, no claim:
    // two atomics per row instead of a look-up and two atomics; every dense aggregation path applies) and the
    // compaction recovers the keys from the cell numbers (config 4, G = 10^6 at 10 %: 3.2 -> 1.6 ms).
    // The same holds for a key without a modulo whose every term is a gathered payload: the tables know the
    // range of each payload among the rows they hold, so the key's range is known before the run (the
    // paper's city x city and city x brand keys, Section 3.3, are of this kind).  Whenever the range fits, the
    // indexed table is chosen: its clear and its compaction touch no more cells than the hash table's (whose
    // size follows the capacity, not the survivors), and a row costs less.
    const uint64_t gslots_all = spec->mode == SJQ_HASHED ? hashed_slots(spec->capacity) : 0;
    bool key_bounded = spec->mode == SJQ_HASHED && key != nullptr;
    __int128 key_lo = key ? key->offset : 0, key_hi = key_lo;
    for (int t = 0; key_bounded && t < key->nterms; ++t) {
        const sjq_term &T = key->t[t];
        if (T.src != SJQ_SRC_PAYLOAD) {
            key_bounded = false;
            break;
        }
        const sjq_dim_layout &L = joins[T.a].table->layout;
        const __int128 a = (__int128)T.mult * L.pay_min[T.b], b = (__int128)T.mult * L.pay_max[T.b];
        key_lo += a < b ? a : b;
        key_hi += a < b ? b : a;
    }
    if (key && key->modulo > 0) {
        // C remainder: the sign follows the dividend, the magnitude stays below the modulus
        const __int128 m1 = (__int128)key->modulo - 1;
        const bool nonneg = key_bounded && key_lo >= 0, nonpos = key_bounded && key_hi <= 0;
        key_lo = nonneg ? 0 : -m1;
        key_hi = nonpos ? 0 : m1;
        key_bounded = spec->mode == SJQ_HASHED;
    }
    const __int128 key_cells = key_hi - key_lo + 1;
    const bool direct_groups = key_bounded && !opts.group_hash_always && key_cells >= 1 &&
                               key_cells <= (__int128)gslots_all + 1 && key_lo > INT64_MIN && key_hi < INT64_MAX;
    const int64_t table_groups = direct_groups ? (int64_t)key_cells : spec->num_groups;
    if (direct_groups) {
        P.post_offset = (int64_t)-key_lo;
        P.want_count = 1; // the counts tell which cells hold a group
    }
    // ------------------------------------------------------------ aggregation path
    int aggp;
    size_t group_bytes = 0;
    const int approx_grid = dev.sm_count * 2;
    if (spec->mode == SJQ_SCALAR) {
        aggp = AGG_SCALAR;
    } else if (spec->mode == SJQ_HASHED && !direct_groups) {
        aggp = AGG_HASH;
    } else if (spec->mode == SJQ_DENSE && spec->num_groups == 1) {
        aggp = AGG_SCALAR; // a single group: register accumulation, key only range-checked
        P.has_key = 1;
    } else {
        const size_t gb = (size_t)table_groups * 8 * (P.want_count ? 2 : 1);
        const bool fits = gb <= (size_t)64 << 10;
        // Every block adds its touched groups to the global table once at its end, so a table per block pays as soon
        // as the rows that would be added one by one approach the cells of all blocks.  Measured over 1 M to 200 M
        // rows, 2 to 4096 groups, skewed and uniform: from 0.35 rows per cell on it is never slower and soon several
        // times faster, since the global cells serialise (0.34: 18.3 against 18.3 us; 1.1: 20.6 against 12.3; 5: 240
        // against 144; 100: 3,600 against 51); at 0.1 to 0.2 the two are within 5 %, below that up to 9 us slower.
        const double blocks = std::min((double)approx_grid, std::max(1.0, (double)plan_rows / (SJQ_LB_THREADS * 4 * P.slots)));
        const bool contended = survivors >= 0.35 * blocks * (double)table_groups;
        if (opts.unfused) {
            aggp = AGG_GLOBAL;
        } else if (opts.agg_path == 1) {
            if (!fits) return SJQ_ERR_UNSUPPORTED;
            aggp = AGG_SMEM;
        } else if (opts.agg_path == 2) {
            aggp = AGG_GLOBAL;
        } else {
            aggp = (fits && contended) ? AGG_SMEM : AGG_GLOBAL;
        }
        if (aggp == AGG_SMEM) group_bytes = gb;
    }
    P.num_groups = spec->mode == SJQ_DENSE ? spec->num_groups : direct_groups ? table_groups : 0;
    // Adding the values of equal keys inside the warp before the atomics is an option, never the default: per-lane
    // shared-memory atomics on a few counters were faster at every group count measured (selectivity sweep at
    // 100 %: 2 groups 4.1 vs 4.4 ms, 4 groups 3.3 vs 5.2, 16 groups 2.7 vs 15, 1000 groups 2.9 vs 34).
    if (opts.warp_agg < 0 || opts.warp_agg > 2) return SJQ_ERR_INVALID_ARG;
    P.warp_agg = (aggp == AGG_SMEM || aggp == AGG_GLOBAL) && !opts.unfused && opts.warp_agg == 1;

    // ------------------------------------------------------------ result buffers
    int64_t *gkeys = nullptr, *cells = nullptr;
    uint64_t gslots = 0;
    if (spec->mode == SJQ_HASHED) {
        size_t need = 0;
        sjq_run_workspace_bytes(spec, &need);
        if (out->workspace_bytes < need) return SJQ_ERR_BUFFER_SMALL;
        gslots = hashed_slots(spec->capacity);
        const size_t arr = align_up((size_t)(gslots + 1) * 8, 256);
        gkeys = reinterpret_cast<int64_t *>(static_cast<char *>(out->workspace));
        // the second and third array together hold the cells: {sum, count} side by side, so that both adds of a row
        // meet one 32-byte sector (add_pairs)
        cells = reinterpret_cast<int64_t *>(static_cast<char *>(out->workspace) + arr);
        P.gmask = gslots - 1;
        P.gkeys = direct_groups ? nullptr : gkeys;
        P.sums = cells;
        P.counts = cells + 1;
        P.cell_shift = 1;
        // Two lanes share a row's adds (cell numbers travel between them as 32-bit words) once at least one row in
        // fifty is expected to survive.  Below that the adds do not bound anything and the exchange only lengthens the
        // kernel: city x brand, one row in eleven thousand, 0.77 ms without and 0.85 with it; the sweep into a million
        // groups with every row surviving 8.56 without and 5.69 with it.
        P.pairs = gslots < 0xFFFFFFFFull && !P.warp_agg && reach[nfilter] >= 0.02;
    } else {
        P.sums = out->sums;
        P.counts = agg->want_count ? out->counts : nullptr;
    }

    // ------------------------------------------------------------ hot-key table
    // The first open-addressing join that filters through its presence bitmap gets a table of its heaviest
    // foreign keys in shared memory (built by three small kernels right before the fused pass), consulted by the
    // bitmap stage and by the exact probe.  Whether the keys are skewed at all is decided on the device (an empty
    // table switches the look-ups off).  Measured on the Zipf-skewed 64-bit-key workload (300 M rows, 2 009 keys
    // held, covering 47 % of the sample): fused kernel 1.61 -> 1.53 ms, whole call 1.65 -> 1.61 ms (the three
    // kernels cost about 40 us), so by default only a kernel compiled for the query on at least 2^26 rows uses it;
    // the interpreted kernel loses with it (3.5 -> 4.9 ms: the look-up does not fit its register budget).
    int hot_stage = -1;
    if (opts.hot_keys != 2 && opts.hot_scratch && opts.hot_scratch_bytes >= SJQ_HOT_SCRATCH_BYTES && !opts.unfused &&
        n > 0 && (opts.hot_keys == 1 || (opts.specialise && n >= ((int64_t)1 << 26)))) {
        for (int s2 = 0; s2 < ns && hot_stage < 0; ++s2)
            if (P.st[s2].op == OP_HASHBITS && P.st[s2].code_bits <= 32) hot_stage = s2;
    }
    size_t hot_bytes = hot_stage >= 0 ? align_up((size_t)(kHotSlots + 1) * 16, 16) : 0;

    // ------------------------------------------------------------ shared memory layout
    // [stage descriptors][staged tables][hot-key table][group table][per-warp survivor queues]
    int block = opts.block_threads ? opts.block_threads : SJQ_LB_THREADS;
    // A compiled kernel without queues whose rows all meet in a shared group table runs as two blocks of 640
    // threads per SM: two copies of the table instead of three and 40 warps instead of 36 (selectivity sweep at
    // 100 %, a thousand groups: 2.73 -> 2.52 ms; 64 groups 2.57 -> 2.39; 4000 groups 3.25 -> 2.56).
    // With register accumulators two blocks of 768 threads (48 warps at 42 registers) help while some rows still
    // drop (the sweep at 50 %, one group: 1.48 -> 1.41 ms) and cost a little when none does (100 %: 2.18 -> 2.22).
    const bool two_wide_blocks = opts.specialise && !opts.unfused && !opts.block_threads && !opts.ctas_per_sm &&
                                 P.nq == 0 && (aggp == AGG_SMEM || (aggp == AGG_SCALAR && reach[nfilter] < 0.8));
    if (two_wide_blocks) block = few_rows && aggp != AGG_SMEM ? 256 : aggp == AGG_SMEM ? 640 : 768;
    const size_t smem_cap = (size_t)dev.max_smem_optin - 1024; // static reduce scratch + slack
    const size_t stage_bytes = align_up((size_t)ns * sizeof(DStage), 16);
    if (hot_bytes && stage_bytes + hot_bytes + group_bytes +
                             (P.nq ? (size_t)(block / 32) * (size_t)(queue0_cap_for(P.slots) + (P.nq - 1) * queue_cap_for(P.rows)) * 4 : 0) >
                         smem_cap) {
        hot_stage = -1; // no room beside the group table and the queues
        hot_bytes = 0;
    }
    auto queue_bytes = [&](int threads) -> size_t {
        const size_t per_warp = (size_t)(queue0_cap_for(P.slots) + (P.nq - 1) * queue_cap_for(P.rows)) * 4;
        return P.nq ? (size_t)(threads / 32) * per_warp : 0;
    };
    // Direct tables (and presence bitmaps) worth a copy in shared memory, most probes per staged byte first.
    auto stage_tables = [&](int threads, size_t *tables_out) -> bool {
        for (int s2 = 0; s2 < ns; ++s2) P.st[s2].in_smem = 0, P.st[s2].smem_off = 0;
        const size_t fixed = stage_bytes + hot_bytes + group_bytes + queue_bytes(threads);
        if (fixed > smem_cap) return false;
        const size_t table_budget = smem_cap - fixed;
        size_t tables = 0;
        if (opts.smem_tables != 1 && !opts.unfused) {
            Order cand;
            for (int s = 0; s < nfilter; ++s)
                if (is_direct_op(P.st[s].op)) cand.push_back(s);
            std::stable_sort(cand.begin(), cand.end(), [&](int a, int b) {
                return reach[a] / (double)P.st[a].tab_bytes > reach[b] / (double)P.st[b].tab_bytes;
            });
            for (int s : cand) {
                DStage &S = P.st[s];
                const size_t tb = align_up(S.tab_bytes, 16);
                if (tables + tb > table_budget) continue;
                // larger tables are left to L1/L2: shared memory taken here is L1 capacity lost to every other table
                if (opts.smem_tables == 0 && tb > kStageBytes) continue;
                if (opts.smem_tables >= 1024 && tb > (size_t)opts.smem_tables) continue; // experiment: size limit in bytes
                // worth it only if a block probes the table more often than it costs to copy
                const double probes_per_cta = (double)plan_rows * reach[s] / approx_grid;
                if (probes_per_cta * 4.0 < (double)tb) continue;
                S.in_smem = 1;
                S.smem_off = (uint32_t)(stage_bytes + tables);
                tables += tb;
                if (s < ndense && gather_of_stage[s] >= 0 && !via_bitmap[s]) { // the sparse copy reads the same staged table
                    P.st[gather_of_stage[s]].in_smem = 1;
                    P.st[gather_of_stage[s]].smem_off = S.smem_off;
                }
            }
        }
        *tables_out = tables;
        return true;
    };
    size_t tables = 0;
    if (!stage_tables(block, &tables)) return SJQ_ERR_UNSUPPORTED;
    // Two blocks per SM each carry their own copies of the staged tables and the group table, and their
    // queues.  A kernel compiled for the query can run as one block of 1024 threads per SM instead: one
    // copy, 32 warps instead of 24.  Measured better whenever the copies are sizeable or shared memory
    // would crowd out the L1 (config 3: 1.43 -> 1.32 ms, config 5: 2.8 -> 1.8 ms), given enough tiles per
    // block to even out the tail (four joins: 140 -> 135 us at 60 M rows, 49 tiles a block; 23.3 -> 23.0 at 6 M; two
    // joins with sixteen rows per thread: 84.8 -> 84.9 at 60 M, 25 tiles, 14.5 -> 15.8 at 6 M, 2 tiles).
    // Failing that, a kernel whose shared memory is moderate (more than three 384-thread blocks
    // could share, at most 100 KB as a 640-thread block) runs as two 640-thread blocks: 40 warps instead of 24 and the
    // L1 keeps half of the SM's memory (two-join workload 0.101 -> 0.094 ms with eight rows per thread).  With sixteen
    // rows per thread its queues leave the L1 too little once survivors gather at random (the sweep, 200 M rows, as two
    // blocks of 640 or of 384: 1 % 201 and 210 us, 3 % 294 and 290, 10 % 462 and 406).
    bool single_block = false, two_wide_queue_blocks = false;
    if (opts.specialise && !opts.block_threads && !opts.ctas_per_sm && P.nq && !opts.unfused) {
        const size_t copies = tables + hot_bytes + group_bytes, as384 = stage_bytes + copies + queue_bytes(block);
        const int64_t tiles_per_block = plan_rows / ((int64_t)1024 * 4 * P.slots) / dev.sm_count;
        size_t other = 0;
        if ((copies >= ((size_t)16 << 10) || as384 > ((size_t)80 << 10)) && tiles_per_block >= 16 && stage_tables(1024, &other)) {
            block = 1024;
            single_block = true;
            tables = other;
        } else if (as384 > ((size_t)48 << 10) && (P.slots == 2 || reach[nd0] < 0.03) && stage_tables(640, &other) &&
                   stage_bytes + other + hot_bytes + group_bytes + queue_bytes(640) <= ((size_t)100 << 10)) {
            block = 640;
            two_wide_queue_blocks = true;
            tables = other;
        } else if (!stage_tables(block, &tables)) {
            return SJQ_ERR_UNSUPPORTED;
        }
    }
    // Nearly every row probes a map too large for the 32 KB above and adds to a global table: the pass is bound by the
    // L2's tags and the requests of the SMs, of which a row costs two to three.  The first part of the map, or all of it,
    // is then staged in shared memory, and a probe asks the L2 only beyond it.  The part is what fits beside the other
    // staged tables in a carve-out of 196 KB, which leaves the L1 60 KB: one step more and it has 28 (a first join with
    // a map of 10 or 30 KB, then one of 750 KB, 100 M rows: 853 and 858 us without staging, 962 and 961 beyond the step,
    // 797 and 809 so).  With a shared group table or register sums the L1's own rate is the bound and the second,
    // divergent load costs what it saves.  No gain for 3 M rows.
    // A million groups as a list, every row left, one block of 768 threads, without and with, 100 M rows: maps of 35 KB
    // 703 and 681, 150 KB 705 and 688, 250 KB 772 and 680, 500 KB 956 and 895, 750 KB 880 and 841; 17 M rows: 75 KB 143
    // and 139, 250 KB 157 and 141, 750 KB 176 and 168.  Lists take no part of a map
    //   of less than 1 1/8 parts, most of which the L1 holds (200 KB 666 and 690, 220 KB 745 and 670), with codes of a
    //   byte, whose divergent loads cost more, of less than 1 3/4 (260 KB 839 and 854, 340 KB 903 and 873);
    //   of more than six parts, where too few probes are answered (17 M rows: 880 KB 179 and 174, 1.1 MB 179 and 179,
    //   1.2 MB 172 and 181, 1.5 MB 171 and 184), unless the group table is moderate (200 thousand groups, 1.2 MB, 166
    //   and 159);
    //   beside a group table of more than 64 MB, whose own misses bound them (4 M groups, 750 KB, 1066 and 1076; 2 M
    //   groups 959 and 855).
    // Lists of few groups and dense results gain from all of these or lose little (20 thousand groups: 200 KB 931 and
    // 928, at 17 M rows 144 and 147; 900 KB 1055 and 961; dense, 50 thousand, 1.5 MB 1482 and 1446).
    int part = -1, probes = 0;
    const size_t beside_part = align_up(stage_bytes + tables, 16);
    const size_t part_bytes = beside_part < kPartCarveOut ? std::min(kPartBytes, (kPartCarveOut - beside_part) & ~(size_t)15) : 0;
    if (mostly_survive && !opts.unfused && !opts.block_threads && !opts.ctas_per_sm && opts.smem_tables == 0 && P.nq == 0 &&
        aggp == AGG_GLOBAL && hot_stage < 0 && plan_rows >= kPartRows && part_bytes > kStageBytes) {
        for (int s = 0; s < nfilter; ++s) {
            const DStage &S = P.st[s];
            const bool bytes = S.op == OP_DIRECT_U8;
            const bool narrow_codes = bytes || S.op == OP_DIRECT_BITMAP || S.op == OP_DIRECT_U2 || S.op == OP_DIRECT_U4;
            const bool whole = align_up(S.tab_bytes, 16) <= part_bytes;
            const bool some = !P.pairs || table_groups <= (int64_t)1 << 17 ||
                              (S.tab_bytes >= kPartBytes / 8 * (bytes ? 14 : 9) && table_groups <= (int64_t)1 << 22 &&
                               (S.tab_bytes <= 6 * part_bytes || table_groups <= (int64_t)1 << 19));
            probes += S.kind == ST_PROBE;
            if (narrow_codes && !S.in_smem && (whole || some) && (part < 0 || S.tab_bytes < P.st[part].tab_bytes)) part = s;
        }
    }
    if (part >= 0) {
        DStage &S = P.st[part];
        // Fewer, longer chains where every row goes all the way, half of the probes or more go beyond the copy and no
        // other probe fills the time.  A million groups, 100 M rows, 768 and 512 threads: 2-bit codes of 350 KB 750 and
        // 761, 400 KB 793 and 785, 500 KB 895 and 822, 625 KB 842 and 818, 750 KB 841 and 831, 900 KB 830 and 843; 4-bit
        // codes of 500 KB 894 and 822, 700 KB 839 and 827; bitmaps of 500 KB 893 and 836, 750 KB 817 and 828; 300 M rows,
        // 400 KB 2467 and 2268, 600 KB 2565 and 2391.  Not so with nine rows in ten left (300 M rows, 750 KB, 2234 and
        // 2305; 19 in 20, 100 M rows, 847 and 814), fewer rows (17 M, 400 KB, 162 and 166), codes of a byte (780 KB, 816
        // and 934) or behind a first join (750 KB, 796 and 846).
        const bool long_chains = S.op != OP_DIRECT_U8 && S.tab_bytes > 2 * kPartBytes && S.tab_bytes <= 4 * kPartBytes &&
                                 probes == 1 && reach[nfilter] >= 0.95 && plan_rows >= kLongChainRows;
        block = long_chains ? 512 : 768;
        S.in_smem = align_up(S.tab_bytes, 16) <= part_bytes ? kTabShared : kTabPart;
        S.smem_off = (uint32_t)beside_part;
        if (S.in_smem == kTabPart) S.tab_bytes = (uint32_t)part_bytes;
        tables = beside_part - stage_bytes + align_up(S.tab_bytes, 16);
        single_block = true;
    }
    P.smem_stages = 0;
    P.smem_groups = (uint32_t)(stage_bytes + tables + hot_bytes);
    P.smem_queue = (uint32_t)(stage_bytes + tables + hot_bytes + group_bytes);
    size_t smem = stage_bytes + tables + hot_bytes + group_bytes + queue_bytes(block);
    if (hot_stage >= 0) {
        // the bitmap stage copies the table into shared memory; every stage of the same join reads that copy
        const void *bucket_array = joins[specs[order[hot_stage]].index].table->slots;
        for (int s2 = 0; s2 < ns; ++s2) {
            DStage &S = P.st[s2];
            const bool same_join = s2 == hot_stage || ((S.op == OP_HASH32 || S.op == OP_HASH64) && S.tab == bucket_array);
            if (!same_join) continue;
            S.hot = s2 == hot_stage ? 1 : 2;
            S.hot_off = (uint32_t)(stage_bytes + tables);
        }
    }

    // ------------------------------------------------------------ bulk-asynchronous staging of the first column
    // A kernel compiled for a query with survivor queues can have its first column copied into shared memory by
    // the copy engine, one tile (block size x 4 x slots values) per copy, three in flight per block.  Only when
    // asked for: measured on the selectivity sweep (600 M rows) the staged kernel is slower than 128-bit loads
    // with L2 prefetch at every point (0.01 %: 0.42 vs 0.37 ms; 1 %: 0.64 vs 0.53; 10 %, 1000 groups: 1.25 vs 1.21)
    // and much slower where its buffers crowd the shared memory (city x city: 1.09 vs 0.73 ms), although a bare
    // scan kernel built on the same copies moves 7.3 TB/s against 6.7 TB/s for loads: the warps of the fused
    // kernel consume a tile at their own pace, so the refill of a buffer waits for the slowest of them.
    const size_t smem_without_bulk = smem;
    if (opts.l0_bulk < 0 || opts.l0_bulk > 3) return SJQ_ERR_INVALID_ARG;
    if (opts.specialise && !opts.unfused && P.nq > 0 && n > 0 && (opts.l0_bulk == 1 || opts.l0_bulk == 3)) {
        const size_t tile_bytes = (size_t)block * 4 * P.slots * (P.st[0].is64 ? 8 : 4);
        const size_t at = align_up(smem, 128);
        const size_t total = at + 3 * tile_bytes + 3 * 8 + 3 * 4 + 4;
        if (total <= smem_cap) {
            P.l0_bulk = opts.l0_bulk == 3 ? 2 : 1; // 2: the kernel waits for copies nobody issues (failure-path test)
            P.smem_l0 = (uint32_t)at;
            smem = total;
        }
    }

    P.may_clear = few_rows && !opts.unfused && spec->mode != SJQ_HASHED && (aggp == AGG_SCALAR || aggp == AGG_SMEM);
    const bool self_clear = P.may_clear && opts.sync && !opts.accumulate && n > 0;

    // ------------------------------------------------------------ form of the ahead-of-time kernel
    bool has_hash = false; // kernels without the hash probe are leaner; pick by what the stages need
    bool narrow = ns <= kFewStages;
    for (int s2 = 0; s2 < ns; ++s2) {
        const DStage &S = P.st[s2];
        has_hash |= S.op == OP_HASH32 || S.op == OP_HASH64 || S.op == OP_HASHBITS;
        const bool hashed_key = S.is64 && (S.acc & 0x7u) == 0 &&
                                (S.op == OP_LOAD || S.op == OP_HASHBITS || (S.op == OP_HASH64 && S.code_bits <= 32));
        const bool plain = !S.is64 && S.op != OP_DIRECT_U64 && S.op != OP_HASH32 && S.op != OP_HASHBITS;
        narrow = narrow && (plain || hashed_key) && (S.acc32 || !S.acc);
    }
    const int form = (has_hash ? kFormHash : 0) | (P.nq == 0 ? kFormDirect : 0) | (narrow ? kFormNarrow : 0);

    // ------------------------------------------------------------ launch shape
    int per_sm = 0;
    const bool jit = opts.specialise != 0 && !opts.unfused;
    // register budget a specialised kernel is compiled for
    // (three blocks of 384 threads when their shared memory leaves the L1 alone: 56 registers are enough for the
    // short pipelines that have so little state, and 36 warps hide more latency than 24)
    const int lb_blocks = single_block ? 1
                          : (two_wide_blocks || two_wide_queue_blocks) ? 2
                          : opts.ctas_per_sm > 0 ? opts.ctas_per_sm
                          : block > 512 ? 1
                          : (block <= 384 && smem_without_bulk <= ((size_t)48 << 10)) ? 3
                                                                        : 2;
    const void *compiled = nullptr;
    st = jit ? jit_prepare(P, aggp, mul, has_hash, block, lb_blocks, smem, &per_sm, &compiled)
             : fused_occupancy(aggp, mul, form, ns, block, smem, &per_sm);
    if (st != SJQ_OK) return st;
    if (per_sm < 1) return SJQ_ERR_UNSUPPORTED;
    if (opts.ctas_per_sm > 0) per_sm = std::min(per_sm, opts.ctas_per_sm);
    const int64_t tile_rows = (int64_t)block * (P.nq ? 4 * P.slots : kDirectRows);
    const int64_t ntiles = (n + tile_rows - 1) / tile_rows;
    if (ntiles >= ((int64_t)1 << 31)) return SJQ_ERR_UNSUPPORTED;
    int grid = (int)std::min<int64_t>((int64_t)dev.sm_count * per_sm, std::max<int64_t>(ntiles, 1));

    // ------------------------------------------------------------ launches
    int launches = 0;
    if (self_clear) {
        P.sync = static_cast<uint64_t *>(opts.sync);
        P.epoch = next_epoch();
        P.clear_late_ms = std::min(std::max(opts.sync_late_ms, 0), 5000);
        P.clear_counts = out->counts;
        P.clear_cells = spec->mode == SJQ_SCALAR ? 1 : spec->num_groups;
        P.clear_blocks = (int32_t)std::min<int64_t>(std::min(grid, kClearBlocks), 1 + P.clear_cells / (2 * block));
    } else if (!opts.accumulate) {
        const int64_t words = spec->mode == SJQ_SCALAR ? 1
                              : spec->mode == SJQ_DENSE ? spec->num_groups
                              : direct_groups           ? 2 * table_groups
                                                        : 2 * ((int64_t)gslots + 1);
        // The pass starts beside the clear, except where its blocks are fewer than the chip holds and the clear's many:
        // then they would be spread unevenly over the SMs (sums and counts of 400,000 groups, 2 M rows: 34.3 us when
        // started at once, 30.5 when the stores are out, 32.5 one kernel after the other; a pass that fills the chip
        // behind the clear of a million groups, 600 M rows: 5,673 and 5,681).
        const int at_once = grid == dev.sm_count * per_sm ? INT32_MAX : dev.sm_count;
        st = clear_launch(P.sums, spec->mode == SJQ_HASHED ? nullptr : out->counts, words, gkeys,
                          (spec->mode == SJQ_HASHED && !direct_groups) ? (int64_t)gslots + 1 : 0, out->n_groups,
                          out->status, at_once, dev.sm_count, stream);
        if (st != SJQ_OK) return st;
        ++launches;
    } else if (spec->mode == SJQ_HASHED) {
        if (cudaMemsetAsync(out->n_groups, 0, sizeof(int64_t), stream) != cudaSuccess) return SJQ_ERR_CUDA;
    }
    if (hot_stage >= 0) {
        const StageSpec &sp = specs[order[hot_stage]];
        const void *hot_table = nullptr;
        st = hot_launch(fact[sp.col].data, fact[sp.col].dtype == SJQ_I64, n, joins[sp.index].table, opts.hot_scratch,
                        stream, &hot_table, &launches);
        if (st != SJQ_OK) return st;
        for (int s2 = 0; s2 < ns; ++s2)
            if (P.st[s2].hot) P.st[s2].hot_tab = hot_table;
    }
    if ((opts.event_before != nullptr) != (opts.event_after != nullptr)) return SJQ_ERR_INVALID_ARG;
    if (opts.event_before && cudaEventRecord((cudaEvent_t)opts.event_before, stream) != cudaSuccess)
        return SJQ_ERR_CUDA;
    if (n > 0 && opts.unfused) {
        if (!aligned16(opts.unfused_scratch)) return SJQ_ERR_ALIGN;
        st = unfused_launch(P, nfilter, aggp, mul, has_hash, opts.unfused_scratch, opts.unfused_scratch_bytes,
                            dev.sm_count, stream, &launches);
        if (st != SJQ_OK) return st;
    } else if (n > 0) {
        // Directly behind the clear the kernel is launched while that one still runs (programmatic dependent launch):
        // it stages its tables, which were complete before the clear began, and waits for the clear before it touches
        // a result (two-join query, 60 M rows: 94 -> 92 us; filter and sum, 6 M rows: 20.5 -> 18.5 us back to back).
        const bool behind = !opts.accumulate && hot_stage < 0 && !opts.event_before;
        st = jit ? jit_launch(compiled, P, grid, block, smem, behind, stream)
                 : fused_launch(aggp, mul, form, grid, block, smem, behind, P, stream);
        if (st != SJQ_OK) return st;
        ++launches;
    }
    if (opts.event_after && cudaEventRecord((cudaEvent_t)opts.event_after, stream) != cudaSuccess)
        return SJQ_ERR_CUDA;
    if (spec->mode == SJQ_HASHED) {
        // (an indexed table has no use for the key array: it holds the block counts of the ordered list)
        // Launched behind the pass, the listing takes 1 to 3 us less (a list of 20,000 groups, 1 % left: 20 M rows
        // 36.4 -> 33.5 us, 2 M 18.5 -> 15.3).  Its blocks wait in the SMs meanwhile: one per SM leaves room for other
        // streams' kernels beside a long pass.
        const bool follows = n > 0 && !opts.unfused && !opts.event_after;
        const int beside = !follows ? 0 : n <= (int64_t)1 << 20 ? INT32_MAX : dev.sm_count;
        st = compact_launch(gkeys, cells, direct_groups ? table_groups : (int64_t)gslots, direct_groups, P.post_offset,
                            direct_groups && !opts.unfused ? reinterpret_cast<unsigned int *>(gkeys) : nullptr,
                            out->keys, out->sums, out->counts, spec->capacity, out->n_groups, out->status,
                            dev.sm_count, beside, stream, &launches);
        if (st != SJQ_OK) return st;
    }
    if (info) {
        std::memset(info, 0, sizeof(*info));
        info->nstages = ns;
        const int shown = std::min<int>(ns, (int)(sizeof(info->order) / sizeof(info->order[0])));
        info->nstages = shown;
        for (int s = 0; s < shown; ++s) {
            info->order[s] = stage_label[s];
            info->stage_in_smem[s] = P.st[s].in_smem;
        }
        info->first_sparse_stage = P.nq ? P.nd0 : 0;
        info->reserved_levels = P.nq;
        info->agg_path = aggp;
        info->grid = grid;
        info->block = block;
        info->smem_bytes = (int32_t)smem;
        info->kernel_launches = launches;
    }
    return SJQ_OK;
}


extern "C" sjq_status sjq_run(const sjq_col *fact, int nfact, const sjq_pred *preds, int npreds,
                              const sjq_join *joins, int njoins, const sjq_key_expr *key, const sjq_agg_expr *agg,
                              const sjq_result_spec *spec, const sjq_result *out, const sjq_run_opts *opts,
                              void *stream, sjq_run_info *info)
{
    return run_planned(fact, nfact, preds, npreds, joins, njoins, key, agg, spec, out, opts, RunContext{}, stream, info);
}

// ---------------------------------------------------------------------------
// Merge of hashed results (the exchange step of a row-sharded run).
extern "C" sjq_status sjq_merge_groups(const int64_t *keys, const int64_t *sums, const int64_t *counts, int64_t n,
                                       int64_t capacity, const sjq_result *out, void *stream_)
{
    if (n < 0 || capacity <= 0 || !out || !out->keys || !out->sums || !out->counts || !out->n_groups ||
        !out->status || !out->workspace || (n > 0 && (!keys || !sums || !counts)))
        return SJQ_ERR_INVALID_ARG;
    if (!aligned16(out->sums) || !aligned16(out->counts) || !aligned16(out->keys) || !aligned16(out->workspace) ||
        (reinterpret_cast<uintptr_t>(keys) & 7u) || (reinterpret_cast<uintptr_t>(sums) & 7u) ||
        (reinterpret_cast<uintptr_t>(counts) & 7u) || (reinterpret_cast<uintptr_t>(out->status) & 3u) ||
        (reinterpret_cast<uintptr_t>(out->n_groups) & 7u))
        return SJQ_ERR_ALIGN;
    sjq_result_spec spec{SJQ_HASHED, 0, capacity};
    size_t need = 0;
    sjq_run_workspace_bytes(&spec, &need);
    if (out->workspace_bytes < need) return SJQ_ERR_BUFFER_SMALL;
    DeviceInfo dev;
    sjq_status st = device_info(&dev);
    if (st != SJQ_OK) return st;
    cudaStream_t stream = (cudaStream_t)stream_;
    const uint64_t gslots = hashed_slots(capacity);
    const size_t arr = align_up((size_t)(gslots + 1) * 8, 256);
    int64_t *gkeys = reinterpret_cast<int64_t *>(static_cast<char *>(out->workspace));
    int64_t *cells = reinterpret_cast<int64_t *>(static_cast<char *>(out->workspace) + arr);
    if ((st = clear_launch(cells, nullptr, 2 * ((int64_t)gslots + 1), gkeys, (int64_t)gslots + 1, out->n_groups, out->status,
                           INT32_MAX, dev.sm_count, stream)) != SJQ_OK)
        return st;
    if ((st = merge_launch(keys, sums, counts, n, gkeys, cells, gslots - 1, out->status, dev.sm_count,
                           stream)) != SJQ_OK)
        return st;
    int launches = 0;
    return compact_launch(gkeys, cells, (int64_t)gslots, false, 0, nullptr, out->keys, out->sums, out->counts, capacity,
                          out->n_groups, out->status, dev.sm_count, 0, stream, &launches);
}

// ---------------------------------------------------------------------------
// Host-buffer entry point: chunked, double-buffered copy + run.
namespace {

struct HostPipe {
    cudaStream_t s[2] = {nullptr, nullptr};
    cudaEvent_t start = nullptr, done[2] = {nullptr, nullptr};
    bool ok = false;
};

thread_local HostPipe g_pipes[64];

HostPipe *host_pipe()
{
    HostPipe *pipes = g_pipes;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    HostPipe &p = pipes[dev];
    if (!p.ok) {
        if (cudaStreamCreateWithFlags(&p.s[0], cudaStreamNonBlocking) != cudaSuccess ||
            cudaStreamCreateWithFlags(&p.s[1], cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&p.start, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&p.done[0], cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&p.done[1], cudaEventDisableTiming) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        p.ok = true;
    }
    return &p;
}

} // namespace

namespace {

enum { HOST_COPY = 0, HOST_IN_PLACE = 1, HOST_SKIP = 2 };

// What a column costs on the bus, in picoseconds per row of the table: copied whole at 53 GB/s, or, where at most
// kInPlaceReach of the rows reach it, the 32-byte sectors that hold one of them, read by the kernel at about half that
// (28 MB in 0.95 ms beside the copies).
constexpr double kInPlaceReach = 0.05;
double bus_ps(int width, double reach)
{
    const double copy = 18.9 * width;
    if (reach > kInPlaceReach) return copy;
    double dead = 1.0 - reach;
    for (int rows = 32 / width; rows > 1; rows >>= 1) dead *= dead;
    return std::min(copy, 1.9 * copy * (1.0 - dead));
}

// How each host-resident column reaches the kernel.  A column most rows still need is copied chunk by
// chunk; one that only a few per cent of the rows reach (lazy loading: it is read for survivors only) is
// read by the kernel straight from the page-locked host buffer, 32 bytes per touched sector, which moves
// far fewer bytes over the bus than the whole column (measured on the four-join workload, 600 M rows:
// revenue and supplycost 16 ms instead of 87 ms of copies; break-even beyond 5 % of the rows); a column the
// query never references is not transferred at all.  `need`: share of the rows each column is first read
// for (< 0: never).  Invalid queries get "copy everything" and are rejected later by sjq_run.
void host_transfer_plan(const sjq_col *fact_host, int nfact, const sjq_pred *preds, int npreds,
                        const sjq_join *joins, int njoins, const sjq_key_expr *key, const sjq_agg_expr *agg,
                        sjq_run_opts *opts_io, std::vector<int> *how_out, std::vector<const char *> *base_out,
                        std::vector<double> *need_out)
{
    sjq_run_opts &opts = *opts_io; // predicates measured here are written back as hints for the runs
    std::vector<int> &how = *how_out;
    std::vector<const char *> &direct_base = *base_out;
    how.assign(nfact, HOST_COPY);
    direct_base.assign(nfact, nullptr);
    need_out->assign(nfact, 1.0);
    const int64_t n = fact_host[0].n;
    bool ok = npreds >= 0 && npreds <= SJQ_MAX_PREDS && njoins >= 0 && njoins <= SJQ_MAX_JOINS &&
              (!npreds || preds) && (!njoins || joins) && n > 0 && agg;
    for (int p = 0; ok && p < npreds; ++p) ok = preds[p].col >= 0 && preds[p].col < nfact;
    for (int j = 0; ok && j < njoins; ++j)
        ok = joins[j].table && joins[j].table->magic == kTableMagic && joins[j].fk_col >= 0 && joins[j].fk_col < nfact;
    auto term_ok = [&](const sjq_term &t) { return t.src != SJQ_SRC_FACT || (t.a >= 0 && t.a < nfact); };
    if (ok && key) {
        ok = key->nterms >= 0 && key->nterms <= SJQ_MAX_KEY_TERMS;
        for (int t = 0; ok && t < key->nterms; ++t) ok = term_ok(key->t[t]);
    }
    ok = ok && term_ok(agg->x) && (agg->op == SJQ_AGG_COL || term_ok(agg->y));
    Specs specs;
    Order order;
    // The columns are in host memory here, so predicates without a measured pass fraction are measured on
    // the spot: a few thousand evenly spaced rows read by the host.  (A guess that is far too low would send
    // a column most rows need over the bus sector by sector.)
    sjq_run_opts &measured = opts;
    for (int p = 0; ok && p < npreds; ++p) {
        if (measured.pass_ppm[p] > 0) continue;
        const sjq_col &c = fact_host[preds[p].col];
        DPred d;
        if (!c.data || !canon_pred(preds[p], c.dtype, &d)) continue;
        const int64_t samples = std::min<int64_t>(n, 8192), stride = n / samples;
        int64_t pass = 0;
        for (int64_t i = 0; i < samples; ++i) {
            const int64_t r = i * stride;
            const int64_t v = c.dtype == SJQ_I64 ? static_cast<const int64_t *>(c.data)[r]
                                                 : (int64_t) static_cast<const int32_t *>(c.data)[r];
            bool in;
            if (d.nset) {
                in = false;
                for (int k = 0; k < d.nset; ++k) in |= v == d.set[k];
            } else {
                in = (v >= d.lo && v <= d.hi) != (bool)d.neg;
            }
            pass += in;
        }
        measured.pass_ppm[p] = ppm_of(pass, samples);
    }
    if (!ok || order_stages(fact_host, preds, npreds, joins, njoins, measured, &specs, &order) != SJQ_OK) return;
    std::vector<const char *> mapped(nfact, nullptr); // device address of a page-locked column
    for (int c = 0; c < nfact; ++c) {
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, fact_host[c].data) == cudaSuccess && attr.type == cudaMemoryTypeHost &&
            attr.devicePointer && aligned16(attr.devicePointer))
            mapped[c] = static_cast<const char *>(attr.devicePointer);
        else
            (void)cudaGetLastError(); // pageable memory: copied
    }
    const bool in_place_allowed = !opts.eager_loads && !opts.host_copy_all;
    // The bus is what a run from host memory waits for, so the filters are ordered by what their columns cost there: a
    // column is copied whole, or read in place where few rows reach it.  Four joins, 16 M rows: with the order of a
    // device-resident run three columns are copied (4,017 us), with this one two (3,373 us); 3 M rows 822 and 711, 700
    // thousand 244 and 218.  Below a million rows the saving is no more than that and the order stays the device's.
    bool by_bus = in_place_allowed && !opts.norder && n >= (int64_t)1 << 20;
    for (const StageSpec &sp : specs) by_bus = by_bus && sp.prefilter == 0 && mapped[sp.col];
    if (by_bus) {
        order = cheapest_order(specs, [](const StageSpec &sp, double reach) { return bus_ps(sp.width, reach); });
        opts.norder = order.size();
        for (int i = 0; i < order.size(); ++i)
            opts.order[i] = specs[order[i]].kind == ST_PRED ? specs[order[i]].index : npreds + specs[order[i]].index;
    }
    std::vector<double> &need = *need_out;
    need.assign(nfact, -1.0);
    double reach = 1.0;
    for (int i : order) {
        if (need[specs[i].col] < 0) need[specs[i].col] = reach;
        reach *= specs[i].sel;
    }
    auto use = [&](const sjq_term &t) {
        if (t.src == SJQ_SRC_FACT && need[t.a] < 0) need[t.a] = reach;
    };
    if (key && key->modulo != 1) // (modulo 1: the planner drops the key's terms)
        for (int t = 0; t < key->nterms; ++t) use(key->t[t]);
    use(agg->x);
    if (agg->op != SJQ_AGG_COL) use(agg->y);
    for (int c = 0; c < nfact; ++c) {
        if (need[c] < 0) {
            how[c] = HOST_SKIP;
        } else if (need[c] <= kInPlaceReach && in_place_allowed && mapped[c]) {
            how[c] = HOST_IN_PLACE;
            direct_base[c] = mapped[c];
        }
    }
}

} // namespace

extern "C" sjq_status sjq_host_transfer_plan(const sjq_col *fact_host, int nfact, const sjq_pred *preds, int npreds,
                                             const sjq_join *joins, int njoins, const sjq_key_expr *key,
                                             const sjq_agg_expr *agg, const sjq_run_opts *opts_, int32_t *how,
                                             double *share)
{
    if (!fact_host || nfact <= 0 || nfact > 64 || !agg || !how) return SJQ_ERR_INVALID_ARG;
    sjq_run_opts opts{};
    if (opts_) opts = *opts_;
    std::vector<int> h;
    std::vector<const char *> base;
    std::vector<double> need;
    host_transfer_plan(fact_host, nfact, preds, npreds, joins, njoins, key, agg, &opts, &h, &base, &need);
    for (int c = 0; c < nfact; ++c) {
        how[c] = h[c];
        if (share) share[c] = need[c] < 0 ? 0.0 : need[c];
    }
    return SJQ_OK;
}

extern "C" sjq_status sjq_run_host(const sjq_col *fact_host, int nfact, const sjq_pred *preds, int npreds,
                                   const sjq_join *joins, int njoins, const sjq_key_expr *key,
                                   const sjq_agg_expr *agg, const sjq_result_spec *spec, const sjq_result *out,
                                   const sjq_run_opts *opts_, void *staging_dev, size_t staging_bytes,
                                   int64_t chunk_rows, int64_t *host_sums, int64_t *host_counts, int64_t *host_keys,
                                   int64_t *host_n_groups, int32_t *host_status, void *stream_)
{
    if (!fact_host || nfact <= 0 || nfact > 64 || !staging_dev || chunk_rows <= 0 || (chunk_rows & 3) || !spec ||
        !out || !agg)
        return SJQ_ERR_INVALID_ARG;
    if (!aligned16(staging_dev)) return SJQ_ERR_ALIGN;
    const int64_t n = fact_host[0].n;
    if (n < 0) return SJQ_ERR_INVALID_ARG;
    size_t half = 0;
    std::vector<size_t> col_off(nfact);
    for (int c = 0; c < nfact; ++c) {
        if (fact_host[c].n != n || (fact_host[c].dtype != SJQ_I32 && fact_host[c].dtype != SJQ_I64) ||
            (n > 0 && !fact_host[c].data))
            return SJQ_ERR_INVALID_ARG;
        col_off[c] = half;
        half += align_up((size_t)chunk_rows * (fact_host[c].dtype == SJQ_I64 ? 8 : 4), 256);
    }
    if (staging_bytes < 2 * half) return SJQ_ERR_BUFFER_SMALL;
    HostPipe *hp = host_pipe();
    if (!hp) return SJQ_ERR_CUDA;
    cudaStream_t stream = (cudaStream_t)stream_;
    sjq_run_opts opts{};
    if (opts_) opts = *opts_;
    opts.event_before = opts.event_after = nullptr;

    std::vector<int> how;
    std::vector<const char *> direct_base;
    std::vector<double> need_share;
    host_transfer_plan(fact_host, nfact, preds, npreds, joins, njoins, key, agg, &opts, &how, &direct_base, &need_share);
    RunContext context;
    context.callers_order = opts_ && opts_->norder != 0;
    for (int c = 0; c < nfact; ++c) context.in_place |= how[c] == HOST_IN_PLACE;
    context.rows = std::min(n, chunk_rows);

    // internal streams start after whatever is already queued on the caller's stream
    if (cudaEventRecord(hp->start, stream) != cudaSuccess) return SJQ_ERR_CUDA;
    for (int b = 0; b < 2; ++b)
        if (cudaStreamWaitEvent(hp->s[b], hp->start, 0) != cudaSuccess) return SJQ_ERR_CUDA;

    const int64_t nchunks = n == 0 ? 1 : (n + chunk_rows - 1) / chunk_rows;
    std::vector<sjq_col> dev_cols(nfact);
    for (int64_t k = 0; k < nchunks; ++k) {
        const int b = (int)(k & 1);
        const int64_t r0 = k * chunk_rows;
        const int64_t rows = std::min<int64_t>(chunk_rows, n - r0);
        char *base = static_cast<char *>(staging_dev) + (size_t)b * half;
        // copies into this half follow run k-2 by stream order and overlap run k-1 on the other stream
        for (int c = 0; c < nfact; ++c) {
            const size_t w = fact_host[c].dtype == SJQ_I64 ? 8 : 4;
            dev_cols[c] = sjq_col{base + col_off[c], fact_host[c].dtype, rows};
            if (how[c] == HOST_SKIP) continue; // never dereferenced
            if (how[c] == HOST_IN_PLACE) {
                dev_cols[c].data = direct_base[c] + (size_t)r0 * w;
                continue;
            }
            if (rows > 0 &&
                cudaMemcpyAsync(base + col_off[c], static_cast<const char *>(fact_host[c].data) + (size_t)r0 * w,
                                (size_t)rows * w, cudaMemcpyHostToDevice, hp->s[b]) != cudaSuccess)
                return SJQ_ERR_CUDA;
        }
        // runs accumulate into the same result and must not overlap: run k waits for run k-1
        if (k > 0 && cudaStreamWaitEvent(hp->s[b], hp->done[b ^ 1], 0) != cudaSuccess) return SJQ_ERR_CUDA;
        opts.accumulate = (k > 0 || (opts_ && opts_->accumulate)) ? 1 : 0;
        opts.hot_keys = 2; // a chunk's foreign keys may still be in host memory: no sampling pass over them
        sjq_status st = run_planned(dev_cols.data(), nfact, preds, npreds, joins, njoins, key, agg, spec, out, &opts,
                                    context, hp->s[b], nullptr);
        if (st != SJQ_OK) return st;
        if (cudaEventRecord(hp->done[b], hp->s[b]) != cudaSuccess) return SJQ_ERR_CUDA;
    }
    const int last = (int)((nchunks - 1) & 1);
    if (cudaStreamWaitEvent(stream, hp->done[last], 0) != cudaSuccess) return SJQ_ERR_CUDA;
    if (nchunks > 1 && cudaStreamWaitEvent(stream, hp->done[last ^ 1], 0) != cudaSuccess) return SJQ_ERR_CUDA;
    const int64_t cells = spec->mode == SJQ_SCALAR ? 1 : spec->mode == SJQ_DENSE ? spec->num_groups : spec->capacity;
    bool ok = true;
    if (host_sums) ok = ok && cudaMemcpyAsync(host_sums, out->sums, (size_t)cells * 8, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
    if (host_counts && out->counts)
        ok = ok && cudaMemcpyAsync(host_counts, out->counts, (size_t)cells * 8, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
    if (host_keys && out->keys)
        ok = ok && cudaMemcpyAsync(host_keys, out->keys, (size_t)cells * 8, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
    if (host_n_groups && out->n_groups)
        ok = ok && cudaMemcpyAsync(host_n_groups, out->n_groups, 8, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
    if (host_status) ok = ok && cudaMemcpyAsync(host_status, out->status, 4, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
    return ok ? SJQ_OK : SJQ_ERR_CUDA;
}


namespace sjq {
int fused_cache_clear();
}

extern "C" int32_t sjq_release(void)
{
    int32_t released = 0;
    int current = 0;
    const bool have_device = cudaGetDevice(&current) == cudaSuccess;
    for (int d = 0; d < 64; ++d) {
        HostPipe &p = g_pipes[d];
        if (!p.ok) continue;
        if (have_device && cudaSetDevice(d) == cudaSuccess) {
            for (cudaStream_t &st : p.s)
                if (st && cudaStreamDestroy(st) == cudaSuccess) ++released;
            for (cudaEvent_t ev : {p.start, p.done[0], p.done[1]})
                if (ev && cudaEventDestroy(ev) == cudaSuccess) ++released;
        }
        p = HostPipe();
    }
    if (have_device) (void)cudaSetDevice(current);
    (void)cudaGetLastError();
    released += sjq::host_stats_release();
    released += sjq_jit_cache_clear();
    released += sjq::fused_cache_clear();
    return released;
}

// ---------------------------------------------------------------------------
// Hashed group-by with the group table in the library's own device image, for
// callers that cannot allocate device memory.
namespace {

// 2 * SJQ_STATIC_MAX_GROUPS slots + the side slot, three int64 arrays, each padded to 256 bytes.
static __device__ __align__(256) unsigned char g_static_group_table[SJQ_STATIC_WORKSPACE_BYTES];

} // namespace

extern "C" sjq_status sjq_run_hashed_static(const sjq_col *fact, int nfact, const sjq_pred *preds, int npreds,
                                            const sjq_join *joins, int njoins, const sjq_key_expr *key,
                                            const sjq_agg_expr *agg, int64_t capacity, const sjq_result *out,
                                            const sjq_run_opts *opts_, void *stream, sjq_run_info *info)
{
    if (!out || capacity <= 0) return SJQ_ERR_INVALID_ARG;
    if (capacity > SJQ_STATIC_MAX_GROUPS) return SJQ_ERR_STATIC_LIMIT;
    sjq_result_spec spec{SJQ_HASHED, 0, capacity};
    size_t need = 0;
    if (sjq_run_workspace_bytes(&spec, &need) != SJQ_OK || need > SJQ_STATIC_WORKSPACE_BYTES)
        return SJQ_ERR_STATIC_LIMIT;

    // In host code the array's name is only a stand-in; the kernels need its device address,
    // looked up once per device with that device current.
    static thread_local void *table_addr[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        (void)cudaGetLastError();
        return SJQ_ERR_CUDA;
    }
    if (!table_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_group_table) != cudaSuccess || !p) {
            (void)cudaGetLastError();
            return SJQ_ERR_CUDA;
        }
        table_addr[dev] = p;
    }
    sjq_result r = *out;
    r.workspace = table_addr[dev];
    r.workspace_bytes = SJQ_STATIC_WORKSPACE_BYTES;
    sjq_run_opts opts{};
    if (opts_) opts = *opts_;
    opts.accumulate = 0; // the shared table holds the last call's groups: always start from a cleared table
    opts.specialise = 0; // loading a compiled module allocates device memory: this entry point only interprets
    return sjq_run(fact, nfact, preds, npreds, joins, njoins, key, agg, &spec, &r, &opts, stream, info);
}
