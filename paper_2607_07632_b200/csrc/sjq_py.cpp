// The marshalling of sjq_run for the Python binding, as a CPython extension module.
//
// A query over few rows takes the GPU some 10 us, so what the binding does before the call decides how fast such
// queries follow one another: filling the argument structures through ctypes took 19 us a call, here it takes 3.
// Nothing is kept from one call for the next, and nothing is decided here: the module reads the same attributes of the
// same objects (columns, predicates, joins, expressions, options) and calls the C ABI.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstring>
#include <vector>

#include "sjq.h"

namespace {

#define SJQ_NAMES(X)                                                                                                   \
    X(data_ptr) X(dtype) X(is_cuda) X(is_contiguous) X(dim) X(numel) X(col) X(op) X(lo) X(hi) X(values) X(handle)       \
    X(terms) X(offset) X(modulo) X(src) X(a) X(b) X(mult) X(x) X(y) X(want_count) X(sums) X(counts) X(keys)             \
    X(n_groups) X(status_dev) X(workspace) X(sync) X(nbytes) X(get_device) X(info) X(block_threads)                     \
    X(ctas_per_sm) X(eager_loads) X(agg_path)                                                                          \
    X(smem_tables) X(compaction) X(accumulate) X(order) X(events) X(cuda_event) X(specialise) X(rows_per_lane)          \
    X(no_filter_bitmap) X(host_copy_all) X(dense_slots) X(group_hash_always) X(warp_agg) X(unfused_scratch)             \
    X(pass_ppm) X(hot_keys) X(hot_scratch) X(l0_bulk)

struct Names {
#define X(n) PyObject *n;
    SJQ_NAMES(X)
#undef X
} N;

PyObject *g_int32, *g_int64, *g_ops, *g_aggs; // torch.int32, torch.int64, names of operators and aggregates -> numbers

// A reference that is given back at the end of its scope.
struct Ref {
    PyObject *p;
    explicit Ref(PyObject *o) : p(o) {}
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
    ~Ref() { Py_XDECREF(p); }
    explicit operator bool() const { return p != nullptr; }
};

// Integers wrap to the field's width, as the fields of a ctypes structure do.
bool as_int(PyObject *o, int64_t *v)
{
    *v = (int64_t)PyLong_AsUnsignedLongLongMask(o);
    return !(*v == -1 && PyErr_Occurred());
}
bool get_int(PyObject *o, PyObject *name, int64_t *v)
{
    Ref a(PyObject_GetAttr(o, name));
    return a && as_int(a.p, v);
}
bool get_int(PyObject *o, PyObject *name, int32_t *v)
{
    int64_t w = 0;
    if (!get_int(o, name, &w)) return false;
    *v = (int32_t)w;
    return true;
}
bool get_flag(PyObject *o, PyObject *name, int32_t *v)
{
    Ref a(PyObject_GetAttr(o, name));
    const int t = a ? PyObject_IsTrue(a.p) : -1;
    *v = t > 0;
    return t >= 0;
}
bool call_int(PyObject *o, PyObject *method, int64_t *v)
{
    Ref a(PyObject_CallMethodNoArgs(o, method));
    return a && as_int(a.p, v);
}
// Address of a tensor's data; None gives NULL.
template <typename T>
bool pointer_of(PyObject *o, T **p, int64_t *numel = nullptr)
{
    *p = nullptr;
    if (numel) *numel = 0;
    if (o == Py_None) return true;
    int64_t v = 0;
    if (!call_int(o, N.data_ptr, &v) || (numel && !call_int(o, N.numel, numel))) return false;
    *p = reinterpret_cast<T *>(v);
    return true;
}
template <typename T>
bool get_pointer(PyObject *o, PyObject *name, T **p, int64_t *numel = nullptr)
{
    Ref a(PyObject_GetAttr(o, name));
    return a && pointer_of(a.p, p, numel);
}
bool number_of(PyObject *names, PyObject *key, int32_t *v)
{
    PyObject *n = PyDict_GetItemWithError(names, key);
    int64_t w = 0;
    if (!n) {
        if (!PyErr_Occurred()) PyErr_SetObject(PyExc_KeyError, key);
        return false;
    }
    if (!as_int(n, &w)) return false;
    *v = (int32_t)w;
    return true;
}

struct Columns {
    std::vector<PyObject *> names; // borrowed
    std::vector<sjq_col> cols;

    bool read(PyObject *dict)
    {
        PyObject *name, *t;
        Py_ssize_t pos = 0;
        names.reserve(PyDict_GET_SIZE(dict));
        cols.reserve(PyDict_GET_SIZE(dict));
        while (PyDict_Next(dict, &pos, &name, &t)) {
            sjq_col c{};
            Ref dtype(PyObject_GetAttr(t, N.dtype)), cuda(PyObject_GetAttr(t, N.is_cuda));
            if (!dtype || !cuda) return false;
            Ref contiguous(PyObject_CallMethodNoArgs(t, N.is_contiguous));
            int64_t dim = 0, data = 0;
            if (!contiguous || !call_int(t, N.dim, &dim)) return false;
            if ((dtype.p != g_int32 && dtype.p != g_int64) || cuda.p != Py_True || contiguous.p != Py_True || dim != 1) {
                PyErr_SetString(PyExc_ValueError, "columns must be contiguous 1-D int32/int64 CUDA tensors");
                return false;
            }
            if (!call_int(t, N.data_ptr, &data) || !call_int(t, N.numel, &c.n)) return false;
            c.data = reinterpret_cast<const void *>(data);
            c.dtype = dtype.p == g_int64 ? SJQ_I64 : SJQ_I32;
            names.push_back(name);
            cols.push_back(c);
        }
        return true;
    }
    bool index(PyObject *name, int32_t *i) const
    {
        for (size_t k = 0; k < names.size(); ++k)
            if (names[k] == name) {
                *i = (int32_t)k;
                return true;
            }
        for (size_t k = 0; k < names.size(); ++k) {
            const int same = PyObject_RichCompareBool(names[k], name, Py_EQ);
            if (same < 0) return false;
            if (same) {
                *i = (int32_t)k;
                return true;
            }
        }
        PyErr_Format(PyExc_ValueError, "%R is not a column", name);
        return false;
    }
};

struct Predicates {
    std::vector<sjq_pred> preds;
    std::vector<std::vector<int64_t>> sets;

    bool read(PyObject *seq, const Columns &C)
    {
        Ref fast(PySequence_Fast(seq, "predicates"));
        if (!fast) return false;
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast.p);
        preds.resize(n);
        sets.resize(n);
        for (Py_ssize_t i = 0; i < n; ++i) {
            PyObject *p = PySequence_Fast_GET_ITEM(fast.p, i);
            sjq_pred &d = preds[i];
            Ref col(PyObject_GetAttr(p, N.col)), op(PyObject_GetAttr(p, N.op)), values(PyObject_GetAttr(p, N.values));
            if (!col || !op || !values || !C.index(col.p, &d.col) || !number_of(g_ops, op.p, &d.op) ||
                !get_int(p, N.lo, &d.lo) || !get_int(p, N.hi, &d.hi))
                return false;
            Ref vals(PySequence_Fast(values.p, "values of a predicate"));
            if (!vals) return false;
            const Py_ssize_t m = PySequence_Fast_GET_SIZE(vals.p);
            sets[i].resize(m > 0 ? m : 1);
            for (Py_ssize_t k = 0; k < m; ++k)
                if (!as_int(PySequence_Fast_GET_ITEM(vals.p, k), &sets[i][k])) return false;
            d.set = sets[i].data();
            d.nset = (int32_t)m;
        }
        return true;
    }
};

bool read_term(PyObject *t, const Columns &C, sjq_term *out)
{
    *out = sjq_term{};
    if (t == Py_None) return true;
    Ref src(PyObject_GetAttr(t, N.src)), a(PyObject_GetAttr(t, N.a));
    if (!src || !a || !get_int(t, N.mult, &out->mult)) return false;
    if (PyUnicode_Check(src.p) && PyUnicode_CompareWithASCIIString(src.p, "FACT") == 0) return C.index(a.p, &out->a);
    out->src = SJQ_SRC_PAYLOAD;
    Ref whole(PyNumber_Long(a.p));
    int64_t join = 0;
    if (!whole || !as_int(whole.p, &join)) return false;
    out->a = (int32_t)join;
    return get_int(t, N.b, &out->b);
}

// `convert`: each entry goes through int() first, as RunOpts.to_c does with measured fractions (they may be floats).
bool read_ints(PyObject *o, PyObject *name, int32_t *out, int most, int32_t *count, bool convert)
{
    Ref seq(PyObject_GetAttr(o, name));
    if (!seq) return false;
    Ref fast(PySequence_Fast(seq.p, "a sequence of integers"));
    if (!fast) return false;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast.p);
    if (n > most) {
        PyErr_SetString(PyExc_IndexError, "more entries than predicates and joins");
        return false;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        int64_t v = 0;
        PyObject *entry = PySequence_Fast_GET_ITEM(fast.p, i);
        Ref whole(convert ? PyNumber_Long(entry) : Py_NewRef(entry));
        if (!whole || !as_int(whole.p, &v)) return false;
        out[i] = (int32_t)v;
    }
    if (count) *count = (int32_t)n;
    return true;
}

bool read_opts(PyObject *p, sjq_run_opts *o)
{
    if (!get_int(p, N.block_threads, &o->block_threads) || !get_int(p, N.ctas_per_sm, &o->ctas_per_sm) ||
        !get_flag(p, N.eager_loads, &o->eager_loads) || !get_int(p, N.agg_path, &o->agg_path) ||
        !get_int(p, N.smem_tables, &o->smem_tables) || !get_int(p, N.compaction, &o->compaction) ||
        !get_flag(p, N.accumulate, &o->accumulate) || !get_flag(p, N.specialise, &o->specialise) ||
        !get_int(p, N.rows_per_lane, &o->rows_per_lane) || !get_flag(p, N.no_filter_bitmap, &o->no_filter_bitmap) ||
        !get_flag(p, N.host_copy_all, &o->host_copy_all) || !get_int(p, N.dense_slots, &o->dense_slots) ||
        !get_flag(p, N.group_hash_always, &o->group_hash_always) || !get_int(p, N.warp_agg, &o->warp_agg) ||
        !get_int(p, N.hot_keys, &o->hot_keys) || !get_int(p, N.l0_bulk, &o->l0_bulk) ||
        !read_ints(p, N.order, o->order, SJQ_MAX_PREDS + SJQ_MAX_JOINS, &o->norder, false) ||
        !read_ints(p, N.pass_ppm, o->pass_ppm, SJQ_MAX_PREDS + SJQ_MAX_JOINS, nullptr, true))
        return false;
    int64_t bytes = 0;
    if (!get_pointer(p, N.hot_scratch, &o->hot_scratch, &bytes)) return false;
    o->hot_scratch_bytes = (size_t)bytes;
    if (!get_pointer(p, N.unfused_scratch, &o->unfused_scratch, &bytes)) return false;
    o->unfused_scratch_bytes = (size_t)bytes;
    o->unfused = o->unfused_scratch != nullptr;
    Ref events(PyObject_GetAttr(p, N.events));
    if (!events) return false;
    if (events.p != Py_None) {
        Ref before(PySequence_GetItem(events.p, 0)), after(PySequence_GetItem(events.p, 1));
        int64_t b = 0, a = 0;
        if (!before || !after || !get_int(before.p, N.cuda_event, &b) || !get_int(after.p, N.cuda_event, &a)) return false;
        o->event_before = reinterpret_cast<void *>(b);
        o->event_after = reinterpret_cast<void *>(a);
    }
    return true;
}

// The scratch with which a pass clears its result: the kernel writes SJQ_SYNC_BYTES through it, so a tensor that is shorter,
// or not on the device of the call, must not reach it.  A result without the attribute, or with None, brings none.
bool read_sync(PyObject *result, int64_t device, void **sync, bool *small)
{
    *small = false;
    Ref t(PyObject_GetAttr(result, N.sync));
    if (!t) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
        PyErr_Clear();
        return true;
    }
    int64_t bytes = 0, at = 0;
    if (!pointer_of(t.p, sync)) return false;
    if (t.p == Py_None) return true;
    if (!get_int(t.p, N.nbytes, &bytes) || !call_int(t.p, N.get_device, &at)) return false;
    Ref contiguous(PyObject_CallMethodNoArgs(t.p, N.is_contiguous));
    if (!contiguous) return false;
    if (at != device || contiguous.p != Py_True) {
        PyErr_SetString(PyExc_ValueError, "the sync words of a result must be a contiguous tensor on the device of its columns");
        return false;
    }
    *small = bytes < SJQ_SYNC_BYTES;
    return true;
}

// run(fact, preds, joins, key, agg, mode, num_groups, capacity, opts, result, stream, hot_scratch, device) -> status
// `hot_scratch()` supplies the scratch of the hot-key table where the options bring none and a join could use it.
PyObject *py_run(PyObject *, PyObject *const *args, Py_ssize_t nargs)
{
    if (nargs != 12 && nargs != 13) {
        PyErr_SetString(PyExc_TypeError, "run takes 12 or 13 arguments");
        return nullptr;
    }
    PyObject *fact = args[0], *joins = args[2], *key = args[3], *agg = args[4], *opts = args[8], *result = args[9];
    Ref columns(nullptr); // of another mapping than a dict
    if (!PyDict_CheckExact(fact)) {
        columns.p = PyDict_New();
        if (!columns || PyDict_Update(columns.p, fact) != 0) return nullptr;
        fact = columns.p;
    }
    Columns C;
    Predicates P;
    if (!C.read(fact) || !P.read(args[1], C)) return nullptr;

    sjq_run_opts o{};
    if (opts != Py_None && !read_opts(opts, &o)) return nullptr;

    Ref fast(PySequence_Fast(joins, "joins"));
    if (!fast) return nullptr;
    const Py_ssize_t njoins = PySequence_Fast_GET_SIZE(fast.p);
    std::vector<sjq_join> J(njoins);
    bool hashed = false;
    for (Py_ssize_t j = 0; j < njoins; ++j) {
        Ref pair(PySequence_Fast(PySequence_Fast_GET_ITEM(fast.p, j), "a join is (column, table)"));
        if (!pair) return nullptr;
        if (PySequence_Fast_GET_SIZE(pair.p) != 2) {
            PyErr_SetString(PyExc_ValueError, "a join is (column, table)");
            return nullptr;
        }
        Ref handle(PyObject_GetAttr(PySequence_Fast_GET_ITEM(pair.p, 1), N.handle));
        int64_t h = 0;
        if (!handle || !C.index(PySequence_Fast_GET_ITEM(pair.p, 0), &J[j].fk_col) ||
            (handle.p != Py_None && !as_int(handle.p, &h)))
            return nullptr;
        J[j].table = reinterpret_cast<const sjq_table *>(h);
        sjq_dim_layout L;
        hashed = hashed || (h && sjq_table_info(J[j].table, &L) == SJQ_OK &&
                            (L.kind == SJQ_TABLE_HASH_I32 || L.kind == SJQ_TABLE_HASH_I64));
    }

    sjq_key_expr K{};
    if (key != Py_None) {
        Ref terms(PyObject_GetAttr(key, N.terms));
        if (!terms) return nullptr;
        Ref seq(PySequence_Fast(terms.p, "terms of a key"));
        if (!seq) return nullptr;
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq.p);
        if (n > SJQ_MAX_KEY_TERMS) {
            PyErr_SetString(PyExc_ValueError, "too many key terms");
            return nullptr;
        }
        K.nterms = (int32_t)n;
        for (Py_ssize_t i = 0; i < n; ++i)
            if (!read_term(PySequence_Fast_GET_ITEM(seq.p, i), C, &K.t[i])) return nullptr;
        if (!get_int(key, N.offset, &K.offset) || !get_int(key, N.modulo, &K.modulo)) return nullptr;
    }

    sjq_agg_expr A{};
    {
        Ref op(PyObject_GetAttr(agg, N.op)), x(PyObject_GetAttr(agg, N.x)), y(PyObject_GetAttr(agg, N.y));
        if (!op || !x || !y || !number_of(g_aggs, op.p, &A.op) || !read_term(x.p, C, &A.x) || !read_term(y.p, C, &A.y) ||
            !get_flag(agg, N.want_count, &A.want_count))
            return nullptr;
    }

    sjq_result_spec S{};
    int64_t mode = 0, stream = 0;
    if (!as_int(args[5], &mode) || !as_int(args[6], &S.num_groups) || !as_int(args[7], &S.capacity) ||
        !as_int(args[10], &stream))
        return nullptr;
    S.mode = (int32_t)mode;

    sjq_result R{};
    int64_t workspace_bytes = 0;
    if (!get_pointer(result, N.sums, &R.sums) || !get_pointer(result, N.counts, &R.counts) ||
        !get_pointer(result, N.keys, &R.keys) || !get_pointer(result, N.n_groups, &R.n_groups) ||
        !get_pointer(result, N.status_dev, &R.status) || !get_pointer(result, N.workspace, &R.workspace, &workspace_bytes))
        return nullptr;
    R.workspace_bytes = (size_t)workspace_bytes;
    int64_t device = 0;
    bool small = false;
    if ((nargs > 12 && !as_int(args[12], &device)) || !read_sync(result, device, &o.sync, &small)) return nullptr;
    if (small) return PyLong_FromLong(SJQ_ERR_BUFFER_SMALL);

    Ref scratch(nullptr); // held until the call has enqueued its work
    if (hashed && !o.hot_scratch && o.hot_keys != 2) {
        scratch.p = PyObject_CallNoArgs(args[11]);
        int64_t bytes = 0;
        if (!scratch || !pointer_of(scratch.p, &o.hot_scratch, &bytes)) return nullptr;
        o.hot_scratch_bytes = (size_t)bytes;
    }

    Ref info(PyObject_GetAttr(result, N.info));
    Py_buffer buffer;
    if (!info || PyObject_GetBuffer(info.p, &buffer, PyBUF_WRITABLE) != 0) return nullptr;
    if (buffer.len < (Py_ssize_t)sizeof(sjq_run_info)) {
        PyBuffer_Release(&buffer);
        PyErr_SetString(PyExc_ValueError, "the result's run information is too small");
        return nullptr;
    }
    sjq_status st;
    Py_BEGIN_ALLOW_THREADS
    st = sjq_run(C.cols.data(), (int)C.cols.size(), P.preds.data(), (int)P.preds.size(), J.data(), (int)njoins,
                 key != Py_None ? &K : nullptr, &A, &S, &R, &o, reinterpret_cast<void *>(stream),
                 static_cast<sjq_run_info *>(buffer.buf));
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&buffer);
    return PyLong_FromLong(st);
}

// init(torch.int32, torch.int64, operators, aggregates): what the other functions compare with.
PyObject *py_init(PyObject *, PyObject *const *args, Py_ssize_t nargs)
{
    if (nargs != 4 || !PyDict_Check(args[2]) || !PyDict_Check(args[3])) {
        PyErr_SetString(PyExc_TypeError, "init(int32, int64, operators, aggregates)");
        return nullptr;
    }
    PyObject **keep[] = {&g_int32, &g_int64, &g_ops, &g_aggs};
    for (int i = 0; i < 4; ++i) {
        Py_INCREF(args[i]);
        Py_XSETREF(*keep[i], args[i]);
    }
    Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"run", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(py_run)), METH_FASTCALL, "sjq_run"},
    {"init", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(py_init)), METH_FASTCALL, "constants"},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", "argument marshalling of the sjq binding", -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

} // namespace

PyMODINIT_FUNC PyInit__marshal(void)
{
#define X(n)                                                                                                           \
    if (!(N.n = PyUnicode_InternFromString(#n))) return nullptr;
    SJQ_NAMES(X)
#undef X
    return PyModule_Create(&g_module);
}
