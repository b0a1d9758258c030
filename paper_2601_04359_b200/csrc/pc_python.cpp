// Native side of the Python binding: takes the binding's Segment / Cache objects and tensors apart and calls the C ABI.
//
// The calls of a frame step are short on the GPU for small frames, so the time that the host takes to issue them decides:
// building the same structs through ctypes took 51 us of host time for a frame step (6.4 us per cache, 9.6 us for the plan,
// 2.3 us per array pointer), more than the launches of the step.  Host time of a
// pass, ctypes against this file: frame step 51 -> 27 us (fp32 62 -> 24, with a shorter launch list), attention over a cache
// 19.8 -> 10.6, mask, score, pack and attend 82 -> 36; the small bf16 step 53.8 -> 37.5 us a pass.
// Tensors are read through their Python methods (data_ptr, is_contiguous, shape), so nothing here depends on torch's C++ ABI.
// Each function returns the pc_status; the Python wrapper raises.  The interpreter lock is released around the library calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>
#include <vector>

#include "packcache.h"

namespace {

PyObject *s_data_ptr, *s_is_contiguous, *s_shape, *s_k, *s_v, *s_pos, *s_n_tokens, *s_anchors, *s_history, *s_frame_count, *s_value;
PyObject *g_as_i32;       // numpy.ascontiguousarray(x, dtype=int32), for anything that is not an int32 array already

bool failed() { return PyErr_Occurred() != nullptr; }

// Address of a tensor (None: null).  Sets an error if it is not contiguous.
void *tensor_ptr(PyObject *t) {
    if (t == Py_None) return nullptr;
    PyObject *c = PyObject_CallMethodNoArgs(t, s_is_contiguous);
    if (!c) return nullptr;
    const int ok = PyObject_IsTrue(c);
    Py_DECREF(c);
    if (ok <= 0) {
        if (ok == 0) PyErr_SetString(PyExc_AssertionError, "tensors passed to the library must be contiguous");
        return nullptr;
    }
    PyObject *p = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!p) return nullptr;
    void *r = PyLong_AsVoidPtr(p);
    Py_DECREF(p);
    return r;
}

int32_t int_of(PyObject *o) { return (int32_t)PyLong_AsLong(o); }

int32_t int_attr(PyObject *o, PyObject *name) {
    PyObject *v = PyObject_GetAttr(o, name);
    if (!v) return 0;
    PyObject *i = PyNumber_Index(v);                  // numpy integers as well
    Py_DECREF(v);
    if (!i) return 0;
    const int32_t r = int_of(i);
    Py_DECREF(i);
    return r;
}

// first extent of a tensor
int32_t rows_of(PyObject *t) {
    PyObject *s = PyObject_GetAttr(t, s_shape);
    if (!s) return 0;
    PyObject *n = PySequence_GetItem(s, 0);
    Py_DECREF(s);
    if (!n) return 0;
    const int32_t r = int_of(n);
    Py_DECREF(n);
    return r;
}

void *handle_of(PyObject *h) {                        // a ctypes c_void_p, or None after close()
    if (h == Py_None) return nullptr;
    PyObject *v = PyObject_GetAttr(h, s_value);
    if (!v) return nullptr;
    void *p = v == Py_None ? nullptr : PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return p;
}

void *stream_of(PyObject *s) { return PyLong_AsVoidPtr(s); }

// A host array of int32 with any number of dimensions, held for the duration of a call.
struct Ints {
    Py_buffer view{};
    const int32_t *p = nullptr;
    int32_t n = 0;            // its length (first extent)
    int64_t size = 0;         // elements in all
    bool take(PyObject *o) {
        if (!as_is(o)) {
            PyObject *a = PyObject_CallOneArg(g_as_i32, o);
            if (!a) return false;
            const bool ok = as_is(a);                 // the buffer holds the array from here on
            Py_DECREF(a);
            if (!ok) {
                if (!failed()) PyErr_SetString(PyExc_TypeError, "an array of integers is expected");
                return false;
            }
        }
        return true;
    }
    bool as_is(PyObject *o) {
        if (!PyObject_CheckBuffer(o)) return false;
        if (PyObject_GetBuffer(o, &view, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS) != 0) {
            PyErr_Clear();
            return false;
        }
        const char *f = view.format ? view.format : "B";
        if (view.itemsize != 4 || view.ndim < 1 || f[1] != '\0' || (f[0] != 'i' && f[0] != 'l')) {
            PyBuffer_Release(&view);
            view = Py_buffer{};
            return false;
        }
        p = static_cast<const int32_t *>(view.buf);
        n = (int32_t)view.shape[0];
        size = view.len / 4;
        return true;
    }
    // the library reads (or writes) this many entries: a shorter array is an error
    bool holds(int32_t want, const char *what) const {
        if (size >= want) return true;
        PyErr_Format(PyExc_ValueError, "%s has %lld entries, %d are needed", what, (long long)size, (int)want);
        return false;
    }
    ~Ints() {
        if (view.obj) PyBuffer_Release(&view);
    }
};

bool segment_of(PyObject *o, pc_segment *out) {
    *out = pc_segment{};
    PyObject *k = PyObject_GetAttr(o, s_k), *v = PyObject_GetAttr(o, s_v), *pos = PyObject_GetAttr(o, s_pos);
    if (k && v && pos) {
        out->k = tensor_ptr(k);
        if (!failed()) out->v = tensor_ptr(v);
        if (!failed()) out->pos = static_cast<int32_t *>(tensor_ptr(pos));
        if (!failed()) out->n_tokens = int_attr(o, s_n_tokens);
        if (!failed() && k != Py_None) out->capacity = rows_of(k);
    }
    Py_XDECREF(k);
    Py_XDECREF(v);
    Py_XDECREF(pos);
    return !failed();
}

struct CacheArg {
    pc_cache c{};
    Ints counts;
    bool take(PyObject *o) {
        PyObject *a = PyObject_GetAttr(o, s_anchors);
        if (!a) return false;
        const bool ok_a = segment_of(a, &c.anchors);
        Py_DECREF(a);
        if (!ok_a) return false;
        PyObject *h = PyObject_GetAttr(o, s_history);
        if (!h) return false;
        const bool ok_h = segment_of(h, &c.history);
        Py_DECREF(h);
        if (!ok_h) return false;
        PyObject *f = PyObject_GetAttr(o, s_frame_count);
        if (!f) return false;
        const bool ok_f = counts.take(f);
        Py_DECREF(f);
        c.n_frames = counts.n;
        c.frame_count = counts.p;
        return ok_f;
    }
};

template <typename F> PyObject *call(F f) {
    pc_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

bool arity(Py_ssize_t got, Py_ssize_t want) {
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, got);
    return false;
}

// Tensors of a call, in order; null for None.
template <int N> struct Tensors {
    void *p[N];
    bool take(PyObject *const *a) {
        for (int i = 0; i < N; ++i) {
            p[i] = tensor_ptr(a[i]);
            if (failed()) return false;
        }
        return true;
    }
};

PyObject *plan_budget(PyObject *, PyObject *const *a, Py_ssize_t n) {       // kind, param, total, keep_full, min_quota, avail, out
    if (!arity(n, 7)) return nullptr;
    pc_budget_params p{};
    p.kind = int_of(a[0]);
    p.param = PyFloat_AsDouble(a[1]);
    p.total = PyLong_AsLongLong(a[2]);
    p.keep_full = int_of(a[3]);
    p.min_quota = int_of(a[4]);
    Ints avail, out;
    if (failed() || !avail.take(a[5]) || !out.take(a[6]) || !out.holds(avail.n, "the budget array")) return nullptr;
    return PyLong_FromLong((long)pc_plan_budget(&p, avail.n, avail.p, const_cast<int32_t *>(out.p)));
}

PyObject *total(PyObject *, PyObject *const *a, Py_ssize_t n) {             // sum of an int32 array
    if (!arity(n, 1)) return nullptr;
    Ints v;
    if (!v.take(a[0])) return nullptr;
    int64_t s = 0;
    for (int64_t i = 0; i < v.size; ++i) s += v.p[i];
    return PyLong_FromLongLong(s);
}

PyObject *score(PyObject *, PyObject *const *a, Py_ssize_t n) {             // ctx, src, q, q_pos, budget, valid, override, scores, sel, stream
    if (!arity(n, 10)) return nullptr;
    CacheArg src;
    Ints budget;
    Tensors<2> q;
    Tensors<4> t;
    void *ctx = handle_of(a[0]), *stream = stream_of(a[9]);
    if (failed() || !src.take(a[1]) || !q.take(a + 2) || !budget.take(a[4]) || !budget.holds(src.c.n_frames, "budget") || !t.take(a + 5)) return nullptr;
    const int32_t n_q = a[2] == Py_None ? 0 : rows_of(a[2]);
    if (failed()) return nullptr;
    return call([&] {
        return pc_score(static_cast<pc_ctx *>(ctx), &src.c, q.p[0], static_cast<int32_t *>(q.p[1]), n_q, budget.p,
                        static_cast<uint8_t *>(t.p[0]), static_cast<float *>(t.p[1]), static_cast<float *>(t.p[2]),
                        static_cast<int32_t *>(t.p[3]), stream);
    });
}

PyObject *compact(PyObject *, PyObject *const *a, Py_ssize_t n) {           // ctx, src, sel, budget, delta_t, dst, stream
    if (!arity(n, 7)) return nullptr;
    CacheArg src, dst;
    Ints budget;
    Tensors<1> sel;
    void *ctx = handle_of(a[0]), *stream = stream_of(a[6]);
    const int32_t delta_t = int_of(a[4]);
    if (failed() || !src.take(a[1]) || !sel.take(a + 2) || !budget.take(a[3]) || !budget.holds(src.c.n_frames, "budget") || !dst.take(a[5])) return nullptr;
    return call([&] { return pc_compact(static_cast<pc_ctx *>(ctx), &src.c, static_cast<int32_t *>(sel.p[0]), budget.p, delta_t, &dst.c, stream); });
}

PyObject *attend_frame(PyObject *, PyObject *const *a, Py_ssize_t n) {      // ctx, cache, current, q, q_pos, out, lse, stream
    if (!arity(n, 8)) return nullptr;
    CacheArg cache;
    pc_segment cur{};
    Tensors<4> t;
    void *ctx = handle_of(a[0]), *stream = stream_of(a[7]);
    if (failed() || !cache.take(a[1]) || (a[2] != Py_None && !segment_of(a[2], &cur)) || !t.take(a + 3)) return nullptr;
    const int32_t n_q = rows_of(a[3]);
    if (failed()) return nullptr;
    return call([&] {
        return pc_attend_frame(static_cast<pc_ctx *>(ctx), &cache.c, a[2] != Py_None ? &cur : nullptr, t.p[0], static_cast<int32_t *>(t.p[1]),
                               n_q, t.p[2], static_cast<float *>(t.p[3]), stream);
    });
}

PyObject *attend_prepare(PyObject *, PyObject *const *a, Py_ssize_t n) {    // ctx, cache, current, stream
    if (!arity(n, 4)) return nullptr;
    CacheArg cache;
    pc_segment cur{};
    void *ctx = handle_of(a[0]), *stream = stream_of(a[3]);
    if (failed() || !cache.take(a[1]) || (a[2] != Py_None && !segment_of(a[2], &cur))) return nullptr;
    return call([&] { return pc_attend_prepare(static_cast<pc_ctx *>(ctx), &cache.c, a[2] != Py_None ? &cur : nullptr, stream); });
}

PyObject *attend_prepared(PyObject *, PyObject *const *a, Py_ssize_t n) {   // ctx, q, q_pos, out, lse, stream
    if (!arity(n, 6)) return nullptr;
    Tensors<4> t;
    void *ctx = handle_of(a[0]), *stream = stream_of(a[5]);
    if (failed() || !t.take(a + 1)) return nullptr;
    const int32_t n_q = rows_of(a[1]);
    if (failed()) return nullptr;
    return call([&] {
        return pc_attend_prepared(static_cast<pc_ctx *>(ctx), t.p[0], static_cast<int32_t *>(t.p[1]), n_q, t.p[2], static_cast<float *>(t.p[3]), stream);
    });
}

PyObject *attend_mass(PyObject *, PyObject *const *a, Py_ssize_t n) {       // ctx, lse, mass, n_keys, stream
    if (!arity(n, 5)) return nullptr;
    Tensors<2> t;
    void *ctx = handle_of(a[0]), *stream = stream_of(a[4]);
    const int32_t n_keys = int_of(a[3]);
    if (failed() || !t.take(a + 1)) return nullptr;
    return call([&] { return pc_attend_mass(static_cast<pc_ctx *>(ctx), static_cast<float *>(t.p[0]), static_cast<float *>(t.p[1]), n_keys, stream); });
}

PyObject *frame_step(PyObject *, PyObject *const *a, Py_ssize_t n) {        // ctx, src, budget, delta_t, dst, q, q_pos, scores, sel, out, lse, stream
    if (!arity(n, 12)) return nullptr;
    CacheArg src, dst;
    Ints budget;
    Tensors<6> t;
    void *ctx = handle_of(a[0]), *stream = stream_of(a[11]);
    const int32_t delta_t = int_of(a[3]);
    if (failed() || !src.take(a[1]) || !budget.take(a[2]) || !budget.holds(src.c.n_frames, "budget") || !dst.take(a[4]) || !t.take(a + 5)) return nullptr;
    const int32_t n_q = rows_of(a[5]);
    if (failed()) return nullptr;
    return call([&] {
        return pc_frame_step(static_cast<pc_ctx *>(ctx), &src.c, budget.p, delta_t, &dst.c, t.p[0], static_cast<int32_t *>(t.p[1]), n_q,
                             static_cast<float *>(t.p[2]), static_cast<int32_t *>(t.p[3]), t.p[4], static_cast<float *>(t.p[5]), stream);
    });
}

PyObject *window_append(PyObject *, PyObject *const *a, Py_ssize_t n) {     // window, frame, stream
    if (!arity(n, 3)) return nullptr;
    pc_segment frame{};
    void *w = handle_of(a[0]), *stream = stream_of(a[2]);
    if (failed() || !segment_of(a[1], &frame)) return nullptr;
    return call([&] { return pc_window_append(static_cast<pc_window *>(w), &frame, stream); });
}

PyObject *window_step(PyObject *, PyObject *const *a, Py_ssize_t n) {       // window, q, q_pos, out, lse, stream -> (status, regime)
    if (!arity(n, 6)) return nullptr;
    Tensors<4> t;
    void *w = handle_of(a[0]), *stream = stream_of(a[5]);
    if (failed() || !t.take(a + 1)) return nullptr;
    const int32_t n_q = rows_of(a[1]);
    if (failed()) return nullptr;
    int32_t regime = -1;
    pc_status st;
    Py_BEGIN_ALLOW_THREADS
    st = pc_window_step(static_cast<pc_window *>(w), t.p[0], static_cast<int32_t *>(t.p[1]), n_q, t.p[2], static_cast<float *>(t.p[3]), &regime, stream);
    Py_END_ALLOW_THREADS
    return Py_BuildValue("ii", (int)st, (int)regime);
}

PyObject *set_i32_converter(PyObject *, PyObject *f) {
    Py_INCREF(f);
    Py_XSETREF(g_as_i32, f);
    Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(plan_budget), FAST(total), FAST(score), FAST(compact), FAST(attend_frame), FAST(attend_prepare), FAST(attend_prepared),
                         FAST(attend_mass), FAST(frame_step), FAST(window_append), FAST(window_step),
                         {"set_i32_converter", set_i32_converter, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_packcache_py", "Calls of libpackcache.so on the binding's objects.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__packcache_py(void) {
    struct { PyObject **at; const char *name; } names[] = {{&s_data_ptr, "data_ptr"}, {&s_is_contiguous, "is_contiguous"}, {&s_shape, "shape"},
        {&s_k, "k"}, {&s_v, "v"}, {&s_pos, "pos"}, {&s_n_tokens, "n_tokens"}, {&s_anchors, "anchors"}, {&s_history, "history"},
        {&s_frame_count, "frame_count"}, {&s_value, "value"}};
    for (auto &x : names)
        if (!(*x.at = PyUnicode_InternFromString(x.name))) return nullptr;
    return PyModule_Create(&module);
}
