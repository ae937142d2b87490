// The hot calls of the Python binding in native code: argument blocks filled from Python objects, and the call made with the
// interpreter's lock released.  What bounds a small call that the caller waits for is the host, before the kernel starts, and a queue
// of calls without a context as well.  Host time of a queued call, marshalled in Python by ctypes / here: one table 5.5 / 3.5 us, 32 tables
// 6.7 / 4.2; avsg_step_noalloc with 1, 8, 32 tables 8.2, 9.9, 13.7 / 4.3, 5.4, 7.8.  Calls alone, to the end: K = 256, one table 17.9 / 16.0 us,
// without a context 20.9 / 17.2; queues of such calls 8.1 / 5.7.
//
// Only what such calls usually carry is handled here (integers, objects with data_ptr(), lists and tuples of integers); the rest
// goes through the binding's own conversions, which are given to each function as a callable, so that what is accepted, and what
// is raised, is theirs.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include <limits>

#include "avsg.h"

namespace {

PyObject *s_data_ptr, *s_shape;

// The module's conversions, set once by the binding (set_binding).
PyObject *b_addr, *b_array, *b_lengths, *b_stream, *b_raw_stream, *b_device;

struct Held {                            // a reference that goes with its scope
    PyObject* o;
    explicit Held(PyObject* p = nullptr) : o(p) {}
    Held(const Held&) = delete;
    Held& operator=(const Held&) = delete;
    ~Held() { Py_XDECREF(o); }
};

// An integer's low 64 bits, as a ctypes field takes it.
bool low_bits(PyObject* o, uint64_t* v)
{
    *v = PyLong_AsUnsignedLongLongMask(o);
    return !(*v == (uint64_t)-1 && PyErr_Occurred());
}

// The address of a tensor, or an integer address itself.
bool address(PyObject* o, uint64_t* v)
{
    if (PyLong_Check(o)) return low_bits(o, v);
    Held p(PyObject_CallMethodNoArgs(o, s_data_ptr));
    if (p.o && PyLong_Check(p.o)) return low_bits(p.o, v);
    PyErr_Clear();
    Held q(PyObject_CallOneArg(b_addr, o));
    return q.o && low_bits(q.o, v);
}
bool address_or_null(PyObject* o, uint64_t* v)
{
    *v = 0;
    return o == Py_None || address(o, v);
}

// n integers that fit T from a list or tuple; false without an exception: something else.
template <typename T>
bool integers(PyObject* values, Py_ssize_t n, T* out)
{
    if (!PyList_CheckExact(values) && !PyTuple_CheckExact(values)) return false;
    if (PySequence_Fast_GET_SIZE(values) != n) return false;
    using limits = std::numeric_limits<T>;
    const long long least = (long long)limits::min(), most = sizeof(T) < 8 ? (long long)limits::max() : std::numeric_limits<long long>::max();
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject* o = PySequence_Fast_GET_ITEM(values, i);             // (exact integers run no code that could change the list)
        if (!PyLong_CheckExact(o)) return false;
        int over = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &over);
        if (over || v < least || v > most) return false;
        out[i] = (T)v;
    }
    return true;
}

// The handle of `stream`: None: the current one.
bool stream_handle(PyObject* stream, uint64_t* v)
{
    if (stream == Py_None && b_raw_stream) {
        Held dev(PyObject_CallNoArgs(b_device));
        if (!dev.o) return false;
        Held h(PyObject_CallOneArg(b_raw_stream, dev.o));
        return h.o && low_bits(h.o, v);
    }
    if (PyLong_Check(stream)) return low_bits(stream, v);
    Held h(PyObject_CallOneArg(b_stream, stream));
    if (!h.o) return false;
    if (h.o == Py_None) { *v = 0; return true; }
    return low_bits(h.o, v);
}

using StepFn = int (*)(avsg_ctx*, const avsg_step_args*, void*);
using NoAllocFn = int (*)(const avsg_noalloc_args*, void*);

// ---- Call: the argument block of a recurring call, in the caller's memory ----
struct Call {
    PyObject_HEAD
    avsg_step_args* args;
    int32_t* lengths;                    // [n]
    const uint64_t* ctx;                 // holds the context's handle, 0 when that is closed
    StepFn step, step_host;
    Py_ssize_t n;
    PyObject* array;                     // the same, for the binding (which takes any iterable of n numbers)
};

int call_init(PyObject* self, PyObject* args, PyObject*)
{
    Call* c = reinterpret_cast<Call*>(self);
    unsigned long long block, lengths, ctx, step, step_host;
    Py_ssize_t n;
    PyObject* array;
    if (!PyArg_ParseTuple(args, "KKnKKKO", &block, &lengths, &n, &ctx, &step, &step_host, &array)) return -1;
    c->args = reinterpret_cast<avsg_step_args*>(block);
    c->lengths = reinterpret_cast<int32_t*>(lengths);
    c->ctx = reinterpret_cast<const uint64_t*>(ctx);
    c->step = reinterpret_cast<StepFn>(step);
    c->step_host = reinterpret_cast<StepFn>(step_host);
    c->n = n;
    Py_INCREF(array);
    Py_XSETREF(c->array, array);
    return 0;
}
int call_traverse(PyObject* self, visitproc visit, void* arg)
{
    Py_VISIT(Py_TYPE(self));
    Py_VISIT(reinterpret_cast<Call*>(self)->array);
    return 0;
}
int call_clear(PyObject* self) { Py_CLEAR(reinterpret_cast<Call*>(self)->array); return 0; }
void call_dealloc(PyObject* self)
{
    PyTypeObject* type = Py_TYPE(self);
    PyObject_GC_UnTrack(self);
    call_clear(self);
    type->tp_free(self);
    Py_DECREF(type);
}

// a: indices, verified_len, slots, hit, miss_count, stream, stage_one_done, arriving
bool fill(Call* c, PyObject* const* a, uint64_t* stream)
{
    avsg_step_args* s = c->args;
    uint64_t v;
    if (!address_or_null(a[7], &v)) return false;
    s->arriving = reinterpret_cast<uint8_t*>(v);
    s->stage_one_done = nullptr;
    s->stage_one_done_value = 0;
    if (a[6] != Py_None) {
        Held word(PySequence_GetItem(a[6], 0)), value(PySequence_GetItem(a[6], 1));
        if (!word.o || !value.o || !address(word.o, &v)) return false;
        s->stage_one_done = reinterpret_cast<uint64_t*>(v);
        Held number(PyNumber_Long(value.o));
        if (!number.o || !low_bits(number.o, &v)) return false;
        s->stage_one_done_value = v;
    }
    s->verified_len_dev = nullptr;
    if (!integers(a[1], c->n, c->lengths)) {
        if (!PyList_CheckExact(a[1]) && !PyTuple_CheckExact(a[1]) && PyObject_HasAttr(a[1], s_data_ptr)) {
            if (!address(a[1], &v)) return false;
            s->verified_len_dev = reinterpret_cast<const int32_t*>(v);
        } else {
            Held done(PyObject_CallFunctionObjArgs(b_lengths, c->array, a[1], nullptr));
            if (!done.o) return false;
        }
    }
    if (!address(a[0], &v)) return false;
    s->indices = reinterpret_cast<const int32_t*>(v);
    if (!address(a[2], &v)) return false;
    s->slots = reinterpret_cast<int32_t*>(v);
    if (!address_or_null(a[3], &v)) return false;
    s->hit = reinterpret_cast<uint8_t*>(v);
    if (!address_or_null(a[4], &v)) return false;
    s->miss_count = reinterpret_cast<int32_t*>(v);
    return stream_handle(a[5], stream);
}

// The same arguments as fill(), then host.
PyObject* call_run(PyObject* self, PyObject* const* a, Py_ssize_t nargs)
{
    Call* c = reinterpret_cast<Call*>(self);
    uint64_t stream = 0;
    if (nargs != 9 || !c->ctx) { PyErr_SetString(PyExc_TypeError, "nine arguments, of a call that has been set up"); return nullptr; }
    const int host = PyObject_IsTrue(a[8]);
    if (host < 0 || !fill(c, a, &stream)) return nullptr;
    avsg_ctx* ctx = reinterpret_cast<avsg_ctx*>(*c->ctx);
    const StepFn fn = host ? c->step_host : c->step;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(ctx, c->args, reinterpret_cast<void*>(stream));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

PyMethodDef call_methods[] = {
    {"run", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(call_run)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyType_Slot call_slots[] = {{Py_tp_init, reinterpret_cast<void*>(call_init)},
                            {Py_tp_new, reinterpret_cast<void*>(PyType_GenericNew)},
                            {Py_tp_dealloc, reinterpret_cast<void*>(call_dealloc)},
                            {Py_tp_traverse, reinterpret_cast<void*>(call_traverse)},
                            {Py_tp_clear, reinterpret_cast<void*>(call_clear)},
                            {Py_tp_methods, call_methods},
                            {0, nullptr}};
PyType_Spec call_spec = {"paper_2609_37538_b200._python_calls.Call", sizeof(Call), 0, Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_GC, call_slots};

// ---- avsg_step_noalloc ----
// A host array of n integers: in `room` where that takes it, else what the binding makes of the values (kept in `owner`).
template <typename T>
bool host_array(PyObject* values, Py_ssize_t n, const char* kind, T* room, Held& owner, const T** at)
{
    *at = nullptr;
    if (values == Py_None) return true;
    if (n <= (Py_ssize_t)AVSG_NOALLOC_MAX_TABLES && integers(values, n, room)) { *at = room; return true; }
    owner.o = PyObject_CallFunction(b_array, "sOn", kind, values, n);                          // (owner, address)
    if (!owner.o) return false;
    uint64_t v = 0;
    PyObject* address_of = PyTuple_GetItem(owner.o, 1);
    if (!address_of || !low_bits(address_of, &v)) return false;
    *at = reinterpret_cast<const T*>(v);
    return true;
}

bool dimension(PyObject* shape, Py_ssize_t i, unsigned long* v)
{
    Held d(PySequence_GetItem(shape, i));
    if (!d.o) return false;
    *v = PyLong_AsUnsignedLongMask(d.o);
    return !(*v == (unsigned long)-1 && PyErr_Occurred());
}

// fn, tok, life, buffer, indices, kv, verified_len, max_lifetime, slots, hit, miss_count, status, row_stride, stream, kv_rows
PyObject* noalloc(PyObject*, PyObject* const* a, Py_ssize_t nargs)
{
    if (nargs != 15) { PyErr_SetString(PyExc_TypeError, "fifteen arguments"); return nullptr; }
    uint64_t fn = 0, v = 0, stream = 0;
    if (!low_bits(a[0], &fn)) return nullptr;
    Held tok_shape(PyObject_GetAttr(a[1], s_shape)), ids_shape(PyObject_GetAttr(a[4], s_shape)), rows_shape(PyObject_GetAttr(a[3], s_shape));
    if (!tok_shape.o || !ids_shape.o || !rows_shape.o) return nullptr;
    if (PySequence_Size(tok_shape.o) != 2 || PySequence_Size(ids_shape.o) != 3) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "tok has two dimensions, indices three");
        return nullptr;
    }
    unsigned long n, S, n_q, K, row_bytes;
    if (!dimension(tok_shape.o, 0, &n) || !dimension(tok_shape.o, 1, &S) || !dimension(ids_shape.o, 1, &n_q) ||
        !dimension(ids_shape.o, 2, &K) || !dimension(rows_shape.o, -1, &row_bytes))
        return nullptr;
    avsg_noalloc_args s = {};
    s.n = (uint32_t)n; s.n_tokens = (uint32_t)n_q; s.topk = (uint32_t)K; s.buffer_slots = (uint32_t)S; s.row_bytes = (uint32_t)row_bytes;
    if (!low_bits(a[7], &v)) return nullptr;
    s.max_lifetime = (int32_t)v;
    uint64_t kv_room[AVSG_NOALLOC_MAX_TABLES], stride_room[AVSG_NOALLOC_MAX_TABLES];
    int32_t length_room[AVSG_NOALLOC_MAX_TABLES];
    uint32_t rows_room[AVSG_NOALLOC_MAX_TABLES];
    Held kv_owner, stride_owner, length_owner, rows_owner;
    const uint64_t *kv = nullptr, *stride = nullptr;
    const int32_t* lengths = nullptr;
    const uint32_t* rows = nullptr;
    bool kv_here = n <= AVSG_NOALLOC_MAX_TABLES && (PyList_CheckExact(a[5]) || PyTuple_CheckExact(a[5])) &&
                   (unsigned long)PySequence_Fast_GET_SIZE(a[5]) == n;
    for (unsigned long i = 0; kv_here && i < n; ++i) {
        kv_here = (unsigned long)PySequence_Fast_GET_SIZE(a[5]) == n;  // (an object's data_ptr() may do anything)
        if (!kv_here) break;
        Held o(PySequence_Fast_GET_ITEM(a[5], i));
        Py_INCREF(o.o);
        if (!address(o.o, kv_room + i)) return nullptr;
    }
    if (kv_here) {
        kv = kv_room;
    } else {
        Held all(PySequence_List(a[5]));
        if (!all.o) return nullptr;
        for (Py_ssize_t i = 0; i < PyList_GET_SIZE(all.o); ++i) {
            if (!address(PyList_GET_ITEM(all.o, i), &v)) return nullptr;
            PyObject* number = PyLong_FromUnsignedLongLong(v);
            if (!number || PyList_SetItem(all.o, i, number) < 0) return nullptr;
        }
        if (!host_array(all.o, (Py_ssize_t)n, "Q", kv_room, kv_owner, &kv)) return nullptr;
    }
    if (!host_array(a[6], (Py_ssize_t)n, "i", length_room, length_owner, &lengths) ||
        !host_array(a[12], (Py_ssize_t)n, "Q", stride_room, stride_owner, &stride) ||
        !host_array(a[14], (Py_ssize_t)n, "I", rows_room, rows_owner, &rows))
        return nullptr;
    s.kv_base = reinterpret_cast<const void* const*>(kv);
    s.row_stride = stride; s.verified_len = lengths; s.kv_rows = rows;
    if (!address(a[1], &v)) return nullptr;
    s.tok = reinterpret_cast<int32_t*>(v);
    if (!address(a[2], &v)) return nullptr;
    s.life = reinterpret_cast<int8_t*>(v);
    if (!address(a[3], &v)) return nullptr;
    s.buffer = reinterpret_cast<void*>(v);
    if (!address(a[4], &v)) return nullptr;
    s.indices = reinterpret_cast<const int32_t*>(v);
    if (!address(a[8], &v)) return nullptr;
    s.slots = reinterpret_cast<int32_t*>(v);
    if (!address_or_null(a[9], &v)) return nullptr;
    s.hit = reinterpret_cast<uint8_t*>(v);
    if (!address_or_null(a[10], &v)) return nullptr;
    s.miss_count = reinterpret_cast<int32_t*>(v);
    if (!address_or_null(a[11], &v)) return nullptr;
    s.status = reinterpret_cast<uint32_t*>(v);
    if (!stream_handle(a[13], &stream)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = reinterpret_cast<NoAllocFn>(fn)(&s, reinterpret_cast<void*>(stream));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// addr, array, lengths, stream handle; raw stream and device functions, or None
PyObject* set_binding(PyObject*, PyObject* args)
{
    PyObject *addr, *array, *lengths, *stream, *raw, *device;
    if (!PyArg_ParseTuple(args, "OOOOOO", &addr, &array, &lengths, &stream, &raw, &device)) return nullptr;
    Py_INCREF(addr); Py_XSETREF(b_addr, addr);
    Py_INCREF(array); Py_XSETREF(b_array, array);
    Py_INCREF(lengths); Py_XSETREF(b_lengths, lengths);
    Py_INCREF(stream); Py_XSETREF(b_stream, stream);
    const bool both = raw != Py_None && device != Py_None;
    if (both) { Py_INCREF(raw); Py_INCREF(device); }
    Py_XSETREF(b_raw_stream, both ? raw : nullptr);
    Py_XSETREF(b_device, both ? device : nullptr);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"noalloc", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(noalloc)), METH_FASTCALL, nullptr},
    {"set_binding", set_binding, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_python_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__python_calls()
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    PyObject* m = PyModule_Create(&module);
    PyObject* type = m ? PyType_FromSpec(&call_spec) : nullptr;
    if (!type || !s_data_ptr || !s_shape || PyModule_AddObject(m, "Call", type) < 0) return nullptr;
    return m;
}
