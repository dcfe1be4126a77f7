// CPython module `_native`: marshals the arguments of the launching entry points of librac.so.
//
// A decode step is two calls of a few microseconds of GPU work each, and looking at a dozen tensors from Python and passing
// them through ctypes took 7.8 us per call before anything was launched; here that takes 0.6 us (one 4096-wide step of one
// sequence, sender and receiver: 21.7 -> 10.2 us).  Every entry is described by one letter per argument; the C++ type of each
// argument is taken from its declaration in rac.h.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <exception>
#include <type_traits>
#include <utility>

#include "../../include/rac.h"

namespace {

union Slot {
    void *p;
    long long i;
    double d;
};
template <typename T>
T slot_as(const Slot &s) {
    if constexpr (std::is_pointer_v<T>) return static_cast<T>(s.p);
    else if constexpr (std::is_floating_point_v<T>) return static_cast<T>(s.d);
    else return static_cast<T>(s.i);
}
template <typename... A, size_t... I>
int apply(int (*fn)(A...), const Slot *s, std::index_sequence<I...>) {
    return fn(slot_as<A>(s[I])...);
}
template <auto Fn>
struct Thunk;
template <typename... A, int (*Fn)(A...)>
struct Thunk<Fn> {
    static constexpr int count = sizeof...(A);
    static int call(const Slot *s) { return apply(Fn, s, std::index_sequence_for<A...>{}); }
};
constexpr int length(const char *s) {
    int n = 0;
    while (s[n]) n++;
    return n;
}

constexpr int kMaxArgs = 24;
// kinds: c rac_codec_cfg, x rac_index_cfg; tensors or addresses: b bf16, h binary16, f float32, i int32, u bytes, a any type;
// numbers: l integer, B truth value, d float; s stream (None = the current one, an address, or what ctypes takes for one)
struct Entry {
    const char *name, *kinds, *args;   // args: names, comma separated (for messages)
    int count;
    int (*call)(const Slot *);
};
template <auto Fn, int Kinds>
constexpr int checked_count() {
    static_assert(Thunk<Fn>::count == Kinds && Kinds <= kMaxArgs, "one letter per argument");
    return Kinds;
}
#define RAC_ENTRY(fn, kinds, args) {#fn, kinds, args, checked_count<fn, length(kinds)>(), Thunk<fn>::call}
const Entry kEntries[] = {
    RAC_ENTRY(rac_match_spans, "ilillliiials",
              "hist_tok,n_hist,query_tok,n_query,min_ngram,max_hits,ref_row,spans,n_spans,workspace,workspace_bytes,stream"),
    RAC_ENTRY(rac_match_spans_static, "ilillliiis",
              "hist_tok,n_hist,query_tok,n_query,min_ngram,max_hits,ref_row,spans,n_spans,stream"),
    RAC_ENTRY(rac_index_reset, "xals",
              "cfg,index,index_bytes,stream"),
    RAC_ENTRY(rac_index_append, "xalills",
              "cfg,index,index_bytes,hist_tok,n_before,n_after,stream"),
    RAC_ENTRY(rac_index_query_live, "xalillilBiiials",
              "cfg,index,index_bytes,hist_tok,n_hist,first_live,query_tok,n_query,intra,ref_row,spans,n_spans,workspace,workspace_bytes,stream"),
    RAC_ENTRY(rac_index_query, "xalililBiiials",
              "cfg,index,index_bytes,hist_tok,n_hist,query_tok,n_query,intra,ref_row,spans,n_spans,workspace,workspace_bytes,stream"),
    RAC_ENTRY(rac_spans_to_rows, "iilis",
              "spans,n_spans,n_query,ref_row,stream"),
    RAC_ENTRY(rac_spans_to_segments, "iilliis",
              "spans,n_spans,T,max_seg,seg_off,n_seg,stream"),
    RAC_ENTRY(rac_encode, "cblblihhffulalis",
              "cfg,X,T,ref_base,ref_rows,ref_row,ref_gain,ref_bias,step,inv_step,payload,payload_cap,workspace,workspace_bytes,dev_status,stream"),
    RAC_ENTRY(rac_encode_reconstruct, "cblblihhffulbalis",
              "cfg,X,T,ref_base,ref_rows,ref_row,ref_gain,ref_bias,step,inv_step,payload,payload_cap,X_hat,workspace,workspace_bytes,dev_status,stream"),
    RAC_ENTRY(rac_decode_reconstruct, "culblihhfbis",
              "cfg,payload,T,ref_base,ref_rows,ref_row,ref_gain,ref_bias,step,X_hat,dev_status,stream"),
    RAC_ENTRY(rac_sender_reconstruct, "culblihhfbis",
              "cfg,payload,T,ref_base,ref_rows,ref_row,ref_gain,ref_bias,step,X_hat,dev_status,stream"),
    RAC_ENTRY(rac_selftest_bounded_wait, "clalblffalalis",
              "cfg,which,in,T,ref_base,ref_rows,step,inv_step,out,out_cap,workspace,workspace_bytes,dev_status,stream"),
    RAC_ENTRY(rac_split_waves, "illiiis",
              "ref_row,T,first_intra_row,wave1,wave2,wave_count,stream"),
    RAC_ENTRY(rac_encode_reconstruct_list, "cbliiblibliihhffulbalis",
              "cfg,X,T,tok_list,tok_count,ref_base,ref_rows,ref_row,intra_base,intra_rows,coef_seg,seg_of,ref_gain,ref_bias,step,inv_step,payload,payload_cap,X_hat,workspace,workspace_bytes,dev_status,stream"),
    RAC_ENTRY(rac_decode_reconstruct_list, "culiiblibliihhfbis",
              "cfg,payload,T,tok_list,tok_count,ref_base,ref_rows,ref_row,intra_base,intra_rows,coef_seg,seg_of,ref_gain,ref_bias,step,X_hat,dev_status,stream"),
    RAC_ENTRY(rac_fit_segments, "cblblihhiliialis",
              "cfg,X,T,ref_base,ref_rows,ref_row,ref_gain,ref_bias,seg_off,n_seg,coef_seg,seg_of,workspace,workspace_bytes,dev_status,stream"),
    RAC_ENTRY(rac_calibrate_steps, "cblblihhdffalis",
              "cfg,X,T,ref_base,ref_rows,ref_row,ref_gain,ref_bias,clip_sigmas,step,inv_step,workspace,workspace_bytes,dev_status,stream"),
    RAC_ENTRY(rac_calibrate_steps_shared, "cblblihhiidffalis",
              "cfg,X,T,ref_base,ref_rows,ref_row,ref_gain,ref_bias,coef_seg,seg_of,clip_sigmas,step,inv_step,workspace,workspace_bytes,dev_status,stream"),
    RAC_ENTRY(rac_recon_error, "bbllaals",
              "X,X_hat,T,d,out,workspace,workspace_bytes,stream"),
};

PyObject *g_check = nullptr;   // binding._check(name, return code): raises for a non-zero code
PyObject *g_codec_cfg = nullptr, *g_index_cfg = nullptr;   // binding.CodecCfg, binding.IndexCfg: the structs of rac.h
PyObject *g_stream = nullptr;  // binding._stream_address(object) -> int, for streams that are neither None nor an address

const char *arg_name(const Entry &e, int k, char *buf, size_t cap) {
    const char *s = e.args;
    for (; k > 0 && *s; s++) k -= *s == ',';
    size_t n = strcspn(s, ",");
    if (n >= cap) n = cap - 1;
    memcpy(buf, s, n);
    buf[n] = 0;
    return buf;
}
const char *kind_name(char kind) {
    switch (kind) {
        case 'b': return "torch.bfloat16";
        case 'h': return "torch.float16";
        case 'f': return "torch.float32";
        case 'i': return "torch.int32";
    }
    return "torch.uint8 or torch.int8";
}
bool dtype_fits(char kind, c10::ScalarType t) {
    switch (kind) {
        case 'b': return t == c10::ScalarType::BFloat16;
        case 'h': return t == c10::ScalarType::Half;
        case 'f': return t == c10::ScalarType::Float;
        case 'i': return t == c10::ScalarType::Int;
        case 'u': return t == c10::ScalarType::Byte || t == c10::ScalarType::Char;
    }
    return true;
}
bool as_integer(PyObject *o, long long *out) {
    if (PyLong_Check(o)) {
        *out = static_cast<long long>(PyLong_AsUnsignedLongLongMask(o));
    } else {
        PyObject *n = PyNumber_Long(o);
        if (!n) return false;
        *out = static_cast<long long>(PyLong_AsUnsignedLongLongMask(n));
        Py_DECREF(n);
    }
    return !(*out == -1 && PyErr_Occurred());
}

// one argument; false with a Python error set
bool marshal(const Entry &e, int k, PyObject *o, Slot *s) {
    const char kind = e.kinds[k];
    char name[32];
    switch (kind) {
        case 'l':
            return as_integer(o, &s->i);
        case 'B': {
            const int v = PyObject_IsTrue(o);
            s->i = v;
            return v >= 0;
        }
        case 'd': {
            PyObject *n = PyNumber_Float(o);
            if (!n) return false;
            s->d = PyFloat_AS_DOUBLE(n);
            Py_DECREF(n);
            return true;
        }
        case 's':
            if (o == Py_None) {
                s->p = c10::cuda::getCurrentCUDAStream().stream();
                return true;
            }
            if (!PyLong_Check(o)) {      // a torch stream, a c_void_p
                PyObject *n = PyObject_CallOneArg(g_stream, o);
                const bool ok = n && as_integer(n, &s->i);
                Py_XDECREF(n);
                return ok;
            }
            return as_integer(o, &s->i);
        case 'c':
        case 'x': {
            // the struct type itself (or a subclass): any other buffer of its size is none
            if (!PyObject_TypeCheck(o, reinterpret_cast<PyTypeObject *>(kind == 'c' ? g_codec_cfg : g_index_cfg))) {
                PyErr_Format(PyExc_TypeError, "%s: expected %s", arg_name(e, k, name, sizeof name), kind == 'c' ? "a CodecCfg" : "an IndexCfg");
                return false;
            }
            Py_buffer v;
            if (PyObject_GetBuffer(o, &v, PyBUF_SIMPLE) != 0) return false;
            s->p = v.buf;      // the caller holds the object for as long as the address is used
            PyBuffer_Release(&v);
            return true;
        }
    }
    if (o == Py_None) {
        s->p = nullptr;
        return true;
    }
    if (PyLong_Check(o)) return as_integer(o, &s->i);
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s: expected a torch tensor, an address or None", arg_name(e, k, name, sizeof name));
        return false;
    }
    const at::Tensor &t = THPVariable_Unpack(o);
    if (!t.is_cuda()) {
        PyErr_Format(PyExc_ValueError, "%s: must be a CUDA tensor", arg_name(e, k, name, sizeof name));
        return false;
    }
    if (!t.is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s: must be contiguous", arg_name(e, k, name, sizeof name));
        return false;
    }
    if (!dtype_fits(kind, t.scalar_type())) {
        PyErr_Format(PyExc_TypeError, "%s: expected %s, got %s", arg_name(e, k, name, sizeof name), kind_name(kind), c10::toString(t.scalar_type()));
        return false;
    }
    s->p = t.data_ptr();
    return true;
}
bool marshal_all(const Entry &e, PyObject *const *args, Py_ssize_t n, Slot *s) {
    if (!g_check) {
        PyErr_SetString(PyExc_RuntimeError, "the module is set up by binding.load()");
        return false;
    }
    if (n != e.count) {
        PyErr_Format(PyExc_TypeError, "%s: expected %d arguments, got %zd", e.name, e.count, n);
        return false;
    }
    try {
        for (int k = 0; k < e.count; k++)
            if (!marshal(e, k, args[k], &s[k])) return false;
    } catch (const std::exception &x) {
        PyErr_SetString(PyExc_RuntimeError, x.what());
        return false;
    }
    return true;
}
PyObject *finish(const Entry &e, const Slot *s) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = e.call(s);
    Py_END_ALLOW_THREADS
    if (rc == RAC_OK) Py_RETURN_NONE;
    return PyObject_CallFunction(g_check, "si", e.name, rc);
}

// ---- an entry point: call(*args) runs it, prepare(args) marshals them once
struct EntryObject {
    PyObject_HEAD
    const Entry *entry;
    vectorcallfunc vectorcall;
};
struct PreparedObject {
    PyObject_HEAD
    const Entry *entry;
    PyObject *args, *keepalive;   // the marshalled arguments themselves, and what the caller gave
    vectorcallfunc vectorcall;
    Slot slots[kMaxArgs];
};
PyObject *entry_call(PyObject *self, PyObject *const *args, size_t nargsf, PyObject *kwnames) {
    const Entry &e = *reinterpret_cast<EntryObject *>(self)->entry;
    if (kwnames && PyTuple_GET_SIZE(kwnames)) return PyErr_Format(PyExc_TypeError, "%s takes no keyword arguments", e.name);
    Slot s[kMaxArgs];
    if (!marshal_all(e, args, PyVectorcall_NARGS(nargsf), s)) return nullptr;
    return finish(e, s);
}
PyObject *prepared_call(PyObject *self, PyObject *const *, size_t nargsf, PyObject *kwnames) {
    auto *p = reinterpret_cast<PreparedObject *>(self);
    if (PyVectorcall_NARGS(nargsf) || (kwnames && PyTuple_GET_SIZE(kwnames)))
        return PyErr_Format(PyExc_TypeError, "a prepared %s takes no arguments", p->entry->name);
    return finish(*p->entry, p->slots);
}
void prepared_dealloc(PyObject *self) {
    Py_XDECREF(reinterpret_cast<PreparedObject *>(self)->args);
    Py_XDECREF(reinterpret_cast<PreparedObject *>(self)->keepalive);
    Py_TYPE(self)->tp_free(self);
}
PyObject *prepared_keepalive(PyObject *self, void *) { return Py_NewRef(reinterpret_cast<PreparedObject *>(self)->keepalive); }
PyGetSetDef prepared_getset[] = {{"keepalive", prepared_keepalive, nullptr, "the (args, kwargs) of the call", nullptr}, {}};
PyTypeObject EntryType = {PyVarObject_HEAD_INIT(nullptr, 0)};
PyTypeObject PreparedType = {PyVarObject_HEAD_INIT(nullptr, 0)};

// prepare(entry, args, keepalive) -> a function without arguments
PyObject *py_prepare(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != 3 || Py_TYPE(args[0]) != &EntryType || !PyTuple_Check(args[1]))
        return PyErr_Format(PyExc_TypeError, "prepare(entry, args, keepalive)");
    auto *p = PyObject_New(PreparedObject, &PreparedType);
    if (!p) return nullptr;
    p->entry = reinterpret_cast<EntryObject *>(args[0])->entry;
    p->vectorcall = prepared_call;
    p->args = Py_NewRef(args[1]);
    p->keepalive = Py_NewRef(args[2]);
    if (!marshal_all(*p->entry, &PyTuple_GET_ITEM(args[1], 0), PyTuple_GET_SIZE(args[1]), p->slots)) {
        Py_DECREF(p);
        return nullptr;
    }
    return reinterpret_cast<PyObject *>(p);
}
// setup(check, stream_address, CodecCfg, IndexCfg): the callbacks into binding and its struct types
PyObject *py_setup(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != 4 || !PyType_Check(args[2]) || !PyType_Check(args[3]))
        return PyErr_Format(PyExc_TypeError, "setup(check, stream_address, CodecCfg, IndexCfg)");
    Py_XSETREF(g_check, Py_NewRef(args[0]));
    Py_XSETREF(g_stream, Py_NewRef(args[1]));
    Py_XSETREF(g_codec_cfg, Py_NewRef(args[2]));
    Py_XSETREF(g_index_cfg, Py_NewRef(args[3]));
    Py_RETURN_NONE;
}
PyMethodDef methods[] = {
    {"prepare", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_prepare)), METH_FASTCALL, nullptr},
    {"setup", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_setup)), METH_FASTCALL, nullptr},
    {}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    EntryType.tp_name = "_native.Entry";
    EntryType.tp_basicsize = sizeof(EntryObject);
    EntryType.tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL;
    EntryType.tp_vectorcall_offset = offsetof(EntryObject, vectorcall);
    EntryType.tp_call = PyVectorcall_Call;
    PreparedType.tp_name = "_native.Prepared";
    PreparedType.tp_basicsize = sizeof(PreparedObject);
    PreparedType.tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL;
    PreparedType.tp_vectorcall_offset = offsetof(PreparedObject, vectorcall);
    PreparedType.tp_call = PyVectorcall_Call;
    PreparedType.tp_dealloc = prepared_dealloc;
    PreparedType.tp_getset = prepared_getset;
    if (PyType_Ready(&EntryType) < 0 || PyType_Ready(&PreparedType) < 0) return nullptr;
    PyObject *m = PyModule_Create(&module);
    if (!m) return nullptr;
    for (const Entry &e : kEntries) {
        auto *o = PyObject_New(EntryObject, &EntryType);
        if (!o) return nullptr;
        o->entry = &e;
        o->vectorcall = entry_call;
        if (PyModule_AddObject(m, e.name, reinterpret_cast<PyObject *>(o)) < 0) return nullptr;
    }
    return m;
}
