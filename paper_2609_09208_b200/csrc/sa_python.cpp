// Python side of the calls that a decode loop makes once per layer: argument marshalling only.
//
// A decode call on a short context takes the GPU 4 - 6 us, less than ctypes and torch.cuda.current_stream() took to
// prepare it (7 of 12.5 us a call).  These functions take the same objects — the ctypes structures of the C header
// through the buffer protocol, torch tensors through data_ptr() — and return the library's status; each tensor costs one
// method call and the stream two plain C++ calls into torch.  The interpreter lock is released around the library call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/sa.h"

namespace {

PyObject *g_data_ptr, *g_nbytes, *g_get_device, *g_get_stream;

struct Args {
    PyObject* const* v;
    Py_ssize_t n, i = 0;
    bool bad = false;

    PyObject* next() {
        if (i >= n) {
            bad = true;
            PyErr_SetString(PyExc_TypeError, "too few arguments");
            return nullptr;
        }
        return v[i++];
    }
    // pointer of a ctypes structure (it outlives the call: the caller holds it)
    template <typename T>
    const T* structure() {
        PyObject* o = bad ? nullptr : next();
        Py_buffer b;
        if (!o || PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) {
            bad = true;
            return nullptr;
        }
        const bool fits = b.len == (Py_ssize_t)sizeof(T);
        const T* p = static_cast<const T*>(b.buf);
        PyBuffer_Release(&b);
        if (!fits) {
            bad = true;
            PyErr_SetString(PyExc_TypeError, "not the structure of the C header");
        }
        return p;
    }
    unsigned long long number_of(PyObject* o) {
        if (!o) {
            bad = true;
            return 0;
        }
        const unsigned long long x = PyLong_AsUnsignedLongLong(o);
        if (x == (unsigned long long)-1 && PyErr_Occurred()) bad = true;
        Py_DECREF(o);
        return x;
    }
    // address of a tensor; None is NULL
    template <typename T>
    T* tensor() {
        PyObject* o = bad ? nullptr : next();
        if (!o || o == Py_None) return nullptr;
        return reinterpret_cast<T*>(number_of(PyObject_CallMethodNoArgs(o, g_data_ptr)));
    }
    void* tensor_and_bytes(size_t* bytes) {
        PyObject* o = bad ? nullptr : next();
        *bytes = 0;
        if (!o) return nullptr;
        *bytes = (size_t)number_of(PyObject_GetAttr(o, g_nbytes));
        return bad ? nullptr : reinterpret_cast<void*>(number_of(PyObject_CallMethodNoArgs(o, g_data_ptr)));
    }
    int integer() {
        PyObject* o = bad ? nullptr : next();
        const long x = o ? PyLong_AsLong(o) : -1;
        if (o && x == -1 && PyErr_Occurred()) bad = true;
        return (int)x;
    }
    // torch's current stream on the current device
    sa_stream stream() {
        if (bad) return nullptr;
        PyObject* dev = PyObject_CallNoArgs(g_get_device);
        if (!dev) {
            bad = true;
            return nullptr;
        }
        PyObject* s = PyObject_CallOneArg(g_get_stream, dev);
        Py_DECREF(dev);
        return reinterpret_cast<sa_stream>(number_of(s));
    }
};

// CALL: an expression of type sa_status over what was unpacked
#define SA_RETURN(CALL)                 \
    do {                                \
        if (a.bad) return nullptr;      \
        sa_status st;                   \
        Py_BEGIN_ALLOW_THREADS          \
        st = (CALL);                    \
        Py_END_ALLOW_THREADS            \
        return PyLong_FromLong(st);     \
    } while (0)

// (cfg, cache, Q, O, workspace, dbg_scores, stages)
PyObject* decode_attention(PyObject*, PyObject* const* v, Py_ssize_t n) {
    Args a{v, n};
    const sa_config* cfg = a.structure<sa_config>();
    const sa_cache* cache = a.structure<sa_cache>();
    const uint16_t* Q = a.tensor<uint16_t>();
    float* O = a.tensor<float>();
    size_t bytes;
    void* ws = a.tensor_and_bytes(&bytes);
    int32_t* dbg = a.tensor<int32_t>();
    const int stages = a.integer();
    const sa_stream s = a.stream();
    SA_RETURN(sa_decode_attention_stages(cfg, cache, Q, O, ws, bytes, dbg, stages, s));
}

// (cfg, cache, Q, O, workspace, stages)
PyObject* decode_attention_fp16(PyObject*, PyObject* const* v, Py_ssize_t n) {
    Args a{v, n};
    const sa_config* cfg = a.structure<sa_config>();
    const sa_cache* cache = a.structure<sa_cache>();
    const uint16_t* Q = a.tensor<uint16_t>();
    float* O = a.tensor<float>();
    size_t bytes;
    void* ws = a.tensor_and_bytes(&bytes);
    const int stages = a.integer();
    const sa_stream s = a.stream();
    SA_RETURN(sa_decode_attention_fp16_stages(cfg, cache, Q, O, ws, bytes, stages, s));
}

// (cfg, cache, Q, K_new, V_new, O, workspace)
PyObject* decode_step(PyObject*, PyObject* const* v, Py_ssize_t n) {
    Args a{v, n};
    const sa_config* cfg = a.structure<sa_config>();
    const sa_cache* cache = a.structure<sa_cache>();
    const uint16_t* Q = a.tensor<uint16_t>();
    const uint16_t* K = a.tensor<uint16_t>();
    const uint16_t* V = a.tensor<uint16_t>();
    float* O = a.tensor<float>();
    size_t bytes;
    void* ws = a.tensor_and_bytes(&bytes);
    const sa_stream s = a.stream();
    SA_RETURN(sa_decode_step(cfg, cache, Q, K, V, O, ws, bytes, s));
}

// (cfg, cache, Q, K_new, V_new, O, staging, workspace), the four in the middle on the host
PyObject* decode_step_host(PyObject*, PyObject* const* v, Py_ssize_t n) {
    Args a{v, n};
    const sa_config* cfg = a.structure<sa_config>();
    const sa_cache* cache = a.structure<sa_cache>();
    const uint16_t* Q = a.tensor<uint16_t>();
    const uint16_t* K = a.tensor<uint16_t>();
    const uint16_t* V = a.tensor<uint16_t>();
    float* O = a.tensor<float>();
    size_t sbytes, bytes;
    void* staging = a.tensor_and_bytes(&sbytes);
    void* ws = a.tensor_and_bytes(&bytes);
    const sa_stream s = a.stream();
    SA_RETURN(sa_decode_step_host(cfg, cache, Q, K, V, O, staging, sbytes, ws, bytes, s));
}

// (cfg, cache, K_new, V_new, bump_lens)
PyObject* append_kv(PyObject*, PyObject* const* v, Py_ssize_t n) {
    Args a{v, n};
    const sa_config* cfg = a.structure<sa_config>();
    const sa_cache* cache = a.structure<sa_cache>();
    const uint16_t* K = a.tensor<uint16_t>();
    const uint16_t* V = a.tensor<uint16_t>();
    const int bump = a.integer();
    const sa_stream s = a.stream();
    SA_RETURN(sa_append_kv(cfg, cache, K, V, bump, s));
}

// (cfg, cache, K, V, cu_lens): cu_lens a contiguous host array of at least batch + 1 64-bit integers, which the library
// reads on the host
PyObject* fill_kv(PyObject*, PyObject* const* v, Py_ssize_t n) {
    Args a{v, n};
    const sa_config* cfg = a.structure<sa_config>();
    const sa_cache* cache = a.structure<sa_cache>();
    const uint16_t* K = a.tensor<uint16_t>();
    const uint16_t* V = a.tensor<uint16_t>();
    PyObject* o = a.bad ? nullptr : a.next();
    Py_buffer cu;
    if (a.bad || PyObject_GetBuffer(o, &cu, PyBUF_SIMPLE) != 0) return nullptr;
    if (cu.len / (Py_ssize_t)sizeof(int64_t) <= (Py_ssize_t)cache->batch) {
        a.bad = true;
        PyErr_Format(PyExc_ValueError, "cu_lens holds %zd bytes, not the batch + 1 = %zd numbers of 8", cu.len, (Py_ssize_t)cache->batch + 1);
    }
    const sa_stream s = a.stream();
    if (a.bad) {
        PyBuffer_Release(&cu);
        return nullptr;
    }
    sa_status st;
    Py_BEGIN_ALLOW_THREADS
    st = sa_fill_kv(cfg, cache, K, V, static_cast<const int64_t*>(cu.buf), s);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&cu);
    return PyLong_FromLong(st);
}

PyMethodDef kMethods[] = {
    {"fill_kv", (PyCFunction)(void (*)(void))fill_kv, METH_FASTCALL, nullptr},
    {"decode_attention", (PyCFunction)(void (*)(void))decode_attention, METH_FASTCALL, nullptr},
    {"decode_attention_fp16", (PyCFunction)(void (*)(void))decode_attention_fp16, METH_FASTCALL, nullptr},
    {"decode_step", (PyCFunction)(void (*)(void))decode_step, METH_FASTCALL, nullptr},
    {"decode_step_host", (PyCFunction)(void (*)(void))decode_step_host, METH_FASTCALL, nullptr},
    {"append_kv", (PyCFunction)(void (*)(void))append_kv, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    PyObject* c = PyImport_ImportModule("torch._C");
    if (!c) return nullptr;
    g_get_device = PyObject_GetAttrString(c, "_cuda_getDevice");
    g_get_stream = PyObject_GetAttrString(c, "_cuda_getCurrentRawStream");
    Py_DECREF(c);
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_nbytes = PyUnicode_InternFromString("nbytes");
    if (!g_get_device || !g_get_stream || !g_data_ptr || !g_nbytes) return nullptr;
    return PyModule_Create(&kModule);
}
