// CPython entry points of the calls a program makes once per kernel or once per model pass.
//
// What a small kernel costs its caller is host time: a ctypes call with marshalled arguments took 4.6 us of the 7.4 us that
// Workload.run took per call, and a chained pass of 108 layers spent 1.9 ms in Python for 0.6 ms of kernels.  These
// functions unpack the Python objects here and call the C ABI with the interpreter lock released.  Everything else
// stays on ctypes.  The library's own entry points are handed over once as addresses (bind), so that this module
// links against nothing.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <algorithm>
#include <vector>
#include "tt.h"

namespace {

typedef tt_status (*RunFn)(tt_workload*, const tt_tensors*, void*);
typedef tt_status (*RunChainFn)(const tt_chain_step*, size_t, void* const*, size_t, size_t*);
RunFn g_run = nullptr;
RunChainFn g_run_chain = nullptr;
PyObject *g_handle_attr = nullptr, *g_kernel_attr = nullptr;   // interned attribute names

PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 2) { PyErr_SetString(PyExc_TypeError, "bind(tt_run, tt_run_chain)"); return nullptr; }
    void* a = PyLong_AsVoidPtr(args[0]);
    void* b = PyLong_AsVoidPtr(args[1]);
    if (PyErr_Occurred()) return nullptr;
    g_run = reinterpret_cast<RunFn>(a);
    g_run_chain = reinterpret_cast<RunChainFn>(b);
    Py_RETURN_NONE;
}

// The tt_tensors inside a ctypes structure.  The bytes belong to the structure, which the caller keeps alive.
bool tensors_of(PyObject* o, tt_tensors* out) {
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return false;
    const bool ok = view.len == (Py_ssize_t)sizeof(tt_tensors);
    if (ok) *out = *static_cast<const tt_tensors*>(view.buf);
    PyBuffer_Release(&view);
    if (!ok) PyErr_SetString(PyExc_TypeError, "a tt_tensors structure is expected");
    return ok;
}

// run(handle, tensors, stream) -> status
PyObject* run(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 3 || !g_run) { PyErr_SetString(PyExc_TypeError, "run(handle, tensors, stream)"); return nullptr; }
    tt_workload* w = static_cast<tt_workload*>(PyLong_AsVoidPtr(args[0]));
    void* stream = PyLong_AsVoidPtr(args[2]);
    tt_tensors t;
    if (PyErr_Occurred() || !tensors_of(args[1], &t)) return nullptr;
    tt_status s;
    Py_BEGIN_ALLOW_THREADS
    s = g_run(w, &t, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)s);
}

bool long_attr(PyObject* o, PyObject* name, void** as_ptr, long* as_long) {
    PyObject* v = PyObject_GetAttr(o, name);
    if (!v) return false;
    if (as_ptr) *as_ptr = v == Py_None ? nullptr : PyLong_AsVoidPtr(v);
    else *as_long = PyLong_AsLong(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}

// The layers of a chain (workloads, steps, tensors, plan: the arguments of workloads.run_chain) as the C ABI takes them.  `held` takes
// over the references made on the way, so that an exception (a container that cannot grow) loses none of them.
struct Chain {
    std::vector<tt_chain_step> steps;
    std::vector<tt_tensors> tensors;
    std::vector<int32_t> waits, node;                     // node: a layer's place among the nodes
    Py_ssize_t nodes = 0;
};
bool read_chain(PyObject* const* args, std::vector<PyObject*>& held, Chain& c) {
    PyObject* seq[4];
    held.reserve(5);
    for (int i = 0; i < 4; ++i) {
        if (!(seq[i] = PySequence_Fast(args[i], "run_chain takes sequences"))) return false;
        held.push_back(seq[i]);
    }
    // (as many nodes as the shortest of the three has)
    c.nodes = std::min({PySequence_Fast_GET_SIZE(seq[1]), PySequence_Fast_GET_SIZE(seq[2]), PySequence_Fast_GET_SIZE(seq[3])});
    const size_t n = (size_t)c.nodes;
    std::vector<int32_t> first_wait, position(n, -1);     // position: node -> its place among the layers
    held.reserve(5 + 2 * n);
    c.tensors.reserve(n); c.steps.reserve(n); c.node.reserve(n); first_wait.reserve(n);
    for (Py_ssize_t i = 0; i < c.nodes; ++i) {
        PyObject* pl = PySequence_Fast_GET_ITEM(seq[3], i);
        if (pl == Py_None) continue;                      // an external tensor
        PyObject* pair = PySequence_Fast(pl, "run_chain: a plan entry is (lane, waits)");
        if (!pair) return false;
        held.push_back(pair);
        if (PySequence_Fast_GET_SIZE(pair) != 2) { PyErr_SetString(PyExc_ValueError, "run_chain: a plan entry is (lane, waits)"); return false; }
        tt_chain_step st{};
        long k = 0;
        void* h = nullptr;
        if (!long_attr(PySequence_Fast_GET_ITEM(seq[1], i), g_kernel_attr, nullptr, &k)) return false;
        if (k < 0 || k >= PySequence_Fast_GET_SIZE(seq[0])) { PyErr_SetString(PyExc_IndexError, "run_chain: no such workload"); return false; }
        if (!long_attr(PySequence_Fast_GET_ITEM(seq[0], k), g_handle_attr, &h, nullptr)) return false;
        st.workload = static_cast<tt_workload*>(h);
        st.lane = (int32_t)PyLong_AsLong(PySequence_Fast_GET_ITEM(pair, 0));
        tt_tensors t;
        if (PyErr_Occurred() || !tensors_of(PySequence_Fast_GET_ITEM(seq[2], i), &t)) return false;
        PyObject* ws = PySequence_Fast(PySequence_Fast_GET_ITEM(pair, 1), "run_chain: waits is a sequence");
        if (!ws) return false;
        held.push_back(ws);
        first_wait.push_back((int32_t)c.waits.size());
        for (Py_ssize_t j = 0; j < PySequence_Fast_GET_SIZE(ws); ++j) {
            const long p = PyLong_AsLong(PySequence_Fast_GET_ITEM(ws, j));
            if (PyErr_Occurred()) return false;
            if (p < 0 || p >= i || position[(size_t)p] < 0) { PyErr_SetString(PyExc_ValueError, "run_chain: a layer waits for a layer in front of it"); return false; }
            c.waits.push_back(position[(size_t)p]);
        }
        st.n_waits = (int32_t)PySequence_Fast_GET_SIZE(ws);
        position[(size_t)i] = (int32_t)c.steps.size();
        c.tensors.push_back(t); c.steps.push_back(st); c.node.push_back((int32_t)i);
    }
    for (size_t i = 0; i < c.steps.size(); ++i) { c.steps[i].tensors = &c.tensors[i]; c.steps[i].waits = c.waits.data() + first_wait[i]; }
    return true;
}

PyObject* enqueue_chain(PyObject* const* args, std::vector<PyObject*>& held) {
    Chain c;
    std::vector<void*> streams;
    if (!read_chain(args, held, c)) return nullptr;
    PyObject* seq = PySequence_Fast(args[4], "run_chain takes sequences");
    if (!seq) return nullptr;
    held.push_back(seq);
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(seq); ++i) {
        streams.push_back(PyLong_AsVoidPtr(PySequence_Fast_GET_ITEM(seq, i)));
        if (PyErr_Occurred()) return nullptr;
    }
    tt_status s = TT_OK;
    size_t at = 0;
    if (!c.steps.empty()) {
        Py_BEGIN_ALLOW_THREADS
        s = g_run_chain(c.steps.data(), c.steps.size(), streams.data(), streams.size(), &at);
        Py_END_ALLOW_THREADS
    }
    return Py_BuildValue("(ii)", (int)s, at < c.node.size() ? (int)c.node[at] : -1);
}

// What a function of the C ABI that takes a chain's layers says about each of them.
PyObject* query_chain(PyObject* const* args, std::vector<PyObject*>& held) {
    typedef tt_status (*QueryFn)(const tt_chain_step*, size_t, size_t*);
    Chain c;
    const QueryFn query = reinterpret_cast<QueryFn>(PyLong_AsVoidPtr(args[4]));
    if (PyErr_Occurred() || !read_chain(args, held, c)) return nullptr;
    std::vector<size_t> of_layer(c.steps.size() + 1, 0);
    const tt_status s = query(c.steps.data(), c.steps.size(), of_layer.data());
    PyObject* values = PyList_New(c.nodes);
    if (!values) return nullptr;
    size_t layer = 0;
    for (Py_ssize_t i = 0; i < c.nodes; ++i) {
        const bool is_layer = layer < c.node.size() && c.node[layer] == (int32_t)i;
        PyObject* v = PyLong_FromSize_t(is_layer ? of_layer[layer] : 0);
        if (!v) { Py_DECREF(values); return nullptr; }
        layer += is_layer;
        PyList_SET_ITEM(values, i, v);
    }
    return Py_BuildValue("(iN)", (int)s, values);
}

PyObject* with_chain(PyObject* (*body)(PyObject* const*, std::vector<PyObject*>&), PyObject* const* args) {
    std::vector<PyObject*> held;
    PyObject* result = nullptr;
    try { result = body(args, held); } catch (...) { PyErr_NoMemory(); }
    for (PyObject* o : held) Py_DECREF(o);
    return result;
}

// run_chain(workloads, steps, tensors, plan, streams) -> (status, index of the step it belongs to)
// The arguments of workloads.run_chain, streams as integers.
PyObject* run_chain(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 5 || !g_run_chain) { PyErr_SetString(PyExc_TypeError, "run_chain(workloads, steps, tensors, plan, streams)"); return nullptr; }
    return with_chain(enqueue_chain, args);
}

// query_chain(workloads, steps, tensors, plan, function) -> (status, a value per node): function is the address of a
// tt_status (steps, n_steps, size_t per step).
PyObject* query(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 5) { PyErr_SetString(PyExc_TypeError, "query_chain(workloads, steps, tensors, plan, function)"); return nullptr; }
    return with_chain(query_chain, args);
}

PyMethodDef kMethods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(bind)), METH_FASTCALL, "bind(tt_run, tt_run_chain): addresses of the library's entry points"},
    {"run", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(run)), METH_FASTCALL, "run(handle, tensors, stream) -> tt_status"},
    {"run_chain", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(run_chain)), METH_FASTCALL,
     "run_chain(workloads, steps, tensors, plan, streams) -> (tt_status, index of the failing node or -1)"},
    {"query_chain", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(query)), METH_FASTCALL,
     "query_chain(workloads, steps, tensors, plan, function) -> (tt_status, a value per node)"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_ttcall", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ttcall(void) {
    g_handle_attr = PyUnicode_InternFromString("address");
    g_kernel_attr = PyUnicode_InternFromString("kernel");
    if (!g_handle_attr || !g_kernel_attr) return nullptr;
    return PyModule_Create(&kModule);
}
