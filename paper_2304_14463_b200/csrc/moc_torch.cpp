// Argument marshalling between torch tensors and the C ABI of libmoc_b200.so, in native code.  A call
// of the evaluator on a small batch takes the GPU a few microseconds; checking five tensors, asking for
// the current stream and allocating three outputs from Python took 15 (n = 20, B = 1024), so that the
// interpreter and not the kernel bounded every small call.  Here the same steps go straight to the
// tensor objects, the caching allocator and the stream of the calling thread.
//
// Every function takes the arguments of the Python function of the same name and returns
//   a tuple / dict-ready tuple of tensors   the call was enqueued;
//   an int                                  the error code of the C ABI (text in moc_last_error);
//   None                                    an argument is not what the fast path takes (wrong type,
//                                           device, layout or size): nothing was called, the Python
//                                           side repeats the checks and raises the matching error.
// The entry points arrive as addresses from the ctypes handle, so that this module and the ctypes
// binding always talk to the same build of the library.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/moc.h"

namespace {

decltype(&moc_eval_batch) f_eval_batch;
decltype(&moc_eval_batch_host) f_eval_batch_host;
decltype(&moc_eval_batch_host16) f_eval_batch_host16;
decltype(&moc_mem_profile) f_mem_profile;
decltype(&moc_check_intervals) f_check_intervals_filled;   // writes the whole rows, -1 behind the sequences
decltype(&moc_cache_build) f_cache_build;
decltype(&moc_eval_edits) f_eval_edits;
decltype(&moc_search_run) f_search_run;
decltype(&moc_search_state) f_search_state_filled;   // writes the whole rows, zeros behind the sequences
decltype(&moc_search_info) f_search_info;

PyObject* s_value;   // interned "value" (the pointer in a ctypes.c_void_p)

// Handle: a ctypes.c_void_p.  false: not one (or null).
bool handle_of(PyObject* o, void** out) {
    PyObject* v = PyObject_GetAttr(o, s_value);
    if (!v) {
        PyErr_Clear();
        return false;
    }
    const bool ok = PyLong_Check(v);
    *out = ok ? PyLong_AsVoidPtr(v) : nullptr;
    Py_DECREF(v);
    if (PyErr_Occurred()) PyErr_Clear();
    return *out != nullptr;
}
bool int_of(PyObject* o, int64_t* out) {
    if (!PyLong_Check(o)) return false;
    *out = (int64_t)PyLong_AsUnsignedLongLongMask(o);   // wraps like a ctypes.c_int64
    if (PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    return true;
}
// A contiguous CUDA tensor of the given type; null otherwise.
const at::Tensor* dev_tensor(PyObject* o, at::ScalarType t) {
    if (!THPVariable_Check(o)) return nullptr;
    const at::Tensor& x = THPVariable_Unpack(o);
    return x.is_cuda() && x.scalar_type() == t && x.is_contiguous() ? &x : nullptr;
}
template <typename T>
T* ptr(const at::Tensor& t) {
    return static_cast<T*>(t.data_ptr());
}
at::Tensor empty(at::IntArrayRef size, at::ScalarType t, at::Device d) {
    return at::Tensor(at::detail::empty_cuda(size, t, d, std::nullopt));
}
void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

// Output argument: None allocates `count` entries on `d`, a tensor is used as it is.  false: unusable.
bool output(PyObject* o, at::ScalarType t, int64_t count, at::Device d, at::Tensor* out) {
    if (o == Py_None) {
        *out = empty({count}, t, d);
        return true;
    }
    const at::Tensor* x = dev_tensor(o, t);
    if (!x || x->numel() < count || x->device() != d) return false;
    *out = *x;
    return true;
}

template <typename... T>
PyObject* tuple_of(const T&... t) {
    PyObject* r = PyTuple_New(sizeof...(T));
    if (!r) return nullptr;
    Py_ssize_t i = 0;
    bool ok = true;
    (([&] {
         PyObject* w = t.defined() ? THPVariable_Wrap(t) : Py_NewRef(Py_None);
         ok = ok && w != nullptr;
         PyTuple_SET_ITEM(r, i++, w);
     }()), ...);
    if (!ok) {
        Py_DECREF(r);
        return nullptr;
    }
    return r;
}

// Runs `call` without the interpreter lock.
template <typename F>
int unlocked(F&& call) {
    PyThreadState* st = PyEval_SaveThread();
    const int rc = call();
    PyEval_RestoreThread(st);
    return rc;
}

// C++ exceptions (an allocation that failed) become Python's.
template <typename F>
PyObject* guarded(F&& body) {
    try {
        return body();
    } catch (const c10::OutOfMemoryError& e) {
        PyObject* torch_mod = PyImport_ImportModule("torch");
        PyObject* type = torch_mod ? PyObject_GetAttrString(torch_mod, "OutOfMemoryError") : nullptr;
        if (type) PyErr_SetString(type, e.what_without_backtrace());
        Py_XDECREF(type);
        Py_XDECREF(torch_mod);
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

#define MOC_NONE_IF(cond) \
    if (cond) return Py_NewRef(Py_None)

// eval_batch(g, seqs, lens, M, out_peak, out_dur, out_feasible)
PyObject* py_eval_batch(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* g;
        int64_t M;
        MOC_NONE_IF(na != 7 || !handle_of(a[0], &g) || !int_of(a[3], &M));
        const at::Tensor *seqs = dev_tensor(a[1], at::kInt), *lens = dev_tensor(a[2], at::kInt);
        MOC_NONE_IF(!seqs || !lens || lens->numel() > INT32_MAX);
        const int64_t B = lens->numel();
        const at::Device d = lens->device();
        at::Tensor pk, du, st;
        MOC_NONE_IF(!output(a[4], at::kLong, B, d, &pk) || !output(a[5], at::kLong, B, d, &du) || !output(a[6], at::kInt, B, d, &st));
        void* cs = stream();
        const int rc = unlocked([&] {
            return f_eval_batch((const moc_graph*)g, ptr<int32_t>(*seqs), ptr<int32_t>(*lens), (int32_t)B, M, ptr<int64_t>(pk),
                                ptr<int64_t>(du), ptr<int32_t>(st), cs);
        });
        if (rc != MOC_OK) return PyLong_FromLong(rc);
        return tuple_of(pk, du, st);
    });
}

// eval_batch_host(g, seqs, lens, M, out_peak, out_dur, out_feasible, bits): CPU tensors; returns its outputs
PyObject* py_eval_batch_host(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* g;
        int64_t M, bits;
        MOC_NONE_IF(na != 8 || !handle_of(a[0], &g) || !int_of(a[3], &M) || !int_of(a[7], &bits));
        const at::ScalarType want[5] = {bits == 16 ? at::kUInt16 : at::kInt, at::kInt, at::kLong, at::kLong, at::kInt};
        const int where[5] = {1, 2, 4, 5, 6};
        const at::Tensor* t[5];
        for (int k = 0; k < 5; ++k) {
            MOC_NONE_IF(!THPVariable_Check(a[where[k]]));
            t[k] = &THPVariable_Unpack(a[where[k]]);
            MOC_NONE_IF(!t[k]->is_cpu() || t[k]->scalar_type() != want[k] || !t[k]->is_contiguous() || t[k]->dim() < 1);
        }
        const int64_t B = t[1]->size(0), n_steps = t[0]->size(0);
        MOC_NONE_IF(B > INT32_MAX);
        void* cs = stream();
        const int rc = unlocked([&] {
            return bits == 16 ? f_eval_batch_host16((const moc_graph*)g, ptr<uint16_t>(*t[0]), n_steps, ptr<int32_t>(*t[1]), (int32_t)B, M,
                                                    ptr<int64_t>(*t[2]), ptr<int64_t>(*t[3]), ptr<int32_t>(*t[4]), cs)
                              : f_eval_batch_host((const moc_graph*)g, ptr<int32_t>(*t[0]), n_steps, ptr<int32_t>(*t[1]), (int32_t)B, M,
                                                  ptr<int64_t>(*t[2]), ptr<int64_t>(*t[3]), ptr<int32_t>(*t[4]), cs);
        });
        if (rc != MOC_OK) return PyLong_FromLong(rc);
        return tuple_of(*t[2], *t[3], *t[4]);
    });
}

// mem_profile(g, seq, want_free)
PyObject* py_mem_profile(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* g;
        MOC_NONE_IF(na != 3 || !handle_of(a[0], &g));
        const at::Tensor* seq = dev_tensor(a[1], at::kInt);
        const int want = PyObject_IsTrue(a[2]);
        if (want < 0) return nullptr;
        MOC_NONE_IF(!seq || seq->numel() > INT32_MAX);
        const int64_t T = seq->numel();
        const at::Device d = seq->device();
        at::Tensor prof = empty({T}, at::kLong, d), fre, st;
        if (want) fre = empty({T}, at::kInt, d);
        st = empty({1}, at::kInt, d);
        void* cs = stream();
        const int rc = unlocked([&] {
            return f_mem_profile((const moc_graph*)g, ptr<int32_t>(*seq), (int32_t)T, ptr<int64_t>(prof), want ? ptr<int32_t>(fre) : nullptr,
                                 ptr<int32_t>(st), cs);
        });
        if (rc != MOC_OK) return PyLong_FromLong(rc);
        return tuple_of(prof, fre, st);
    });
}

// cache_build(cache, seqs, lens, M)
PyObject* py_cache_build(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* c;
        int64_t M;
        MOC_NONE_IF(na != 4 || !handle_of(a[0], &c) || !int_of(a[3], &M));
        const at::Tensor *seqs = dev_tensor(a[1], at::kInt), *lens = dev_tensor(a[2], at::kInt);
        MOC_NONE_IF(!seqs || !lens || lens->numel() > INT32_MAX);
        const int64_t P = lens->numel();
        const at::Device d = lens->device();
        at::Tensor pk = empty({P}, at::kLong, d), du = empty({P}, at::kLong, d), st = empty({P}, at::kInt, d);
        void* cs = stream();
        const int rc = unlocked([&] {
            return f_cache_build((moc_cache*)c, ptr<int32_t>(*seqs), ptr<int32_t>(*lens), (int32_t)P, M, ptr<int64_t>(pk), ptr<int64_t>(du),
                                 ptr<int32_t>(st), cs);
        });
        if (rc != MOC_OK) return PyLong_FromLong(rc);
        return tuple_of(pk, du, st);
    });
}

// eval_edits(cache, parent, op, q, j, M)
PyObject* py_eval_edits(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* c;
        int64_t M;
        MOC_NONE_IF(na != 6 || !handle_of(a[0], &c) || !int_of(a[5], &M));
        const at::Tensor* e[4];
        for (int k = 0; k < 4; ++k) {
            e[k] = dev_tensor(a[1 + k], at::kInt);
            MOC_NONE_IF(!e[k]);
        }
        const int64_t B = e[0]->numel();
        MOC_NONE_IF(B > INT32_MAX);
        const at::Device d = e[0]->device();
        at::Tensor pk = empty({B}, at::kLong, d), du = empty({B}, at::kLong, d), st = empty({B}, at::kInt, d);
        void* cs = stream();
        const int rc = unlocked([&] {
            return f_eval_edits((const moc_cache*)c, ptr<int32_t>(*e[0]), ptr<int32_t>(*e[1]), ptr<int32_t>(*e[2]), ptr<int32_t>(*e[3]),
                                (int32_t)B, M, ptr<int64_t>(pk), ptr<int64_t>(du), ptr<int32_t>(st), nullptr, cs);
        });
        if (rc != MOC_OK) return PyLong_FromLong(rc);
        return tuple_of(pk, du, st);
    });
}

// check_intervals(g, s, e, a, M, D, topo_index, want_seqs) -> (mask, peak, dur, seqs, lens)
PyObject* py_check_intervals(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* g;
        int64_t M, D;
        MOC_NONE_IF(na != 8 || !handle_of(a[0], &g) || !int_of(a[4], &M) || !int_of(a[5], &D));
        const at::Tensor *s = dev_tensor(a[1], at::kInt), *e = dev_tensor(a[2], at::kInt), *f = dev_tensor(a[3], at::kInt), *topo = nullptr;
        MOC_NONE_IF(!s || !e || !f || s->dim() != 3 || s->size(0) > INT32_MAX);
        if (a[6] != Py_None) {
            topo = dev_tensor(a[6], at::kInt);
            MOC_NONE_IF(!topo);
        }
        const int want = PyObject_IsTrue(a[7]);
        if (want < 0) return nullptr;
        const int64_t B = s->size(0), K = s->size(1) * s->size(2);
        const at::Device d = s->device();
        at::Tensor pk = empty({B}, at::kLong, d), du = empty({B}, at::kLong, d), mask = empty({B}, at::kInt, d), seqs, lens;
        if (want) {
            seqs = empty({B, K}, at::kInt, d);
            lens = empty({B}, at::kInt, d);
        }
        void* cs = stream();
        const int rc = unlocked([&] {
            return f_check_intervals_filled((const moc_graph*)g, ptr<int32_t>(*s), ptr<int32_t>(*e), ptr<int32_t>(*f), (int32_t)B, D,
                                     topo ? ptr<int32_t>(*topo) : nullptr, M, ptr<int64_t>(pk), ptr<int64_t>(du), ptr<int32_t>(mask),
                                     want ? ptr<int32_t>(seqs) : nullptr, want ? ptr<int32_t>(lens) : nullptr, cs);
        });
        if (rc != MOC_OK) return PyLong_FromLong(rc);
        return tuple_of(mask, pk, du, seqs, lens);
    });
}

// search_run(search, n_generations)
PyObject* py_search_run(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* s;
        int64_t k;
        MOC_NONE_IF(na != 2 || !handle_of(a[0], &s) || !int_of(a[1], &k));
        void* cs = stream();
        const int rc = unlocked([&] { return f_search_run((moc_search*)s, (int32_t)k, cs); });
        return PyLong_FromLong(rc);
    });
}

// search_state(search, want_rows) -> (rows, lens, peak, dur, status, accepted)
PyObject* py_search_state(PyObject*, PyObject* const* a, Py_ssize_t na) {
    return guarded([&]() -> PyObject* {
        void* s;
        MOC_NONE_IF(na != 2 || !handle_of(a[0], &s));
        const int want = PyObject_IsTrue(a[1]);
        if (want < 0) return nullptr;
        int32_t P = 0, stride = 0;
        const int ri = f_search_info((const moc_search*)s, &P, &stride, nullptr);
        if (ri != MOC_OK) return PyLong_FromLong(ri);
        void* cs = stream();
        const at::Device d(at::kCUDA, c10::cuda::current_device());
        at::Tensor rows, lens = empty({P}, at::kInt, d), pk = empty({P}, at::kLong, d), du = empty({P}, at::kLong, d),
                         st = empty({P}, at::kInt, d), acc = empty({P}, at::kInt, d);
        if (want) {
            rows = empty({P, stride}, at::kInt, d);
        }
        const int rc = unlocked([&] {
            return f_search_state_filled((const moc_search*)s, want ? ptr<int32_t>(rows) : nullptr, ptr<int32_t>(lens), ptr<int64_t>(pk),
                                  ptr<int64_t>(du), ptr<int32_t>(st), ptr<int32_t>(acc), cs);
        });
        if (rc != MOC_OK) return PyLong_FromLong(rc);
        return tuple_of(rows, lens, pk, du, st, acc);
    });
}

// bind({entry point: address})
PyObject* py_bind(PyObject*, PyObject* d) {
    auto get = [&](const char* name) -> void* {
        PyObject* v = PyDict_GetItemString(d, name);
        if (!v) {
            PyErr_Format(PyExc_KeyError, "%s", name);
            return nullptr;
        }
        return PyLong_AsVoidPtr(v);
    };
#define MOC_BIND(fn)                               \
    f_##fn = (decltype(f_##fn))get("moc_" #fn);    \
    if (PyErr_Occurred()) return nullptr
    MOC_BIND(eval_batch);
    MOC_BIND(eval_batch_host);
    MOC_BIND(eval_batch_host16);
    MOC_BIND(mem_profile);
    MOC_BIND(check_intervals_filled);
    MOC_BIND(cache_build);
    MOC_BIND(eval_edits);
    MOC_BIND(search_run);
    MOC_BIND(search_state_filled);
    MOC_BIND(search_info);
#undef MOC_BIND
    Py_RETURN_NONE;
}

#define MOC_FAST(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {MOC_FAST(eval_batch),      MOC_FAST(eval_batch_host), MOC_FAST(mem_profile), MOC_FAST(cache_build),  MOC_FAST(eval_edits),
                         MOC_FAST(check_intervals), MOC_FAST(search_run),  MOC_FAST(search_state), {"bind", py_bind, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_moc_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__moc_torch(void) {
    s_value = PyUnicode_InternFromString("value");
    return s_value ? PyModule_Create(&module) : nullptr;
}
