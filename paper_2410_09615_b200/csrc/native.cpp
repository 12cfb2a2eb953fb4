// Call path of the entry points from Python: argument checks, the output tensors, the current stream and
// the call into libslim, without interpreted code in between.  A small-batch call takes the GPU about as long as
// one launch takes the host, so the path from the interpreter to the launch is part of its time: through ctypes and
// per-argument Python checks a call took the host 22-23 us, this way 4-8 (three to four of them the launch).
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime.h>
#include <algorithm>
#include <cstdint>
#include <mutex>

namespace {

using FwdFn = int (*)(const void*, int, const uint8_t*, const uint8_t*, float, const void*, const void*, int, int, int, void*, void*,
                      size_t, uint32_t*, void*, int);
using TiledFn = int (*)(const void*, int, const void*, int, float, const void*, const void*, int, int, int, void*, void*, size_t,
                        uint32_t*, void*);
using QFn = int (*)(const void*, int, const uint8_t*, const uint8_t*, float, const uint8_t*, const void*, const uint8_t*, const void*,
                    int, int, int, void*, void*, size_t, uint32_t*, void*);
using BytesFn = size_t (*)(int, int, int);
using PackFn = int (*)(const int8_t*, const uint8_t*, int, int, uint8_t*, uint8_t*, uint32_t*, void*);
using QuantFn = int (*)(const float*, int, int, int8_t*, float*, void*, size_t, uint32_t*, void*);
using QuantBytesFn = size_t (*)(int, int);
using MaskFn = int (*)(const int8_t*, const float*, int, int, uint8_t*, uint32_t*, void*);
using AdapterFn = int (*)(const void*, int, int, uint8_t*, void*, void*);
using TextFn = const char* (*)(int);

FwdFn g_fwd = nullptr;
TiledFn g_tiled = nullptr;
QFn g_q = nullptr;
BytesFn g_tiled_bytes = nullptr;
PackFn g_pack = nullptr;
QuantFn g_quant = nullptr;
QuantBytesFn g_quant_bytes = nullptr;
MaskFn g_mask = nullptr;
AdapterFn g_pack_adapter = nullptr;
TextFn g_text = nullptr;
PyObject* g_error = nullptr;            // SlimError(code, where, text)

// A contiguous CUDA tensor of the given type, or a TypeError.
const at::Tensor* device_tensor(PyObject* o, at::ScalarType type, const char* name, const char* type_name) {
    if (THPVariable_Check(o)) {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (t.is_cuda() && t.scalar_type() == type && t.is_contiguous()) return &t;
    }
    PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor of %s", name, type_name);
    return nullptr;
}
const at::Tensor* bf16_tensor(PyObject* o, const char* name) { return device_tensor(o, at::kBFloat16, name, "torch.bfloat16"); }
const at::Tensor* u8_tensor(PyObject* o, const char* name) { return device_tensor(o, at::kByte, name, "torch.uint8"); }

// Any tensor's address, NULL for None (outputs, workspace and status).
bool address(PyObject* o, const char* name, void** p, size_t* bytes = nullptr) {
    *p = nullptr;
    if (o == Py_None) return true;
    if (!THPVariable_Check(o)) { PyErr_Format(PyExc_TypeError, "%s: expected a tensor", name); return false; }
    const at::Tensor& t = THPVariable_Unpack(o);
    *p = t.data_ptr();
    if (bytes) *bytes = (size_t)t.numel();
    return true;
}

bool rank2(const at::Tensor* t, const char* name) {
    if (t->dim() == 2) return true;
    PyErr_Format(PyExc_ValueError, "%s: expected a matrix", name);
    return false;
}

PyObject* output(PyObject* given, int64_t b, int64_t d_out, const at::Tensor& like, void** p) {
    if (given != Py_None) {
        if (!address(given, "Y", p)) return nullptr;
        Py_INCREF(given);
        return given;
    }
    at::Tensor made = at::detail::empty_cuda({b, d_out}, at::kBFloat16, like.device(), std::nullopt);
    *p = made.data_ptr();
    return THPVariable_Wrap(std::move(made));
}

PyObject* finish(int code, PyObject* y, const char* where) {
    if (code == 0) return y;
    Py_XDECREF(y);
    PyObject* e = PyObject_CallFunction(g_error, "iss", code, where, g_text(code));
    if (e) { PyErr_SetObject(g_error, e); Py_DECREF(e); }
    return nullptr;
}

bool bound(Py_ssize_t given, Py_ssize_t wanted) {
    if (!g_fwd) { PyErr_SetString(PyExc_RuntimeError, "bind() has not been called"); return false; }
    if (given == wanted) return true;
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return false;
}

// bf16 adapters L [d_out, r], R [r, d_in]; None: r = 0.
bool adapters(PyObject* oL, PyObject* oR, int64_t d_out, int64_t d_in, void** L, void** R, int64_t* r) {
    *L = *R = nullptr; *r = 0;
    if (oL == Py_None) return true;
    if (!THPVariable_Check(oL)) return bf16_tensor(oL, "L") != nullptr;
    const at::Tensor& l = THPVariable_Unpack(oL);
    if (!rank2(&l, "L")) return false;
    *r = l.size(1);
    if (*r == 0) return true;
    const at::Tensor *pl = bf16_tensor(oL, "L"), *pr = pl ? bf16_tensor(oR, "R") : nullptr;
    if (!pr) return false;
    if (pl->size(0) != d_out || pr->dim() != 2 || pr->size(0) != *r || pr->size(1) != d_in) {
        PyErr_SetString(PyExc_ValueError, "adapter shapes do not match the weight");
        return false;
    }
    *L = pl->data_ptr(); *R = pr->data_ptr();
    return true;
}

// A call into the library, with the interpreter free for other threads: a launch waits where the stream's queue is full.
template <typename F, typename... A>
int unlocked(F f, A... args) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f(args...);
    Py_END_ALLOW_THREADS
    return rc;
}

// linear_fwd(X, vals, meta, s, L, R, Y, workspace, status, kernel)
PyObject* linear_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!bound(n, 10)) return nullptr;
    const at::Tensor *X = bf16_tensor(a[0], "X"), *v = X ? u8_tensor(a[1], "vals") : nullptr, *m = v ? u8_tensor(a[2], "meta") : nullptr;
    if (!m || !rank2(X, "X") || !rank2(v, "vals") || !rank2(m, "meta")) return nullptr;
    const double s = PyFloat_AsDouble(a[3]);
    const long kernel = PyLong_AsLong(a[9]);
    if (PyErr_Occurred()) return nullptr;
    const int64_t b = X->size(0), d_in = X->size(1), d_out = v->size(0);
    void *L, *R, *Y, *ws, *status;
    int64_t r;
    if (!adapters(a[4], a[5], d_out, d_in, &L, &R, &r)) return nullptr;
    if (v->size(1) * 4 != d_in || m->size(0) != d_out || m->size(1) != d_in / 8) {
        PyErr_SetString(PyExc_ValueError, "packed weight does not match X");
        return nullptr;
    }
    size_t ws_bytes = 0;
    if (!address(a[7], "workspace", &ws, &ws_bytes) || !address(a[8], "status", &status)) return nullptr;
    PyObject* y = output(a[6], b, d_out, *X, &Y);
    if (!y) return nullptr;
    void* stream = c10::cuda::getCurrentCUDAStream().stream();
    const int rc = unlocked(g_fwd, X->data_ptr(), (int)b, (const uint8_t*)v->data_ptr(), (const uint8_t*)m->data_ptr(), (float)s, L, R, (int)r,
                            (int)d_out, (int)d_in, Y, ws, ws_bytes, (uint32_t*)status, stream, (int)kernel);
    return finish(rc, y, "slim_linear_fwd");
    END_HANDLE_TH_ERRORS
}

// linear_fwd_tiled(X, tiled, d_out, s, L, R, Y, workspace, status, layout)
PyObject* linear_fwd_tiled(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!bound(n, 10)) return nullptr;
    const at::Tensor *X = bf16_tensor(a[0], "X"), *t = X ? u8_tensor(a[1], "tiled") : nullptr;
    if (!t || !rank2(X, "X")) return nullptr;
    const long d_out = PyLong_AsLong(a[2]);
    const double s = PyFloat_AsDouble(a[3]);
    const long layout = PyLong_AsLong(a[9]);
    if (PyErr_Occurred()) return nullptr;
    const int64_t b = X->size(0), d_in = X->size(1);
    void *L, *R, *Y, *ws, *status;
    int64_t r;
    if (!adapters(a[4], a[5], d_out, d_in, &L, &R, &r)) return nullptr;
    if ((size_t)t->numel() != g_tiled_bytes((int)d_out, (int)d_in, (int)layout)) {
        PyErr_SetString(PyExc_ValueError, "tiled weight does not match the shape");
        return nullptr;
    }
    size_t ws_bytes = 0;
    if (!address(a[7], "workspace", &ws, &ws_bytes) || !address(a[8], "status", &status)) return nullptr;
    PyObject* y = output(a[6], b, d_out, *X, &Y);
    if (!y) return nullptr;
    void* stream = c10::cuda::getCurrentCUDAStream().stream();
    const int rc = unlocked(g_tiled, X->data_ptr(), (int)b, t->data_ptr(), (int)layout, (float)s, L, R, (int)r, (int)d_out, (int)d_in, Y, ws,
                            ws_bytes, (uint32_t*)status, stream);
    return finish(rc, y, "slim_linear_fwd_tiled");
    END_HANDLE_TH_ERRORS
}

// linear_fwd_q(X, vals, meta, s, Lq, Ls, Rq, Rs, Y, workspace, status)
PyObject* linear_fwd_q(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!bound(n, 11)) return nullptr;
    const at::Tensor *X = bf16_tensor(a[0], "X"), *v = X ? u8_tensor(a[1], "vals") : nullptr, *m = v ? u8_tensor(a[2], "meta") : nullptr;
    const at::Tensor *Lq = m ? u8_tensor(a[4], "Lq") : nullptr, *Ls = Lq ? bf16_tensor(a[5], "Ls") : nullptr;
    const at::Tensor *Rq = Ls ? u8_tensor(a[6], "Rq") : nullptr, *Rs = Rq ? bf16_tensor(a[7], "Rs") : nullptr;
    if (!Rs || !rank2(X, "X") || !rank2(v, "vals") || !rank2(Lq, "Lq") || !rank2(Rq, "Rq")) return nullptr;
    const double s = PyFloat_AsDouble(a[3]);
    if (PyErr_Occurred()) return nullptr;
    const int64_t b = X->size(0), d_in = X->size(1), d_out = v->size(0), r = Lq->size(1) * 2;
    if (Lq->size(0) != d_out || Rq->size(0) != r || Rq->size(1) != d_in / 2) {
        PyErr_SetString(PyExc_ValueError, "adapter code shapes do not match the weight");
        return nullptr;
    }
    void *Y, *ws, *status;
    size_t ws_bytes = 0;
    if (!address(a[9], "workspace", &ws, &ws_bytes) || !address(a[10], "status", &status)) return nullptr;
    PyObject* y = output(a[8], b, d_out, *X, &Y);
    if (!y) return nullptr;
    void* stream = c10::cuda::getCurrentCUDAStream().stream();
    const int rc = unlocked(g_q, X->data_ptr(), (int)b, (const uint8_t*)v->data_ptr(), (const uint8_t*)m->data_ptr(), (float)s,
                            (const uint8_t*)Lq->data_ptr(), Ls->data_ptr(), (const uint8_t*)Rq->data_ptr(), Rs->data_ptr(), (int)r, (int)d_out,
                            (int)d_in, Y, ws, ws_bytes, (uint32_t*)status, stream);
    return finish(rc, y, "slim_linear_fwd_q");
    END_HANDLE_TH_ERRORS
}

// ---- producers of the packed weight
at::Tensor fresh(at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like) {
    return at::detail::empty_cuda(shape, type, like.device(), std::nullopt);
}

// Words the kernels can set a status bit in and the host can read without a copy: pinned memory, handed out one to a
// call and given back.  A kernel touches its word only when it has an error to report.
class StatusWords {
    static constexpr int kWords = 64, kStride = 16;            // a word per 64 bytes
    uint32_t* page_ = nullptr;
    uint64_t used_ = 0;
    std::mutex m_;
public:
    uint32_t* take() {
        std::lock_guard<std::mutex> lock(m_);
        if (!page_ && cudaHostAlloc(reinterpret_cast<void**>(&page_), kWords * kStride * 4, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();
            page_ = nullptr;
        }
        if (!page_ || used_ == ~0ull) return nullptr;
        const int i = __builtin_ctzll(~used_);
        used_ |= 1ull << i;
        page_[i * kStride] = 0;
        return page_ + i * kStride;
    }
    void give(uint32_t* w) {
        std::lock_guard<std::mutex> lock(m_);
        used_ &= ~(1ull << ((w - page_) / kStride));
    }
};
StatusWords g_words;

// pack(codes, mask, vals, meta, status, check) -> (vals, meta)
PyObject* pack(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!bound(n, 6)) return nullptr;
    const at::Tensor *c = device_tensor(a[0], at::kChar, "codes", "torch.int8"), *m = c ? u8_tensor(a[1], "mask") : nullptr;
    if (!m || !rank2(c, "codes")) return nullptr;
    const int64_t d_out = c->size(0), d_in = c->size(1);
    const int check = PyObject_IsTrue(a[5]);
    if (check < 0) return nullptr;
    void *vp, *mp, *status;
    if (!address(a[2], "vals", &vp) || !address(a[3], "meta", &mp) || !address(a[4], "status", &status)) return nullptr;
    at::Tensor vals, meta, own;
    if (!vp) { vals = fresh({d_out, d_in / 4}, at::kByte, *c); vp = vals.data_ptr(); } else vals = THPVariable_Unpack(a[2]);
    if (!mp) { meta = fresh({d_out, d_in / 8}, at::kByte, *c); mp = meta.data_ptr(); } else meta = THPVariable_Unpack(a[3]);
    const auto stream = c10::cuda::getCurrentCUDAStream();
    uint32_t* word = nullptr;
    const bool look = check && !status;
    if (look) {
        word = g_words.take();
        if (!word) { own = at::zeros({1}, c->options().dtype(at::kInt)); }
        status = word ? word : own.data_ptr();
    }
    const void *cp = c->data_ptr(), *kp = m->data_ptr();
    int rc;
    uint32_t bits = 0;
    Py_BEGIN_ALLOW_THREADS
    rc = g_pack((const int8_t*)cp, (const uint8_t*)kp, (int)d_out, (int)d_in, (uint8_t*)vp, (uint8_t*)mp, (uint32_t*)status, stream.stream());
    if (word) {
        if (rc == 0 && cudaStreamSynchronize(stream.stream()) != cudaSuccess) rc = 6;          // SLIM_ERR_CUDA
        bits = *static_cast<volatile uint32_t*>(word);
        g_words.give(word);
    }
    Py_END_ALLOW_THREADS
    if (look && !word && rc == 0) bits = (uint32_t)own.item<int>();
    for (int code : {3, 4})                                    // SLIM_ERR_BAD_MASK, SLIM_ERR_CODE_RANGE
        if (rc == 0 && (bits & (1u << code))) rc = code;
    if (rc != 0) return finish(rc, nullptr, "slim_pack");
    return Py_BuildValue("(NN)", THPVariable_Wrap(std::move(vals)), THPVariable_Wrap(std::move(meta)));
    END_HANDLE_TH_ERRORS
}

// mask_top2(codes, xbar, status) -> mask
PyObject* mask_top2(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!bound(n, 3)) return nullptr;
    const at::Tensor* c = device_tensor(a[0], at::kChar, "codes", "torch.int8");
    if (!c || !rank2(c, "codes")) return nullptr;
    const at::Tensor* x = a[1] == Py_None ? nullptr : device_tensor(a[1], at::kFloat, "xbar", "torch.float32");
    if (a[1] != Py_None && !x) return nullptr;
    void* status;
    if (!address(a[2], "status", &status)) return nullptr;
    at::Tensor mask = fresh(c->sizes(), at::kByte, *c);
    const int rc = unlocked(g_mask, (const int8_t*)c->data_ptr(), x ? (const float*)x->data_ptr() : nullptr, (int)c->size(0), (int)c->size(1),
                            (uint8_t*)mask.data_ptr(), (uint32_t*)status, c10::cuda::getCurrentCUDAStream().stream());
    return rc == 0 ? THPVariable_Wrap(std::move(mask)) : finish(rc, nullptr, "slim_mask_top2");
    END_HANDLE_TH_ERRORS
}

// pack_adapter(A) -> (codes, scales)
PyObject* pack_adapter(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!bound(n, 1)) return nullptr;
    const at::Tensor* A = bf16_tensor(a[0], "A");
    if (!A || !rank2(A, "A")) return nullptr;
    const int64_t rows = A->size(0), cols = A->size(1);
    if (rows < 1 || cols < 2 || cols % 2 != 0) return finish(1, nullptr, "slim_pack_adapter");      // SLIM_ERR_INVALID_ARG
    at::Tensor codes = fresh({rows, cols / 2}, at::kByte, *A), scales = fresh({rows, (cols + 127) / 128}, at::kBFloat16, *A);
    const int rc = unlocked(g_pack_adapter, A->data_ptr(), (int)rows, (int)cols, (uint8_t*)codes.data_ptr(), scales.data_ptr(),
                            c10::cuda::getCurrentCUDAStream().stream());
    if (rc != 0) return finish(rc, nullptr, "slim_pack_adapter");
    return Py_BuildValue("(NN)", THPVariable_Wrap(std::move(codes)), THPVariable_Wrap(std::move(scales)));
    END_HANDLE_TH_ERRORS
}

// quant(W, status) -> (codes, scale_alpha, table, alpha)
PyObject* quant(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!bound(n, 2)) return nullptr;
    const at::Tensor* W = device_tensor(a[0], at::kFloat, "W", "torch.float32");
    if (!W || !rank2(W, "W")) return nullptr;
    void* status;
    if (!address(a[1], "status", &status)) return nullptr;
    const int64_t d_out = W->size(0), d_in = W->size(1);
    const size_t bytes = g_quant_bytes((int)d_out, (int)d_in);
    at::Tensor ws = fresh({(int64_t)bytes}, at::kByte, *W), codes = fresh({d_out, d_in}, at::kChar, *W), sa = fresh({4}, at::kFloat, *W);
    const int rc = unlocked(g_quant, (const float*)W->data_ptr(), (int)d_out, (int)d_in, (int8_t*)codes.data_ptr(), (float*)sa.data_ptr(),
                            ws.data_ptr(), bytes, (uint32_t*)status, c10::cuda::getCurrentCUDAStream().stream());
    if (rc != 0) return finish(rc, nullptr, "slim_quant");
    const int64_t bins = std::max<int64_t>(512, std::min<int64_t>(d_out * d_in / 1000, 20000)), at_ = 256 + (bins * 4 + 255) / 256 * 256;
    at::Tensor tab = ws.slice(0, at_, at_ + 59 * 8).view(at::kDouble);
    return Py_BuildValue("(NNNN)", THPVariable_Wrap(std::move(codes)), THPVariable_Wrap(sa.slice(0, 0, 2)),
                         THPVariable_Wrap(tab.slice(0, 0, 58).view({29, 2})), THPVariable_Wrap(tab.select(0, 58)));
    END_HANDLE_TH_ERRORS
}

// bind(SlimError, addresses of the functions in the loaded libslim)
PyObject* bind(PyObject*, PyObject* args) {
    PyObject* err;
    unsigned long long f, t, q, by, tx, pk, qu, qb, mk, pa;
    if (!PyArg_ParseTuple(args, "OKKKKKKKKKK", &err, &f, &t, &q, &by, &tx, &pk, &qu, &qb, &mk, &pa)) return nullptr;
    Py_INCREF(err);
    Py_XDECREF(g_error);
    g_error = err;
    g_fwd = reinterpret_cast<FwdFn>(f); g_tiled = reinterpret_cast<TiledFn>(t); g_q = reinterpret_cast<QFn>(q);
    g_tiled_bytes = reinterpret_cast<BytesFn>(by); g_text = reinterpret_cast<TextFn>(tx);
    g_pack = reinterpret_cast<PackFn>(pk); g_quant = reinterpret_cast<QuantFn>(qu); g_quant_bytes = reinterpret_cast<QuantBytesFn>(qb);
    g_mask = reinterpret_cast<MaskFn>(mk); g_pack_adapter = reinterpret_cast<AdapterFn>(pa);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, nullptr},
    {"linear_fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(linear_fwd)), METH_FASTCALL, nullptr},
    {"linear_fwd_tiled", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(linear_fwd_tiled)), METH_FASTCALL, nullptr},
    {"linear_fwd_q", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(linear_fwd_q)), METH_FASTCALL, nullptr},
    {"pack", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(pack)), METH_FASTCALL, nullptr},
    {"mask_top2", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(mask_top2)), METH_FASTCALL, nullptr},
    {"pack_adapter", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(pack_adapter)), METH_FASTCALL, nullptr},
    {"quant", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(quant)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_slim_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__slim_native() { return PyModule_Create(&module); }
