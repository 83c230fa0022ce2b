// The per-call half of the Python binding in native code: argument checks, result allocation and the call into the C
// ABI of include/meteora.h.
//
// A decode call is 11 - 16 us on the GPU; marshalling it through ctypes (a dozen attribute reads and tensor checks in
// Python, six tensor ops for the two views of the routing) took 26 us on the host, so a caller that does not capture
// CUDA graphs waited for Python, not for the kernel.  The checks, messages and results are those of binding.py's
// documented functions; nothing of the layer is computed here and nothing is kept between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <stdexcept>
#include <string>
#include <vector>

#include "meteora.h"

namespace {

PyObject* g_error = nullptr;   // binding.MeteoraError, set by init()

// A Python exception is already set.
struct PySet {};

[[noreturn]] void fail(PyObject* type, const std::string& text) {
    PyErr_SetString(type, text.c_str());
    throw PySet{};
}

void check(int status, const char* where) {
    if (status == METEORA_OK) return;
    PyObject* e = PyObject_CallFunction(g_error, "is", status, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw PySet{};
}

// A call into the library with the GIL released, as ctypes makes it: a launch can block on a full queue and a copy of
// pageable memory does, and other Python threads go on meanwhile.  Arguments are worked out before (under the GIL); the
// caller's references keep their tensors.
template <class Call>
int released(Call&& call) {
    struct Gil {
        PyThreadState* state = PyEval_SaveThread();
        ~Gil() { PyEval_RestoreThread(state); }
    } gil;
    return call();
}

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, std::string(name) + " must be a torch.Tensor");
    return THPVariable_Unpack(o);
}

int64_t integer(PyObject* o) {
    const int64_t direct = PyLong_Check(o) ? PyLong_AsLongLong(o) : -1;
    if (PyLong_Check(o)) {
        if (direct == -1 && PyErr_Occurred()) throw PySet{};
        return direct;
    }
    PyObject* n = PyNumber_Long(o);
    if (!n) throw PySet{};
    const int64_t v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw PySet{};
    return v;
}

double real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PySet{};
    return v;
}

void dims(const at::Tensor& t, int64_t n, const char* name) {
    if (t.dim() != n) fail(PyExc_ValueError, std::string(name) + ": expected " + std::to_string(n) + " dimensions, got " + std::to_string(t.dim()));
}

meteora_dtype_t dtype_code(const at::Tensor& t) {
    const auto st = t.scalar_type();
    if (st == at::kFloat) return METEORA_F32;
    if (st == at::kBFloat16) return METEORA_BF16;
    fail(PyExc_TypeError, std::string("unsupported dtype torch.") + c10::toString(st) + "; the layer runs in float32 or bfloat16");
}

std::string size_text(at::IntArrayRef s) {
    std::string out = "(";
    for (size_t i = 0; i < s.size(); ++i) out += (i ? ", " : "") + std::to_string(s[i]);
    return out + (s.size() == 1 ? ",)" : ")");
}

// A contiguous CUDA tensor of this shape and type, or an exception.
void* dev(const at::Tensor& t, at::IntArrayRef shape, at::ScalarType dt, const char* name) {
    if (!t.is_cuda() || !t.is_contiguous()) fail(PyExc_ValueError, std::string(name) + " must be a contiguous CUDA tensor");
    if (t.sizes() != shape || t.scalar_type() != dt)
        fail(PyExc_ValueError, std::string(name) + ": expected " + size_text(shape) + " " + c10::toString(dt) + ", got " +
                                   size_text(t.sizes()) + " " + c10::toString(t.scalar_type()));
    return t.data_ptr();
}
void* dev(PyObject* o, at::IntArrayRef shape, at::ScalarType dt, const char* name) { return dev(tensor(o, name), shape, dt, name); }

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor empty(at::IntArrayRef shape, at::ScalarType dt, const at::Tensor& like) {
    return at::empty(shape, at::TensorOptions().dtype(dt).device(like.device()));
}

meteora_shape_t make_shape(int64_t T, int64_t d_in, int64_t d_out, int64_t N, int64_t r, int64_t k, meteora_dtype_t dt, double temperature) {
    return meteora_shape_t{(int)T, (int)d_in, (int)d_out, (int)N, (int)r, (int)k, dt, (float)temperature};
}

at::Tensor zeroed(size_t bytes, const at::Tensor& like, const char* where) {
    // (the header alone needs zeros: clearing all of it took 2 to 30 us of a decode call made without a workspace)
    if (bytes == 0) check(METEORA_ERR_INVALID_ARG, where);
    at::Tensor ws = empty({(int64_t)bytes}, at::kByte, like);
    void* const st = stream();
    check(released([&] { return meteora_workspace_init(ws.data_ptr(), st); }), where);
    return ws;
}

// A [T, k] tensor over 4-byte values inside `workspace`: shares its storage and version counter, as a view does.
at::Tensor view_of(const at::Tensor& workspace, const void* ptr, at::ScalarType dt, int64_t T, int64_t k) {
    const int64_t off = (const char*)ptr - (const char*)workspace.storage().data();
    if (off % 4 != 0) fail(PyExc_RuntimeError, "the workspace does not start on a 4-byte boundary of its storage");
    auto impl = c10::make_intrusive<c10::TensorImpl>(c10::TensorImpl::VIEW, c10::Storage(workspace.storage()), workspace.key_set(),
                                                     c10::scalarTypeToTypeMeta(dt));
    impl->set_storage_offset(off / 4);
    const int64_t sizes[2] = {T, k};
    impl->set_sizes_contiguous(at::IntArrayRef(sizes, 2));
    impl->set_version_counter(workspace.unsafeGetTensorImpl()->version_counter());
    return at::Tensor(std::move(impl));
}

PyObject* wrap(const at::Tensor& t) {
    PyObject* o = THPVariable_Wrap(t);
    if (!o) throw PySet{};
    return o;
}

PyObject* keep(PyObject* o) {
    Py_INCREF(o);
    return o;
}

template <class... P>
PyObject* tuple(P... parts) {
    PyObject* out = PyTuple_Pack(sizeof...(P), parts...);
    (Py_DECREF(parts), ...);
    if (!out) throw PySet{};
    return out;
}

typedef PyObject* (*Body)(PyObject* const* a);

template <Body body, int n_args>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    if (nargs != n_args) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", n_args, nargs);
        return nullptr;
    }
    try {
        return body(args);
    } catch (const PySet&) {
        return nullptr;
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// (x, Wg, k, temperature, want_logits) -> (idx, w, logits or None)
PyObject* gate_topk(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0], "x"), &Wg = tensor(a[1], "Wg");
    dims(x, 2, "x");
    dims(Wg, 2, "Wg");
    const int64_t T = x.size(0), d_in = x.size(1), N = Wg.size(0), k = integer(a[2]);
    const meteora_shape_t s = make_shape(T, d_in, 1, N, 1, k, dtype_code(x), real(a[3]));
    const bool want = PyObject_IsTrue(a[4]) == 1;
    void *px = dev(x, {T, d_in}, x.scalar_type(), "x"), *pg = dev(Wg, {N, d_in}, x.scalar_type(), "Wg");
    at::Tensor idx = empty({T, k}, at::kInt, x), w = empty({T, k}, at::kFloat, x), logits;
    if (want) logits = empty({T, N}, at::kFloat, x);
    int32_t* const pi = (int32_t*)idx.data_ptr();
    float *const pw = (float*)w.data_ptr(), *const pl = want ? (float*)logits.data_ptr() : nullptr;
    void* const st = stream();
    check(released([&] { return meteora_gate_topk(px, pg, &s, pi, pw, pl, st); }), "meteora_gate_topk");
    return tuple(wrap(idx), wrap(w), want ? wrap(logits) : keep(Py_None));
}

// (topk_idx, N) -> (counts, offsets, perm)
PyObject* route(PyObject* const* a) {
    const at::Tensor& idx = tensor(a[0], "topk_idx");
    dims(idx, 2, "topk_idx");
    const int64_t T = idx.size(0), k = idx.size(1), N = integer(a[1]);
    void* p = dev(idx, {T, k}, at::kInt, "topk_idx");
    at::Tensor counts = empty({N}, at::kInt, idx), offsets = empty({N + 1}, at::kInt, idx), perm = empty({T * k}, at::kInt, idx);
    int32_t *const pc = (int32_t*)counts.data_ptr(), *const po = (int32_t*)offsets.data_ptr(), *const pp = (int32_t*)perm.data_ptr();
    void* const st = stream();
    check(released([&] { return meteora_route((const int32_t*)p, (int)T, (int)k, (int)N, pc, po, pp, st); }), "meteora_route");
    return tuple(wrap(counts), wrap(offsets), wrap(perm));
}

// (x, A, B, topk_idx, topk_w, offsets, perm, workspace or out, static) -> delta
PyObject* lora_delta(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0], "x"), &A = tensor(a[1], "A"), &B = tensor(a[2], "B"), &idx = tensor(a[3], "topk_idx");
    dims(x, 2, "x");
    dims(A, 3, "A");
    dims(B, 3, "B");
    dims(idx, 2, "topk_idx");
    const int64_t T = x.size(0), d_in = x.size(1), N = A.size(0), r = A.size(1), d_out = B.size(1), k = idx.size(1);
    const bool is_static = a[8] == Py_True;
    const meteora_shape_t s = make_shape(T, d_in, d_out, N, r, k, dtype_code(x), 1.0);
    const auto dt = x.scalar_type();
    at::Tensor ws, delta;
    if (is_static && a[7] != Py_None) delta = tensor(a[7], "out");
    if (!is_static) ws = a[7] == Py_None ? zeroed(meteora_workspace_bytes(&s), x, "meteora_workspace_bytes") : tensor(a[7], "workspace");
    if (!delta.defined()) delta = empty({T, d_out}, at::kFloat, x);
    const void *px = dev(x, {T, d_in}, dt, "x"), *pA = dev(A, {N, r, d_in}, dt, "A"), *pB = dev(B, {N, d_out, r}, dt, "B");
    const int32_t* pi = (const int32_t*)dev(idx, {T, k}, at::kInt, "topk_idx");
    const float* pw = (const float*)dev(a[4], {T, k}, at::kFloat, "topk_w");
    const int32_t* po = (const int32_t*)dev(a[5], {N + 1}, at::kInt, "offsets");
    const int32_t* pp = (const int32_t*)dev(a[6], {T * k}, at::kInt, "perm");
    float* const out = (float*)dev(delta, {T, d_out}, at::kFloat, "delta");
    void *const pws = is_static ? nullptr : ws.data_ptr(), *const st = stream();
    const size_t ws_bytes = is_static ? 0 : (size_t)ws.numel();
    check(released([&] {
              return is_static ? meteora_lora_delta_static(px, pA, pB, pi, pw, po, pp, &s, out, st)
                               : meteora_lora_delta(px, pA, pB, pi, pw, po, pp, &s, out, pws, ws_bytes, st);
          }),
          is_static ? "meteora_lora_delta_static" : "meteora_lora_delta");
    return wrap(delta);
}

// (x, W0, A, B, Wg, k, temperature, workspace, out, return_routing) -> y or (y, idx, w)
PyObject* linear_forward(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0], "x"), &W0 = tensor(a[1], "W0"), &A = tensor(a[2], "A");
    dims(x, 2, "x");
    dims(A, 3, "A");
    if (W0.dim() < 1) dims(W0, 2, "W0");
    const int64_t T = x.size(0), d_in = x.size(1), d_out = W0.size(0), N = A.size(0), r = A.size(1), k = integer(a[5]);
    const meteora_shape_t s = make_shape(T, d_in, d_out, N, r, k, dtype_code(x), real(a[6]));
    const auto dt = x.scalar_type();
    at::Tensor made_ws, made_y;
    if (a[7] == Py_None) made_ws = zeroed(meteora_workspace_bytes(&s), x, "meteora_workspace_bytes");
    if (a[8] == Py_None) made_y = empty({T, d_out}, dt, x);
    const at::Tensor &ws = made_ws.defined() ? made_ws : tensor(a[7], "workspace"), &y = made_y.defined() ? made_y : tensor(a[8], "out");
    const void *px = dev(x, {T, d_in}, dt, "x"), *pW = dev(W0, {d_out, d_in}, dt, "W0"), *pA = dev(A, {N, r, d_in}, dt, "A"),
               *pB = dev(a[3], {N, d_out, r}, dt, "B"), *pG = dev(a[4], {N, d_in}, dt, "Wg");
    void *const py = dev(y, {T, d_out}, dt, "y"), *const pws = ws.data_ptr(), *const st = stream();
    const size_t ws_bytes = (size_t)ws.numel();
    check(released([&] { return meteora_linear_forward(px, pW, pA, pB, pG, &s, py, pws, ws_bytes, st); }), "meteora_linear_forward");
    PyObject* y_obj = made_y.defined() ? wrap(y) : keep(a[8]);
    if (PyObject_IsTrue(a[9]) != 1) return y_obj;
    int32_t* p_idx = nullptr;
    float* p_w = nullptr;
    check(meteora_workspace_routing(&s, ws.data_ptr(), &p_idx, &p_w), "meteora_workspace_routing");
    return tuple(y_obj, wrap(view_of(ws, p_idx, at::kInt, T, k)), wrap(view_of(ws, p_w, at::kFloat, T, k)));
}

// (x_host, W0, A, B, Wg, k, y_host, workspace, temperature) -> y_host
PyObject* linear_forward_host(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0], "x_host"), &W0 = tensor(a[1], "W0"), &A = tensor(a[2], "A"), &y = tensor(a[6], "y_host"),
                     &ws = tensor(a[7], "workspace");
    dims(x, 2, "x_host");
    dims(A, 3, "A");
    if (W0.dim() < 1) dims(W0, 2, "W0");
    const int64_t T = x.size(0), d_in = x.size(1), d_out = W0.size(0), N = A.size(0), r = A.size(1), k = integer(a[5]);
    const auto dt = W0.scalar_type();
    const meteora_shape_t s = make_shape(T, d_in, d_out, N, r, k, dt == at::kFloat ? METEORA_F32 : METEORA_BF16, real(a[8]));
    for (int i = 0; i < 2; ++i) {
        const at::Tensor& t = i ? y : x;
        if (t.is_cuda() || !t.is_contiguous() || t.scalar_type() != dt)
            fail(PyExc_ValueError, std::string(i ? "y_host" : "x_host") + " must be a contiguous host tensor of dtype " + c10::toString(dt));
    }
    if (y.dim() != 2 || y.size(0) != T || y.size(1) != d_out) fail(PyExc_ValueError, "y_host has the wrong shape");
    const void *px = x.data_ptr(), *pW = dev(W0, {d_out, d_in}, dt, "W0"), *pA = dev(A, {N, r, d_in}, dt, "A"),
               *pB = dev(a[3], {N, d_out, r}, dt, "B"), *pG = dev(a[4], {N, d_in}, dt, "Wg");
    void *const py = y.data_ptr(), *const pws = ws.data_ptr(), *const st = stream();
    const size_t ws_bytes = (size_t)ws.numel();
    check(released([&] { return meteora_linear_forward_host(px, pW, pA, pB, pG, &s, py, pws, ws_bytes, st); }), "meteora_linear_forward_host");
    return keep(a[6]);
}

// (x, A, B, dy, topk_idx, topk_w, temperature, Bt, workspace) -> (dWg, dlogit)
PyObject* gate_backward(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0], "x"), &A = tensor(a[1], "A"), &idx = tensor(a[4], "topk_idx");
    const bool bt = a[7] != Py_None;
    const at::Tensor& B = tensor(bt ? a[7] : a[2], bt ? "Bt" : "B");
    dims(x, 2, "x");
    dims(A, 3, "A");
    dims(B, 3, bt ? "Bt" : "B");
    dims(idx, 2, "topk_idx");
    const int64_t T = x.size(0), d_in = x.size(1), N = A.size(0), r = A.size(1), d_out = B.size(bt ? 2 : 1), k = idx.size(1);
    const auto dt = x.scalar_type();
    const meteora_shape_t s = make_shape(T, d_in, d_out, N, r, k, dt == at::kFloat ? METEORA_F32 : METEORA_BF16, real(a[6]));
    const size_t need = meteora_gate_backward_workspace_bytes(&s);
    if (need == 0) check(METEORA_ERR_INVALID_ARG, "meteora_gate_backward_workspace_bytes");
    at::Tensor ws = a[8] == Py_None ? empty({(int64_t)need}, at::kByte, x) : tensor(a[8], "workspace");
    at::Tensor dWg = empty({N, d_in}, at::kFloat, x), dlogit = empty({T, k}, at::kFloat, x);
    const void* pB = bt ? dev(B, {N, r, d_out}, dt, "Bt") : dev(B, {N, d_out, r}, dt, "B");
    const auto fn = bt ? meteora_gate_backward_bt : meteora_gate_backward;
    const void *px = dev(x, {T, d_in}, dt, "x"), *pA = dev(A, {N, r, d_in}, dt, "A"), *pdy = dev(a[3], {T, d_out}, dt, "dy");
    const int32_t* pi = (const int32_t*)dev(idx, {T, k}, at::kInt, "topk_idx");
    const float* pw = (const float*)dev(a[5], {T, k}, at::kFloat, "topk_w");
    float *const pl = (float*)dlogit.data_ptr(), *const pd = (float*)dWg.data_ptr();
    void *const pws = ws.data_ptr(), *const st = stream();
    const size_t ws_bytes = (size_t)ws.numel();
    check(released([&] { return fn(px, pA, pB, pdy, pi, pw, &s, pl, pd, pws, ws_bytes, st); }), "meteora_gate_backward");
    return tuple(wrap(dWg), wrap(dlogit));
}

// (x, W0s, As, Bs, Wgs, k, temperature, workspace, return_routing) -> [y] or ([y], [(idx, w)])
PyObject* linear_forward_group(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    dims(x, 2, "x");
    const int64_t T = x.size(0), d_in = x.size(1), k = integer(a[5]);
    const double temperature = real(a[6]);
    const meteora_dtype_t code = dtype_code(x);
    const auto dt = x.scalar_type();
    struct Held {                        // the four sequences, as tuples or lists whose items can be read directly
        PyObject* o[4] = {};
        ~Held() {
            for (PyObject* p : o) Py_XDECREF(p);
        }
    } seq;
    const char* names[4] = {"W0", "A", "B", "Wg"};
    for (int i = 0; i < 4; ++i)
        if (!(seq.o[i] = PySequence_Fast(a[1 + i], "expected a sequence of tensors"))) throw PySet{};
    const Py_ssize_t G = PySequence_Fast_GET_SIZE(seq.o[0]);
    for (int i = 1; i < 4; ++i)
        if (PySequence_Fast_GET_SIZE(seq.o[i]) < G) fail(PyExc_IndexError, "a list of the group is shorter than W0s");
    if (G == 0) fail(PyExc_IndexError, "an empty group");
    auto item = [&](int i, Py_ssize_t m) -> const at::Tensor& { return tensor(PySequence_Fast_GET_ITEM(seq.o[i], m), names[i]); };
    dims(item(1, 0), 3, "A");
    const int64_t N = item(1, 0).size(0), r = item(1, 0).size(1);
    std::vector<int> d_out(G);
    for (Py_ssize_t m = 0; m < G; ++m) {
        if (item(0, m).dim() < 1) dims(item(0, m), 2, "W0");
        d_out[m] = (int)item(0, m).size(0);
    }
    const meteora_shape_t s = make_shape(T, d_in, d_out[0], N, r, k, code, temperature);
    at::Tensor ws = a[7] == Py_None ? zeroed(meteora_group_workspace_bytes(&s, d_out.data(), (int)G), x, "meteora_group_workspace_bytes")
                                    : tensor(a[7], "workspace");
    std::vector<at::Tensor> ys(G), held;                             // (held: another thread may change the lists meanwhile)
    held.reserve(4 * G);
    std::vector<const void*> ptr[4];
    for (auto& p : ptr) p.resize(G);
    std::vector<void*> py(G);
    for (Py_ssize_t m = 0; m < G; ++m) {
        ys[m] = empty({T, d_out[m]}, dt, x);
        py[m] = ys[m].data_ptr();
        ptr[0][m] = dev(item(0, m), {d_out[m], d_in}, dt, "W0");
        ptr[1][m] = dev(item(1, m), {N, r, d_in}, dt, "A");
        ptr[2][m] = dev(item(2, m), {N, d_out[m], r}, dt, "B");
        ptr[3][m] = dev(item(3, m), {N, d_in}, dt, "Wg");
        for (int i = 0; i < 4; ++i) held.push_back(item(i, m));
    }
    const void* px = dev(x, {T, d_in}, dt, "x");
    void *const pws = ws.data_ptr(), *const st = stream();
    const size_t ws_bytes = (size_t)ws.numel();
    check(released([&] {
              return meteora_linear_forward_group(px, ptr[0].data(), ptr[1].data(), ptr[2].data(), ptr[3].data(), d_out.data(), (int)G, &s,
                                                  py.data(), pws, ws_bytes, st);
          }),
          "meteora_linear_forward_group");
    PyObject* out = PyList_New(G);
    if (!out) throw PySet{};
    for (Py_ssize_t m = 0; m < G; ++m) PyList_SET_ITEM(out, m, wrap(ys[m]));
    if (PyObject_IsTrue(a[8]) != 1) return out;
    PyObject* routing = PyList_New(G);
    if (!routing) throw PySet{};
    for (Py_ssize_t m = 0; m < G; ++m) {
        int32_t* p_idx = nullptr;
        float* p_w = nullptr;
        check(meteora_group_workspace_routing(&s, d_out.data(), (int)G, (int)m, ws.data_ptr(), &p_idx, &p_w), "meteora_group_workspace_routing");
        PyList_SET_ITEM(routing, m, tuple(wrap(view_of(ws, p_idx, at::kInt, T, k)), wrap(view_of(ws, p_w, at::kFloat, T, k))));
    }
    return tuple(out, routing);
}

PyObject* init(PyObject* const* a) {
    Py_XDECREF(g_error);
    g_error = keep(a[0]);
    return keep(Py_None);
}

#define METEORA_METHOD(name, n) {#name, (PyCFunction)(void (*)(void))entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METEORA_METHOD(gate_topk, 5),           METEORA_METHOD(route, 2),
                         METEORA_METHOD(lora_delta, 9),          METEORA_METHOD(linear_forward, 10),
                         METEORA_METHOD(linear_forward_host, 9), METEORA_METHOD(gate_backward, 9),
                         METEORA_METHOD(linear_forward_group, 9), METEORA_METHOD(init, 1),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
