// Native half of the Python binding: size checks of the tensors, their pointers, the current stream and the call
// of the C ABI, in one C++ function per entry point.
//
// A decode step is a chain of calls whose kernels take a few microseconds.  Marshalling the arguments in Python and
// through ctypes took 5.5 us (three arguments) to 11.5 us (ten) a call besides the launch itself, more than most of
// those kernels.  Host time of a call here, its launch included (medians on two hosts): one product 2.5-2.9 us, a planned
// list's two launches 4.1-4.9, packing 2.1-2.5 and 0.9 more where it allocates its output, decode_packed with two outputs
// 4.2-4.5; a call that launches nothing takes 0.2 us.  tetra.py keeps the public functions (names, defaults,
// documentation) and passes their arguments on by position.
#include <Python.h>
#include <dlfcn.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdarg>
#include <cstdint>
#include <string>

#include "../../include/tetra.h"
#include "../../include/tetra_q4.h"

namespace {

// The C ABI, looked up in the library tetra.py names.
struct Api {
    decltype(&tetra_status_string) status_string;
    decltype(&tetra_table_bytes) table_bytes;
    decltype(&tetra_gemv) gemv;
    decltype(&tetra_gemv_tail) gemv_tail;
    decltype(&tetra_gemv_list) gemv_list;
    decltype(&tetra_gemv_grouped_run) grouped_run;
    decltype(&tetra_gemv_batched) gemv_batched;
    decltype(&tetra_gemv_noalloc) gemv_noalloc;
    decltype(&tetra_codes_bytes) codes_bytes;
    decltype(&tetra_pack_codes) pack_codes;
    decltype(&tetra_decode_packed) decode_packed;
    decltype(&tetra_encode_blocks) encode_blocks;
    decltype(&tetra_q4_packed_bytes) q4_packed_bytes;
    decltype(&tetra_q4_pack) q4_pack;
    decltype(&tetra_q4_gemv) q4_gemv;
    decltype(&tetra_q4_rows) q4_rows;
    decltype(&tetra_q4_list_run) q4_list_run;
} api;
PyObject* tetra_error = nullptr;  // the exception class

struct Failed {};  // a Python exception has been set

[[noreturn]] void fail(PyObject* type, const char* format, ...) {
    va_list args;
    va_start(args, format);
    PyErr_FormatV(type, format, args);
    va_end(args);
    throw Failed();
}

void check(int rc, const char* what) {
    if (rc != 0) fail(tetra_error, "%s failed: %s (%d)", what, api.status_string(rc), rc);
}

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a tensor, got %s", Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
}
void* pointer(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }

// The tensor holds at least nbytes, contiguously, where the call reads or writes it.  The C ABI sees plain
// pointers; a tensor that is too small would be read or written past its end.
void* need(PyObject* o, size_t nbytes, const char* what, const char* name) {
    if (o == Py_None) return nullptr;
    const at::Tensor& t = tensor(o);
    const size_t have = size_t(t.numel()) * t.element_size();
    if (have < nbytes) fail(tetra_error, "%s%s: tensor of %zu bytes, the call needs %zu", what, name, have, nbytes);
    if (!t.is_contiguous()) fail(tetra_error, "%s%s: tensor is not contiguous", what, name);
    if (!t.is_cuda() && !t.is_pinned())  // pinned host memory is mapped into the device's address space
        fail(tetra_error, "%s%s: tensor is neither on the device nor in pinned host memory", what, name);
    return t.data_ptr();
}

// The blob of tetra_build_table.
void* table_of(PyObject* o, const char* what) { return need(o, api.table_bytes(), what, " table"); }

int integer(PyObject* o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return int(v);
}

bool truth(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw Failed();
    return v != 0;
}

void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* handle = PyObject_GetAttrString(o, "cuda_stream");
    if (!handle) throw Failed();
    void* s = PyLong_AsVoidPtr(handle);
    Py_DECREF(handle);
    if (PyErr_Occurred()) throw Failed();
    return s;
}

// A call of the C ABI: other Python threads may run meanwhile (a full launch queue makes it wait).
template <typename F>
int unlocked(F&& f) {
    PyThreadState* state = PyEval_SaveThread();
    const int rc = f();
    PyEval_RestoreThread(state);
    return rc;
}

template <typename F>
PyObject* guarded(Py_ssize_t have, Py_ssize_t want, F&& body) {
    try {
        if (have != want) fail(PyExc_TypeError, "%zd arguments, %zd expected", have, want);
        return body();
    } catch (const Failed&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
PyObject* same(PyObject* o) {
    Py_INCREF(o);
    return o;
}
#define FASTCALL(name) PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)

// Device memory from torch's caching allocator, without the dispatcher's detour (0.5 us a tensor; loading a layer
// makes 22 of them).  Not a function that torch promises to keep: a binding serves the version it was built for only.
at::Tensor device_empty(at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like) {
    if (!like.is_cuda()) fail(tetra_error, "expected a tensor on the device");
    return at::detail::empty_cuda(shape, type, like.device(), c10::nullopt);
}

int blocks_of(int K, bool tail_rule) { return (tail_rule || K % 24 == 0) ? K / 24 : (K + 23) / 24; }

struct GemvArgs {
    void *codes, *row_scales, *table, *x, *y, *tail;
    int N, K, batch;
};
// Sizes of the tensors of one product (tail_rule: floor(K/24) words per row plus a float16 tail); a shape the
// library rejects is passed on unchecked.
GemvArgs gemv_args(PyObject* codes, PyObject* row_scales, PyObject* table, PyObject* x, PyObject* y, int N, int K, int batch,
                   PyObject* tail, bool tail_rule, const char* what) {
    GemvArgs g{nullptr, nullptr, table_of(table, what), nullptr, nullptr, nullptr, N, K, batch};
    if (N <= 0 || K <= 0 || batch <= 0) {
        g.codes = pointer(codes);
        g.row_scales = pointer(row_scales);
        g.x = pointer(x);
        g.y = pointer(y);
        g.tail = pointer(tail);
        return g;
    }
    const size_t B = size_t(blocks_of(K, tail_rule)), rows = size_t(N), v = size_t(batch);
    g.codes = B ? need(codes, (rows + 7) / 8 * B * 48, what, " codes") : pointer(codes);
    g.row_scales = need(row_scales, 4 * rows, what, " row_scales");
    g.x = need(x, 2 * v * size_t(K), what, " x");
    g.y = need(y, 4 * v * rows, what, " y");
    g.tail = tail_rule && K % 24 ? need(tail, 2 * rows * size_t(K % 24), what, " tail") : pointer(tail);
    return g;
}

// codes, row_scales, table, x, y, N, K, batch, stream
FASTCALL(py_gemv) {
    return guarded(n, 9, [&] {
        const GemvArgs g = gemv_args(a[0], a[1], a[2], a[3], a[4], integer(a[5]), integer(a[6]), integer(a[7]), Py_None, false, "tetra_gemv");
        void* s = stream_of(a[8]);
        check(unlocked([&] { return api.gemv(g.codes, static_cast<float*>(g.row_scales), g.table, g.x, static_cast<float*>(g.y), g.N, g.K, g.batch, s); }),
              "tetra_gemv");
        return same(a[4]);
    });
}
// codes, row_scales, table, x, y, N, K, batch, tail, stream
FASTCALL(py_gemv_tail) {
    return guarded(n, 10, [&] {
        const GemvArgs g = gemv_args(a[0], a[1], a[2], a[3], a[4], integer(a[5]), integer(a[6]), integer(a[7]), a[8], a[8] != Py_None, "tetra_gemv_tail");
        void* s = stream_of(a[9]);
        check(unlocked([&] { return api.gemv_tail(g.codes, static_cast<float*>(g.row_scales), g.table, g.x, static_cast<float*>(g.y), g.N, g.K, g.batch, g.tail, s); }),
              "tetra_gemv_tail");
        return same(a[4]);
    });
}
// codes, row_scales, table, x, y, N, K, tail, stream
FASTCALL(py_gemv_noalloc) {
    return guarded(n, 9, [&] {
        const GemvArgs g = gemv_args(a[0], a[1], a[2], a[3], a[4], integer(a[5]), integer(a[6]), 1, a[7], a[7] != Py_None, "tetra_gemv_noalloc");
        void* s = stream_of(a[8]);
        check(unlocked([&] { return api.gemv_noalloc(g.codes, static_cast<float*>(g.row_scales), g.table, g.x, static_cast<float*>(g.y), g.N, g.K, g.tail, s); }),
              "tetra_gemv_noalloc");
        return same(a[4]);
    });
}
// codes, row_scales, table, x, y, N, K, batch, tail, workspace, stream
FASTCALL(py_gemv_batched) {
    return guarded(n, 11, [&] {
        const GemvArgs g = gemv_args(a[0], a[1], a[2], a[3], a[4], integer(a[5]), integer(a[6]), integer(a[7]), a[8], a[8] != Py_None, "tetra_gemv_batched");
        const at::Tensor& ws = tensor(a[9]);
        void* wp = ws.data_ptr();
        const size_t wn = size_t(ws.numel()) * ws.element_size();
        void* s = stream_of(a[10]);
        check(unlocked([&] {
                  return api.gemv_batched(g.codes, static_cast<float*>(g.row_scales), g.table, g.x, static_cast<float*>(g.y), g.N, g.K, g.batch, g.tail, wp, wn, s);
              }),
              "tetra_gemv_batched");
        return same(a[4]);
    });
}
// problems (array of tetra_problem with the buffer interface), table, stream
FASTCALL(py_gemv_list) {
    return guarded(n, 3, [&] {
        void* table = table_of(a[1], "tetra_gemv_list");
        void* s = stream_of(a[2]);
        Py_buffer b;
        if (PyObject_GetBuffer(a[0], &b, PyBUF_SIMPLE) != 0) throw Failed();
        const auto* problems = static_cast<const tetra_problem*>(b.buf);
        const int count = int(b.len / Py_ssize_t(sizeof(tetra_problem)));
        const int rc = unlocked([&] { return api.gemv_list(problems, count, table, s); });
        PyBuffer_Release(&b);
        check(rc, "tetra_gemv_list");
        return same(Py_None);
    });
}
// workspace, table, stream
FASTCALL(py_grouped_run) {
    return guarded(n, 3, [&] {
        void *ws = pointer(a[0]), *table = table_of(a[1], "tetra_gemv_grouped_run"), *s = stream_of(a[2]);
        check(unlocked([&] { return api.grouped_run(ws, table, s); }), "tetra_gemv_grouped_run");
        return same(Py_None);
    });
}

void need_bytes_type(const at::Tensor& t, size_t nbytes, const char* what) {
    if (t.scalar_type() != at::kByte || !t.is_cuda() || !t.is_contiguous() || (nbytes && size_t(t.numel()) != nbytes))
        fail(PyExc_AssertionError, "%s: codes must be a contiguous uint8 tensor on the device, six bytes per word", what);
}
// codes, table, N, nblocks, out, stream
FASTCALL(py_pack_codes) {
    return guarded(n, 6, [&] {
        const at::Tensor& codes = tensor(a[0]);
        void* table = table_of(a[1], "tetra_pack_codes");
        const int N = integer(a[2]), B = integer(a[3]);
        need_bytes_type(codes, 0, "tetra_pack_codes");
        if (long(codes.numel()) != long(N) * B * 6)
            fail(PyExc_AssertionError, "tetra_pack_codes: codes hold %lld bytes, not %lld", (long long)codes.numel(), (long long)N * B * 6);
        const size_t nbytes = api.codes_bytes(N, B);
        void* s = stream_of(a[5]);
        const at::Tensor out = a[4] == Py_None ? device_empty({int64_t(nbytes)}, at::kByte, codes) : tensor(a[4]);
        if (size_t(out.numel()) < nbytes) fail(PyExc_AssertionError, "tetra_pack_codes: out holds fewer than %zu bytes", nbytes);
        void *src = codes.data_ptr(), *dst = a[4] == Py_None ? out.data_ptr() : need(a[4], nbytes, "tetra_pack_codes", " out");
        check(unlocked([&] { return api.pack_codes(src, table, dst, N, B, s); }), "tetra_pack_codes");
        return a[4] == Py_None ? THPVariable_Wrap(out) : same(a[4]);
    });
}
// packed, table, N, nblocks, want_mg, stream
FASTCALL(py_decode_packed) {
    return guarded(n, 6, [&] {
        const at::Tensor& packed = tensor(a[0]);
        const int N = integer(a[2]), B = integer(a[3]);
        const bool want = truth(a[4]);
        void* src = need(a[0], api.codes_bytes(N, B), "tetra_decode_packed", " packed");
        void* table = table_of(a[1], "tetra_decode_packed");
        void* s = stream_of(a[5]);
        const at::Tensor y = device_empty({N, B, 24}, at::kChar, packed);
        at::Tensor mg;
        if (want) mg = device_empty({N, B, 2}, at::kByte, packed);
        void *dy = y.data_ptr(), *dm = want ? mg.data_ptr() : nullptr;
        check(unlocked([&] { return api.decode_packed(src, table, static_cast<int8_t*>(dy), static_cast<uint8_t*>(dm), N, B, s); }), "tetra_decode_packed");
        return Py_BuildValue("(NN)", THPVariable_Wrap(y), want ? THPVariable_Wrap(mg) : same(Py_None));
    });
}
// w, table, sigma, want_cosine, stream
FASTCALL(py_encode_blocks) {
    return guarded(n, 5, [&] {
        const at::Tensor& w = tensor(a[0]);
        const int64_t count = w.numel() / 24;
        const bool want = truth(a[3]);
        void* table = table_of(a[1], "tetra_encode_blocks");
        void* wp = need(a[0], size_t(4) * 24 * size_t(count), "tetra_encode_blocks", " w");
        void* sigma = need(a[2], size_t(4) * size_t(count), "tetra_encode_blocks", " sigma");
        void* s = stream_of(a[4]);
        const at::Tensor codes = device_empty({count, 6}, at::kByte, w);
        at::Tensor cos;
        if (want) cos = device_empty({count}, at::kFloat, w);
        void *cp = codes.data_ptr(), *fp = want ? cos.data_ptr() : nullptr;
        check(unlocked([&] {
                  return api.encode_blocks(static_cast<float*>(wp), static_cast<float*>(sigma), table, cp, static_cast<float*>(fp), size_t(count), s);
              }),
              "tetra_encode_blocks");
        return Py_BuildValue("(NN)", THPVariable_Wrap(codes), want ? THPVariable_Wrap(cos) : same(Py_None));
    });
}

// q, scale, offset, N, K, G, stream
FASTCALL(py_q4_pack) {
    return guarded(n, 7, [&] {
        const int N = integer(a[3]), K = integer(a[4]), G = integer(a[5]);
        const size_t nbytes = api.q4_packed_bytes(N, K, G);
        if (nbytes == 0) fail(tetra_error, "tetra_q4_packed_bytes: shape rejected (N=%d, K=%d, G=%d)", N, K, G);
        void* q = need(a[0], size_t(N) * size_t(K / 2), "tetra_q4_pack", " q");
        void* scale = need(a[1], 2 * size_t(N) * size_t(K / G), "tetra_q4_pack", " scale");
        void* offset = need(a[2], 2 * size_t(N) * size_t(K / G), "tetra_q4_pack", " offset");
        void* s = stream_of(a[6]);
        const at::Tensor out = device_empty({int64_t(nbytes)}, at::kByte, tensor(a[0]));
        void* dst = out.data_ptr();
        check(unlocked([&] { return api.q4_pack(q, scale, offset, dst, nbytes, N, K, G, s); }), "tetra_q4_pack");
        return THPVariable_Wrap(out);
    });
}
// packed, x, y, N, K, G, batch, stream
FASTCALL(py_q4_gemv) {
    return guarded(n, 8, [&] {
        const int N = integer(a[3]), K = integer(a[4]), G = integer(a[5]), batch = integer(a[6]);
        const size_t nbytes = api.q4_packed_bytes(N, K, G);
        const bool known = nbytes != 0 && batch > 0;  // otherwise the library rejects the shape
        void* packed = known ? need(a[0], nbytes, "tetra_q4_gemv", " packed") : pointer(a[0]);
        void* x = known ? need(a[1], 2 * size_t(batch) * size_t(K), "tetra_q4_gemv", " x") : pointer(a[1]);
        void* y = known ? need(a[2], 4 * size_t(batch) * size_t(N), "tetra_q4_gemv", " y") : pointer(a[2]);
        void* s = stream_of(a[7]);
        check(unlocked([&] { return api.q4_gemv(packed, x, static_cast<float*>(y), N, K, G, batch, s); }), "tetra_q4_gemv");
        return same(a[2]);
    });
}
// packed, ids, out, N, K, G, stream
FASTCALL(py_q4_rows) {
    return guarded(n, 7, [&] {
        const int N = integer(a[3]), K = integer(a[4]), G = integer(a[5]);
        const size_t nbytes = api.q4_packed_bytes(N, K, G);
        const size_t count = size_t(tensor(a[1]).numel());
        void* packed = nbytes ? need(a[0], nbytes, "tetra_q4_rows", " packed") : pointer(a[0]);
        void* ids = need(a[1], 4 * count, "tetra_q4_rows", " ids");
        void* out = need(a[2], K > 0 ? 2 * count * size_t(K) : 0, "tetra_q4_rows", " out");
        void* s = stream_of(a[6]);
        check(unlocked([&] { return api.q4_rows(packed, static_cast<int32_t*>(ids), int(count), out, N, K, G, s); }), "tetra_q4_rows");
        return same(a[2]);
    });
}
// workspace, G, stream
FASTCALL(py_q4_list_run) {
    return guarded(n, 3, [&] {
        void* ws = pointer(a[0]);
        const int G = integer(a[1]);
        void* s = stream_of(a[2]);
        check(unlocked([&] { return api.q4_list_run(ws, G, s); }), "tetra_q4_list_run");
        return same(Py_None);
    });
}

// library path, exception class
FASTCALL(py_setup) {
    return guarded(n, 2, [&] {
        const char* path = PyUnicode_AsUTF8(a[0]);
        if (!path) throw Failed();
        void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
        if (!lib) fail(PyExc_OSError, "%s", dlerror());
        auto get = [&](auto& f, const char* name) {
            f = reinterpret_cast<std::remove_reference_t<decltype(f)>>(dlsym(lib, name));
            if (!f) fail(PyExc_OSError, "%s: no symbol %s", path, name);
        };
        get(api.status_string, "tetra_status_string");
        get(api.table_bytes, "tetra_table_bytes");
        get(api.gemv, "tetra_gemv");
        get(api.gemv_tail, "tetra_gemv_tail");
        get(api.gemv_list, "tetra_gemv_list");
        get(api.grouped_run, "tetra_gemv_grouped_run");
        get(api.gemv_batched, "tetra_gemv_batched");
        get(api.gemv_noalloc, "tetra_gemv_noalloc");
        get(api.codes_bytes, "tetra_codes_bytes");
        get(api.pack_codes, "tetra_pack_codes");
        get(api.decode_packed, "tetra_decode_packed");
        get(api.encode_blocks, "tetra_encode_blocks");
        get(api.q4_packed_bytes, "tetra_q4_packed_bytes");
        get(api.q4_pack, "tetra_q4_pack");
        get(api.q4_gemv, "tetra_q4_gemv");
        get(api.q4_rows, "tetra_q4_rows");
        get(api.q4_list_run, "tetra_q4_list_run");
        Py_XDECREF(tetra_error);
        tetra_error = same(a[1]);
        return same(Py_None);
    });
}

#define METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(setup),        METHOD(gemv),          METHOD(gemv_tail), METHOD(gemv_noalloc), METHOD(gemv_batched),
                         METHOD(gemv_list),    METHOD(grouped_run),   METHOD(pack_codes), METHOD(decode_packed), METHOD(encode_blocks),
                         METHOD(q4_pack),      METHOD(q4_gemv),       METHOD(q4_rows),   METHOD(q4_list_run),  {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", "Argument marshalling of the Tetra C ABI.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", TETRA_BUILT_FOR) != 0) {  // see build.py
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
