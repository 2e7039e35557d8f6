// Native half of the Python binding: the calls a program makes once per layer.  Argument marshalling only -- tensors to
// pointers, the output allocated where none is given, the current stream -- for entry points of libiptq.so, which are looked
// up in the library api.py has loaded (bind()).
//
// Through ctypes a call cost 11 us of host time (torch.empty, current_stream(), data_ptr() per argument, conversion of each
// argument), several times what the device needs for a small layer.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <dlfcn.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "iptq.h"

namespace {

struct Api {
    decltype(&iptq_softmax) softmax;
    decltype(&iptq_gelu) gelu;
    decltype(&iptq_layernorm) layernorm;
    decltype(&iptq_layernorm_gather) layernorm_gather;
    decltype(&iptq_linear_bits) linear_bits;
    decltype(&iptq_gather_rows) gather_rows;
    decltype(&iptq_patchify) patchify;
    decltype(&iptq_attention_block) attention_block;
    decltype(&iptq_mlp_block) mlp_block;
    decltype(&iptq_encoder_block) encoder_block;
    decltype(&iptq_softmax_prepare) softmax_prepare;
    decltype(&iptq_gelu_prepare) gelu_prepare;
    decltype(&iptq_layernorm_prepare) layernorm_prepare;
    decltype(&iptq_op_count) op_count;
    decltype(&iptq_analyze_softmax) analyze_softmax;
    decltype(&iptq_analyze_gelu) analyze_gelu;
    decltype(&iptq_analyze_layernorm) analyze_layernorm;
    decltype(&iptq_sqnr_db) sqnr_db;
    decltype(&iptq_metric_term) metric_term;
    decltype(&iptq_metric_select) metric_select;
} api;
PyObject* raise_error = nullptr;      // Python callable (status, name) that raises IptqError

// Every helper below returns false / nullptr with a Python exception set.
struct Failed {};

[[noreturn]] void fail(PyObject* type, const char* what)
{
    PyErr_SetString(type, what);
    throw Failed{};
}

const at::Tensor& tensor(PyObject* o)
{
    if (!THPVariable_Check(o)) fail(PyExc_AssertionError, "expected a contiguous CUDA tensor");
    return THPVariable_Unpack(o);
}
// a contiguous CUDA tensor
const at::Tensor& device_tensor(PyObject* o)
{
    const at::Tensor& t = tensor(o);
    if (!t.is_cuda() || !t.is_contiguous()) fail(PyExc_AssertionError, "expected a contiguous CUDA tensor");
    return t;
}
template <typename T>
T* dev(PyObject* o)                   // None -> null
{
    return o == Py_None ? nullptr : static_cast<T*>(device_tensor(o).data_ptr());
}
// the bytes of a ctypes structure
template <typename T>
T* host_struct(PyObject* o)
{
    if (o == Py_None) return nullptr;
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw Failed{};
    T* p = static_cast<T*>(b.buf);
    const bool ok = (size_t)b.len >= sizeof(T);
    PyBuffer_Release(&b);             // the structure is kept alive by the caller's reference
    if (!ok) fail(PyExc_TypeError, "expected a ctypes structure of the library");
    return p;
}
// a contiguous host buffer of n floats (a numpy float32 array)
const float* host_floats(PyObject* o, int n)
{
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw Failed{};
    const float* p = static_cast<const float*>(b.buf);
    const bool ok = (size_t)b.len == (size_t)n * sizeof(float);
    PyBuffer_Release(&b);
    if (!ok) fail(PyExc_ValueError, "expected one float32 value per channel");
    return p;
}
int64_t integer(PyObject* o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    return v;
}
void* address(PyObject* o)
{
    if (o == Py_None) return nullptr;
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) throw Failed{};
    return p;
}
double real(PyObject* o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Failed{};
    return v;
}
void rank2(const at::Tensor& t)
{
    if (t.dim() != 2) fail(PyExc_ValueError, "expected a tensor of two dimensions");
}
cudaStream_t stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
// A library call without the interpreter's lock, which a launch into a full queue would otherwise keep from every other thread
// until the device catches up.  The arguments have been read by then.
template <typename... P, typename... A>
int unlocked(int (*call)(P...), A... a)
{
    struct Unlock {
        PyThreadState* state = PyEval_SaveThread();
        ~Unlock() { PyEval_RestoreThread(state); }
    } unlock;
    return call(a...);
}
void check(int rc, const char* what)
{
    if (rc == IPTQ_OK) return;
    PyObject* r = PyObject_CallFunction(raise_error, "is", rc, what);
    Py_XDECREF(r);
    throw Failed{};
}
// the output: the tensor that was handed in, or a new one on the device of `like`
struct Out {
    PyObject* given;
    at::Tensor made;
    void* ptr;
    Out(PyObject* o, at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) : given(o)
    {
        if (o == Py_None) {
            made = at::detail::empty_cuda(sizes, type, like.device(), std::nullopt);
            ptr = made.data_ptr();
        } else {
            ptr = device_tensor(o).data_ptr();
        }
    }
    PyObject* result()
    {
        if (given != Py_None) { Py_INCREF(given); return given; }
        return THPVariable_Wrap(std::move(made));
    }
};

template <PyObject* (*F)(PyObject* const*, Py_ssize_t), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n)
{
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "%d arguments expected, %zd given", N, n);
        return nullptr;
    }
    try {
        return F(args, n);
    } catch (const Failed&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// softmax(scores, consts, bias, out)
PyObject* softmax(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    rank2(x);
    const int64_t period = a[2] == Py_None ? 1 : tensor(a[2]).size(0);
    Out out(a[3], x.sizes(), at::kByte, x);
    check(unlocked(api.softmax, static_cast<const int32_t*>(x.data_ptr()), static_cast<uint8_t*>(out.ptr), x.size(0), (int)x.size(1),
                      dev<int32_t>(a[2]), period, host_struct<iptq_softmax_consts>(a[1]), stream()), "iptq_softmax");
    return out.result();
}

// gelu(x, consts, out)
PyObject* gelu(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    Out out(a[2], x.sizes(), at::kChar, x);
    check(unlocked(api.gelu, static_cast<const int32_t*>(x.data_ptr()), static_cast<int8_t*>(out.ptr), x.numel(),
                   host_struct<iptq_gelu_consts>(a[1]), stream()), "iptq_gelu");
    return out.result();
}

// layernorm(x, gamma_q, beta_q, consts, ptf_shift, out)
PyObject* layernorm(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    rank2(x);
    Out out(a[5], x.sizes(), at::kChar, x);
    check(unlocked(api.layernorm, static_cast<const int8_t*>(x.data_ptr()), static_cast<int8_t*>(out.ptr), x.size(0), (int)x.size(1),
                        dev<int32_t>(a[1]), dev<int32_t>(a[2]), dev<uint8_t>(a[4]), host_struct<iptq_ln_consts>(a[3]), stream()),
          "iptq_layernorm");
    return out.result();
}

// layernorm_gather(x, index, gamma_q, beta_q, consts, ptf_shift, out)
PyObject* layernorm_gather(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    const at::Tensor& index = device_tensor(a[1]);
    rank2(x); rank2(index);
    const int64_t rows = index.size(0), parts = index.size(1), sizes[2] = {rows, parts * x.size(1)};
    Out out(a[6], sizes, at::kChar, x);
    check(unlocked(api.layernorm_gather, static_cast<const int8_t*>(x.data_ptr()), static_cast<int8_t*>(out.ptr), rows, (int)sizes[1],
                               static_cast<const int32_t*>(index.data_ptr()), (int)parts, dev<int32_t>(a[2]), dev<int32_t>(a[3]),
                               dev<uint8_t>(a[5]), host_struct<iptq_ln_consts>(a[4]), stream()), "iptq_layernorm_gather");
    return out.result();
}

// linear(x, w, w_bits, bias, mult, shift, out_zp, residual, residual_rq, out_bits, ws_ptr, ws_bytes, out)
PyObject* linear(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    const at::Tensor& w = device_tensor(a[1]);
    rank2(x);
    const int64_t M = x.size(0), K = x.size(1), N = w.size(0);
    const int64_t sizes[2] = {M, N};
    Out out(a[12], sizes, at::kChar, x);
    check(unlocked(api.linear_bits, static_cast<const int8_t*>(x.data_ptr()), w.data_ptr(), (int)integer(a[2]), dev<int32_t>(a[3]), dev<int32_t>(a[4]),
                          dev<int8_t>(a[5]), (int)integer(a[6]), dev<int8_t>(a[7]), host_struct<iptq_requant>(a[8]),
                          static_cast<int8_t*>(out.ptr), M, (int)N, (int)K, (int)integer(a[9]), address(a[10]),
                          (size_t)integer(a[11]), stream()), "iptq_linear");
    return out.result();
}

// gather_rows(src, index, out)
PyObject* gather_rows(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& src = device_tensor(a[0]);
    const at::Tensor& index = device_tensor(a[1]);
    rank2(src); rank2(index);
    const int64_t sizes[2] = {index.size(0), index.size(1) * src.size(1)};
    Out out(a[2], sizes, at::kChar, src);
    check(unlocked(api.gather_rows, static_cast<const int8_t*>(src.data_ptr()), static_cast<int8_t*>(out.ptr),
                          static_cast<const int32_t*>(index.data_ptr()), index.size(0), (int)index.size(1), (int)src.size(1), stream()),
          "iptq_gather_rows");
    return out.result();
}

// patchify(img, patch, out)
PyObject* patchify(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& img = device_tensor(a[0]);
    const int64_t P = integer(a[1]);
    if (img.dim() != 4 || P < 1) fail(PyExc_ValueError, "expected an image tensor [B, C, H, W] and a positive patch size");
    const int64_t B = img.size(0), C = img.size(1), H = img.size(2), W = img.size(3);
    const int64_t sizes[2] = {B * (H / P) * (W / P), C * P * P};
    Out out(a[2], sizes, at::kChar, img);
    check(unlocked(api.patchify, static_cast<const int8_t*>(img.data_ptr()), static_cast<int8_t*>(out.ptr), B, (int)C, (int)H, (int)W, (int)P,
                       stream()), "iptq_patchify");
    return out.result();
}

// attention_block(q, k, v, sm, out_rq, ws_ptr, ws_bytes, bias, mask_id, out, bias_t)
PyObject* attention_block(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& q = device_tensor(a[0]);
    if (q.dim() != 4) fail(PyExc_ValueError, "expected q of four dimensions [B, H, N, dh]");
    const int64_t B = q.size(0), H = q.size(1), N = q.size(2), dh = q.size(3);
    const int64_t sizes[3] = {B, N, H * dh};
    Out out(a[9], sizes, at::kChar, q);
    check(unlocked(api.attention_block, static_cast<const int8_t*>(q.data_ptr()), dev<int8_t>(a[1]), dev<int8_t>(a[2]), static_cast<int8_t*>(out.ptr),
                              B, (int)H, (int)N, (int)dh, dev<int32_t>(a[7]), dev<int32_t>(a[10]), dev<uint8_t>(a[8]),
                              host_struct<iptq_softmax_consts>(a[3]), host_struct<iptq_requant>(a[4]), address(a[5]),
                              (size_t)integer(a[6]), stream()), "iptq_attention_block");
    return out.result();
}

// mlp_block(x, w1, b1, m1, s1, gelu, ws_ptr, ws_bytes, w2, b2, m2, s2, out_zp, residual, residual_rq, w_bits, out)
PyObject* mlp_block(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    const at::Tensor& w1 = device_tensor(a[1]);
    rank2(x);
    const int64_t M = x.size(0), D = x.size(1), Dh = w1.size(0);
    const int64_t sizes[2] = {M, a[8] == Py_None ? Dh : D};
    Out out(a[16], sizes, at::kChar, x);
    check(unlocked(api.mlp_block, static_cast<const int8_t*>(x.data_ptr()), w1.data_ptr(), dev<int32_t>(a[2]), dev<int32_t>(a[3]), dev<int8_t>(a[4]),
                        host_struct<iptq_gelu_consts>(a[5]), dev<void>(a[8]), dev<int32_t>(a[9]), dev<int32_t>(a[10]),
                        dev<int8_t>(a[11]), (int)integer(a[12]), dev<int8_t>(a[13]), host_struct<iptq_requant>(a[14]),
                        static_cast<int8_t*>(out.ptr), M, (int)D, (int)Dh, (int)integer(a[15]), address(a[6]), (size_t)integer(a[7]),
                        stream()), "iptq_mlp_block");
    return out.result();
}

// encoder_block(x, out, params, ws_ptr, ws_bytes)
PyObject* encoder_block(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    rank2(x);
    Out out(a[1], x.sizes(), at::kChar, x);
    check(unlocked(api.encoder_block, static_cast<const int8_t*>(x.data_ptr()), static_cast<int8_t*>(out.ptr), host_struct<iptq_block_params>(a[2]),
                            address(a[3]), (size_t)integer(a[4]), stream()), "iptq_encoder_block");
    return out.result();
}

// ---------------------------------------------------------------- Unified-Metric analysis (Sec. 3.5)
// The candidates of a layer: those of `variants` that have integer constants at this scale and width.
template <typename Consts, typename Prepare>
int prepare_candidates(PyObject* variants, Consts* consts, int* ids, Prepare&& prepare)
{
    int n = 0;
    PyObject* seq = PySequence_Fast(variants, "expected a sequence of variants");
    if (!seq) throw Failed{};
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(seq); ++i) {
        const int v = (int)PyLong_AsLong(PySequence_Fast_GET_ITEM(seq, i));
        if (v == -1 && PyErr_Occurred()) { Py_DECREF(seq); throw Failed{}; }
        if (n == IPTQ_ANALYZE_MAX_CANDIDATES) { Py_DECREF(seq); fail(PyExc_ValueError, "too many candidates for one layer"); }
        if (prepare(v, &consts[n]) == IPTQ_OK) ids[n++] = v;
    }
    Py_DECREF(seq);
    return n;
}
// [(variant, operation count), ...]
PyObject* candidate_list(int kind, const int* ids, int n, int64_t rows, int64_t row_len)
{
    PyObject* l = PyList_New(n);
    if (!l) throw Failed{};
    for (int i = 0; i < n; ++i) {
        PyObject* t = Py_BuildValue("(id)", ids[i], api.op_count(kind, ids[i], rows, (int)row_len));
        if (!t) { Py_DECREF(l); throw Failed{}; }
        PyList_SET_ITEM(l, i, t);
    }
    return l;
}

// analyze_softmax(scores, in_scale, variants, out_bits, sums_ptr, work_ptr)
PyObject* analyze_softmax(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    rank2(x);
    const double scale = real(a[1]);
    const int bits = (int)integer(a[3]);
    iptq_softmax_consts c[IPTQ_ANALYZE_MAX_CANDIDATES];
    int ids[IPTQ_ANALYZE_MAX_CANDIDATES];
    const int n = prepare_candidates(a[2], c, ids, [&](int v, iptq_softmax_consts* out) {
        return api.softmax_prepare(scale, (int)x.size(1), v == IPTQ_SM_LOG2 ? 4 : bits, (iptq_softmax_variant)v, out);   // 4-bit codes
    });
    if (n)
        check(unlocked(api.analyze_softmax, static_cast<const int32_t*>(x.data_ptr()), x.size(0), (int)x.size(1), scale, c, n,
                                  static_cast<double*>(address(a[4])), address(a[5]), stream()), "iptq_analyze_softmax");
    return candidate_list(IPTQ_LAYER_SOFTMAX, ids, n, x.size(0), x.size(1));
}

// analyze_gelu(x, in_scale, in_bits, out_scale, out_zp, out_bits, variants, sums_ptr, work_ptr)
PyObject* analyze_gelu(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    const double in_scale = real(a[1]), out_scale = real(a[3]);
    const int in_bits = (int)integer(a[2]), zp = (int)integer(a[4]), bits = (int)integer(a[5]);
    iptq_gelu_consts c[IPTQ_ANALYZE_MAX_CANDIDATES];
    int ids[IPTQ_ANALYZE_MAX_CANDIDATES];
    const int n = prepare_candidates(a[6], c, ids, [&](int v, iptq_gelu_consts* out) {
        return api.gelu_prepare(in_scale, in_bits, out_scale, zp, bits, (iptq_gelu_variant)v, out);
    });
    if (n)
        check(unlocked(api.analyze_gelu, static_cast<const int32_t*>(x.data_ptr()), x.numel(), in_scale, out_scale, zp, c, n,
                               static_cast<double*>(address(a[7])), address(a[8]), stream()), "iptq_analyze_gelu");
    return candidate_list(IPTQ_LAYER_GELU, ids, n, x.numel(), 1);
}

// analyze_layernorm(x, gamma, beta (host float32 buffers), out_scale, out_zp, out_bits, variants, ptf_shift, sums_ptr, work_ptr)
PyObject* analyze_layernorm(PyObject* const* a, Py_ssize_t)
{
    const at::Tensor& x = device_tensor(a[0]);
    rank2(x);
    const int dim = (int)x.size(1), zp = (int)integer(a[4]), bits = (int)integer(a[5]);
    const float *gamma = host_floats(a[1], dim), *beta = host_floats(a[2], dim);
    const double out_scale = real(a[3]);
    std::vector<int32_t> q((size_t)2 * dim);
    int32_t *gq = q.data(), *bq = q.data() + dim;
    iptq_ln_consts c[IPTQ_ANALYZE_MAX_CANDIDATES];
    int ids[IPTQ_ANALYZE_MAX_CANDIDATES];
    const int n = prepare_candidates(a[6], c, ids, [&](int v, iptq_ln_consts* out) {
        if (v == IPTQ_LN_PTF && a[7] == Py_None) return (int)IPTQ_ERR_NULL;      // a candidate for inputs with such factors alone
        if (out != c && v >= IPTQ_LN_SHIFT && v <= IPTQ_LN_PTF) {       // the variant is all that differs between the candidates
            *out = c[0];
            out->variant = v;
            return (int)IPTQ_OK;
        }
        check(api.layernorm_prepare(dim, gamma, beta, out_scale, zp, bits, (iptq_ln_variant)v, gq, bq, out), "iptq_layernorm_prepare");
        return (int)IPTQ_OK;
    });
    if (n)
        check(unlocked(api.analyze_layernorm, static_cast<const int8_t*>(x.data_ptr()), x.size(0), dim, gamma, beta, gq, bq, dev<uint8_t>(a[7]),
                                    out_scale, zp, c, n, static_cast<double*>(address(a[8])), address(a[9]), stream()),
              "iptq_analyze_layernorm");
    return candidate_list(IPTQ_LAYER_LAYERNORM, ids, n, x.size(0), dim);
}

// metric_scores(host sums ptr, first slot, operation counts, c_unit)
//   -> (index of the best term, [(sum_x2, sum_err2, sqnr_db, term), ...])
PyObject* metric_scores(PyObject* const* a, Py_ssize_t)
{
    const double* sums = static_cast<const double*>(address(a[0])) + 2 * integer(a[1]);
    const double c_unit = real(a[3]);
    const Py_ssize_t n = PyList_Size(a[2]);
    if (n < 0) throw Failed{};
    std::vector<double> terms((size_t)n);
    PyObject* l = PyList_New(n);
    if (!l) throw Failed{};
    for (Py_ssize_t i = 0; i < n; ++i) {
        const double x2 = sums[2 * i], e2 = sums[2 * i + 1], q = api.sqnr_db(x2, e2);
        terms[(size_t)i] = api.metric_term(q, e2, PyFloat_AsDouble(PyList_GET_ITEM(a[2], i)), c_unit);
        PyObject* t = Py_BuildValue("(dddd)", x2, e2, q, terms[(size_t)i]);
        if (!t) { Py_DECREF(l); throw Failed{}; }
        PyList_SET_ITEM(l, i, t);
    }
    return Py_BuildValue("(iN)", api.metric_select(terms.data(), (int)n), l);
}

// bind(dlopen handle of libiptq.so, raise_error)
PyObject* bind(PyObject* const* a, Py_ssize_t)
{
    void* h = address(a[0]);
    auto get = [&](auto& fn, const char* name) {
        fn = reinterpret_cast<std::remove_reference_t<decltype(fn)>>(dlsym(h, name));
        if (!fn) fail(PyExc_ImportError, name);
    };
    get(api.softmax, "iptq_softmax"); get(api.gelu, "iptq_gelu"); get(api.layernorm, "iptq_layernorm"); get(api.layernorm_gather, "iptq_layernorm_gather");
    get(api.linear_bits, "iptq_linear_bits"); get(api.gather_rows, "iptq_gather_rows"); get(api.patchify, "iptq_patchify");
    get(api.attention_block, "iptq_attention_block"); get(api.mlp_block, "iptq_mlp_block");
    get(api.encoder_block, "iptq_encoder_block");
    get(api.softmax_prepare, "iptq_softmax_prepare"); get(api.gelu_prepare, "iptq_gelu_prepare");
    get(api.layernorm_prepare, "iptq_layernorm_prepare"); get(api.op_count, "iptq_op_count");
    get(api.analyze_softmax, "iptq_analyze_softmax"); get(api.analyze_gelu, "iptq_analyze_gelu");
    get(api.analyze_layernorm, "iptq_analyze_layernorm");
    get(api.sqnr_db, "iptq_sqnr_db"); get(api.metric_term, "iptq_metric_term"); get(api.metric_select, "iptq_metric_select");
    Py_INCREF(a[1]);
    Py_XSETREF(raise_error, a[1]);
    Py_RETURN_NONE;
}

#define IPTQ_ENTRY(f, n) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<f, n>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    IPTQ_ENTRY(bind, 2), IPTQ_ENTRY(softmax, 4), IPTQ_ENTRY(gelu, 3), IPTQ_ENTRY(layernorm, 6), IPTQ_ENTRY(layernorm_gather, 7), IPTQ_ENTRY(linear, 13),
    IPTQ_ENTRY(gather_rows, 3), IPTQ_ENTRY(patchify, 3), IPTQ_ENTRY(attention_block, 11), IPTQ_ENTRY(mlp_block, 17),
    IPTQ_ENTRY(encoder_block, 5), IPTQ_ENTRY(analyze_softmax, 6), IPTQ_ENTRY(analyze_gelu, 9), IPTQ_ENTRY(analyze_layernorm, 10),
    IPTQ_ENTRY(metric_scores, 4), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
