// Native argument marshalling of the hot entry points (api.py): tensors in, output allocation, one C ABI call (without the GIL).  The
// same work through ctypes costs 10-20 us a call, more than a small layer takes on the GPU.  No arithmetic of the method and no decision
// about it is made here.
#include <ATen/cuda/EmptyTensor.h>
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "bitserial.h"

namespace {

struct Fail {};      // a Python error is set

const at::Tensor& tensor(PyObject* o)
{
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a tensor"); throw Fail(); }
    return THPVariable_Unpack(o);
}
void* pointer(const at::Tensor& t)
{
    if (!t.is_cuda() || !t.is_contiguous()) { PyErr_SetString(PyExc_ValueError, "expected a contiguous CUDA tensor"); throw Fail(); }
    return t.data_ptr();
}
// The library call runs without the GIL: a launch can wait for room in the stream's queue.
struct NoGil {
    PyThreadState* state = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(state); }
};
void* pointer_or_null(PyObject* o) { return o == Py_None ? nullptr : pointer(tensor(o)); }
int integer(PyObject* o)
{
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Fail();
    if (v > 0x7fffffffL || v < -0x7fffffffL - 1) { PyErr_SetString(PyExc_OverflowError, "integer argument out of range"); throw Fail(); }
    return static_cast<int>(v);
}
float real(PyObject* o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Fail();
    return static_cast<float>(v);
}
// `stream` argument: None (the current stream) or a torch stream.
void* stream_of(PyObject* o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* s = PyObject_GetAttrString(o, "cuda_stream");
    if (!s) throw Fail();
    void* p = reinterpret_cast<void*>(PyLong_AsUnsignedLongLong(s));
    Py_DECREF(s);
    if (PyErr_Occurred()) throw Fail();
    return p;
}
at::Tensor words(at::IntArrayRef shape, const at::Tensor& like)
{
    return at::detail::empty_cuda(shape, at::kInt, like.device(), std::nullopt);
}
PyObject* give(const at::Tensor& t) { return t.defined() ? THPVariable_Wrap(t) : Py_NewRef(Py_None); }

PyObject* result(int status, const at::Tensor& a, const at::Tensor& b)
{
    return Py_BuildValue("(iNN)", status, give(a), give(b));
}

void need(Py_ssize_t got, Py_ssize_t want)
{
    if (got != want) { PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, got); throw Fail(); }
}

template <typename F>
PyObject* guarded(F f)
{
    try {
        return f();
    } catch (const Fail&) {
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

// Prepared filters of three bits for narrow activations hold both forms, int8 and nibbles (tc_prepare_weights in api.py): the nibbles where they are
// wanted, with the sign that says so.
const int8_t* prepared(const at::Tensor& t, int O, int C, int R, int S, int w_bits, int a_bits, int& w_sign)
{
    const int8_t* p = static_cast<const int8_t*>(pointer(t));
    if (w_bits != 3 || a_bits > 2 || w_sign != BS_SIGNED) return p;
    const size_t bytes = bs_tc_weights_bytes(O, C, R, S);
    if (bytes == 0 || t.nbytes() != 2 * bytes) return p;
    w_sign = BS_SIGNED_NIBBLES;
    return p + bytes;
}

void mismatch(const char* what) { PyErr_SetString(PyExc_ValueError, what); throw Fail(); }

// act, wgt, C, stride, pad, a_sign, w_sign, scale, bias, relu, out_bits, out_sign, residual, res_scale, res_bits, res_sign, res_c_offset,
// res_c_total, out_i32, want_i32, i32_layout, out_packed, out_c_offset, out_c_total, workspace, wgt_tc, chained, stream
PyObject* conv2d(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&] {
        need(n, 28);
        const at::Tensor &act = tensor(a[0]), &wgt = tensor(a[1]);
        if (act.dim() != 5 || wgt.dim() != 5) mismatch("packed tensors of five dimensions expected");
        bs_conv_params p{};
        p.C = integer(a[2]);
        if (act.size(3) != wgt.size(3) || act.size(3) != (p.C + 31) / 32) mismatch("channel words of activations and weights disagree");
        p.N = static_cast<int>(act.size(0)); p.H = static_cast<int>(act.size(1)); p.W = static_cast<int>(act.size(2));
        p.a_bits = static_cast<int>(act.size(4));
        p.O = static_cast<int>(wgt.size(0)); p.R = static_cast<int>(wgt.size(1)); p.S = static_cast<int>(wgt.size(2));
        p.w_bits = static_cast<int>(wgt.size(4));
        p.stride = integer(a[3]); p.pad = integer(a[4]); p.a_sign = integer(a[5]); p.w_sign = integer(a[6]);
        if (p.stride == 0) mismatch("stride is zero");
        p.scale = static_cast<const float*>(pointer_or_null(a[7])); p.bias = static_cast<const float*>(pointer_or_null(a[8]));
        p.relu = PyObject_IsTrue(a[9]);
        p.out_bits = integer(a[10]); p.out_sign = integer(a[11]);
        p.residual = static_cast<const uint32_t*>(pointer_or_null(a[12]));
        p.res_scale = real(a[13]); p.res_bits = integer(a[14]); p.res_sign = integer(a[15]); p.res_c_offset = integer(a[16]);
        p.res_c_total = integer(a[17]);
        if (p.res_c_total == 0) p.res_c_total = p.res_c_offset + p.O;
        p.i32_layout = integer(a[20]);
        p.out_c_offset = integer(a[22]); p.out_c_total = integer(a[23]);
        auto fdiv = [](int x, int y) { return x / y - (x % y != 0 && (x < 0) != (y < 0)); };
        const int64_t P = fdiv(p.H + 2 * p.pad - p.R, p.stride) + 1, Q = fdiv(p.W + 2 * p.pad - p.S, p.stride) + 1;
        const uint32_t* ap = static_cast<const uint32_t*>(pointer(act));
        const int8_t* tc = a[25] == Py_None ? nullptr : prepared(tensor(a[25]), p.O, p.C, p.R, p.S, p.w_bits, p.a_bits, p.w_sign);
        const uint32_t* wp = tc ? nullptr : static_cast<const uint32_t*>(pointer(wgt));
        at::Tensor i32, packed;
        if (a[18] != Py_None) i32 = tensor(a[18]);
        else if (PyObject_IsTrue(a[19])) i32 = p.i32_layout == BS_NCHW ? words({p.N, p.O, P, Q}, act) : words({p.N, P, Q, p.O}, act);
        if (p.out_bits > 0) {
            if (p.out_c_total == 0) p.out_c_total = p.out_c_offset + p.O;
            if (a[21] != Py_None) {
                packed = tensor(a[21]);
            } else {
                const int64_t ow = (p.out_c_total + 31) / 32;
                packed = words({p.N, P, Q, ow, p.out_bits}, act);
                // the layer overwrites its own channel words in full; words of other channels of a wider tensor start at zero
                if (ow != (p.O + 31) / 32) packed.zero_();
            }
        }
        void* st = stream_of(a[27]);
        int32_t* ip = i32.defined() ? static_cast<int32_t*>(pointer(i32)) : nullptr;
        uint32_t* op = packed.defined() ? static_cast<uint32_t*>(pointer(packed)) : nullptr;
        void* ws = tc || a[24] == Py_None ? nullptr : pointer(tensor(a[24]));
        const size_t ws_bytes = ws ? tensor(a[24]).nbytes() : 0;
        const bool use_ws = !tc && a[24] != Py_None, chained = PyObject_IsTrue(a[26]);
        int rc;
        {
            NoGil free;
            rc = tc ? (chained ? bitserial_conv2d_tc_chained(ap, tc, &p, ip, op, st) : bitserial_conv2d_tc(ap, tc, &p, ip, op, st))
                 : use_ws ? bitserial_conv2d_ws(ap, wp, &p, ip, op, ws, ws_bytes, st)
                          : bitserial_conv2d(ap, wp, &p, ip, op, st);
        }
        return result(rc, i32, packed);
    });
}

// a, w (packed rows) or w_tc, N, w_bits (both -1 with packed rows), K, a_sign, w_sign, scale, bias, relu, out_bits, out_sign, out_i32, want_i32,
// out_packed, workspace, stream
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&] {
        need(n, 17);
        const at::Tensor &x = tensor(a[0]), &w = tensor(a[1]);
        if (x.dim() != 3) mismatch("packed rows of three dimensions expected");
        const int M = static_cast<int>(x.size(0)), a_bits = static_cast<int>(x.size(2)), K = integer(a[4]);
        int N = integer(a[2]), w_bits = integer(a[3]);
        const bool tc = N >= 0;
        if (!tc) {
            if (w.dim() != 3) mismatch("packed rows of three dimensions expected");
            if (x.size(1) != w.size(1) || x.size(1) != (static_cast<int64_t>(K) + 31) / 32) mismatch("reduction words of the operands disagree");
            N = static_cast<int>(w.size(0)); w_bits = static_cast<int>(w.size(2));
        }
        const int a_sign = integer(a[5]);
        int w_sign = integer(a[6]);
        const float *scale = static_cast<const float*>(pointer_or_null(a[7])), *bias = static_cast<const float*>(pointer_or_null(a[8]));
        const int relu = PyObject_IsTrue(a[9]), out_bits = integer(a[10]), out_sign = integer(a[11]);
        const uint32_t* xp = static_cast<const uint32_t*>(pointer(x));
        const void* wp = tc ? prepared(w, N, K, 1, 1, w_bits, a_bits, w_sign) : pointer(w);
        at::Tensor i32, packed;
        if (a[12] != Py_None) i32 = tensor(a[12]);
        else if (PyObject_IsTrue(a[13])) i32 = words({M, N}, x);
        if (out_bits > 0) packed = a[14] != Py_None ? tensor(a[14]) : words({M, (static_cast<int64_t>(N) + 31) / 32, out_bits}, x);
        void* st = stream_of(a[16]);
        int32_t* ip = i32.defined() ? static_cast<int32_t*>(pointer(i32)) : nullptr;
        uint32_t* op = packed.defined() ? static_cast<uint32_t*>(pointer(packed)) : nullptr;
        const bs_sign_t as = static_cast<bs_sign_t>(a_sign), wsn = static_cast<bs_sign_t>(w_sign), os = static_cast<bs_sign_t>(out_sign);
        const bool use_ws = !tc && a[15] != Py_None;
        void* ws = use_ws ? pointer(tensor(a[15])) : nullptr;
        const size_t ws_bytes = use_ws ? tensor(a[15]).nbytes() : 0;
        const int8_t* w8 = static_cast<const int8_t*>(wp);
        const uint32_t* w32 = static_cast<const uint32_t*>(wp);
        int rc;
        {
            NoGil free;
            rc = tc ? bitserial_gemm_tc(xp, w8, M, N, K, a_bits, as, w_bits, wsn, scale, bias, relu, out_bits, os, ip, op, st)
                 : use_ws ? bitserial_gemm_ws(xp, w32, M, N, K, a_bits, as, w_bits, wsn, scale, bias, relu, out_bits, os, ip, op, ws, ws_bytes, st)
                          : bitserial_gemm(xp, w32, M, N, K, a_bits, as, w_bits, wsn, scale, bias, relu, out_bits, os, ip, op, st);
        }
        return result(rc, i32, packed);
    });
}

// x, act_scale, a_bits, a_sign, layout, out, stream
PyObject* bitpack(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&] {
        need(n, 7);
        const at::Tensor& x = tensor(a[0]);
        if (x.scalar_type() != at::kFloat && x.scalar_type() != at::kChar) mismatch("x must be float32 or int8");
        if (x.dim() != 4) mismatch("x must have four dimensions");
        const int bits = integer(a[2]), sign = integer(a[3]), layout = integer(a[4]);
        const bool nchw = layout == BS_NCHW;
        const int64_t N = x.size(0), C = x.size(nchw ? 1 : 3), H = x.size(nchw ? 2 : 1), W = x.size(nchw ? 3 : 2), Cw = (C + 31) / 32;
        const float scale = real(a[1]);
        const void* xp = pointer(x);
        const at::Tensor out = a[5] != Py_None ? tensor(a[5]) : words({N, H, W, Cw, bits > 0 ? bits : 1}, x);
        uint32_t* op = static_cast<uint32_t*>(pointer(out));
        void* st = stream_of(a[6]);
        const bool f32 = x.scalar_type() == at::kFloat;
        int rc;
        {
            NoGil free;
            rc = bitpack_activations(xp, f32, static_cast<bs_layout_t>(layout), static_cast<int>(N), static_cast<int>(C), static_cast<int>(H),
                                     static_cast<int>(W), scale, bits, static_cast<bs_sign_t>(sign), op, st);
        }
        at::Tensor view = out;
        if (rc == BS_OK && a[5] != Py_None) view = out.view({N, H, W, Cw, bits});
        return result(rc, view, at::Tensor());
    });
}

// x, act_scale, a_bits, out, operands (of a sequence), stream
PyObject* bitpack_operands(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&] {
        need(n, 6);
        const at::Tensor &x = tensor(a[0]), &out = tensor(a[3]);
        if (x.scalar_type() != at::kFloat) mismatch("x must be float32");
        if (x.dim() != 4) mismatch("x must have four dimensions");
        const float scale = real(a[1]);
        const int bits = integer(a[2]);
        const float* xp = static_cast<const float*>(pointer(x));
        uint32_t* op = static_cast<uint32_t*>(pointer(out));
        const bs_operand_tensor* to = reinterpret_cast<const bs_operand_tensor*>(PyLong_AsUnsignedLongLong(a[4]));
        if (PyErr_Occurred()) throw Fail();
        void* st = stream_of(a[5]);
        int rc;
        {
            NoGil free;
            rc = bitpack_activations_operands(xp, static_cast<int>(x.size(0)), static_cast<int>(x.size(1)), static_cast<int>(x.size(2)),
                                              static_cast<int>(x.size(3)), scale, bits, op, to, st);
        }
        return result(rc, at::Tensor(), at::Tensor());
    });
}

// sequence, stream, ready (an operand tensor of it, or None)
PyObject* sequence_run(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&] {
        need(n, 3);
        bs_sequence* s = reinterpret_cast<bs_sequence*>(PyLong_AsUnsignedLongLong(a[0]));
        if (PyErr_Occurred()) throw Fail();
        void* st = stream_of(a[1]);
        const bs_operand_tensor* ready = a[2] == Py_None ? nullptr : reinterpret_cast<const bs_operand_tensor*>(PyLong_AsUnsignedLongLong(a[2]));
        if (PyErr_Occurred()) throw Fail();
        int rc;
        {
            NoGil free;
            rc = bs_sequence_run_ready(s, ready, st);
        }
        return PyLong_FromLong(rc);
    });
}

// dicts, values, addresses (three tuples): whether the dicts, one after the other, still hold these very objects, the tensors among them
// (address not None) at these addresses.  A pass asks this of a few hundred entries (362: 2.8 us,
// while its first kernel runs).
PyObject* unchanged(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&] {
        need(n, 3);
        if (!PyTuple_Check(a[0]) || !PyTuple_Check(a[1]) || !PyTuple_Check(a[2]) || PyTuple_GET_SIZE(a[1]) != PyTuple_GET_SIZE(a[2])) mismatch("three tuples expected, two of one length");
        const Py_ssize_t count = PyTuple_GET_SIZE(a[1]);
        Py_ssize_t at = 0;
        for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(a[0]); ++i) {
            PyObject *d = PyTuple_GET_ITEM(a[0], i), *key, *value;
            if (!PyDict_Check(d)) mismatch("dict expected");
            Py_ssize_t pos = 0;
            while (PyDict_Next(d, &pos, &key, &value)) {
                if (at == count || value != PyTuple_GET_ITEM(a[1], at)) Py_RETURN_FALSE;
                PyObject* address = PyTuple_GET_ITEM(a[2], at++);
                if (address == Py_None) continue;
                const at::Tensor& t = THPVariable_CheckExact(value) ? THPVariable_Unpack(value) : tensor(value);
                if (t.const_data_ptr() != PyLong_AsVoidPtr(address)) Py_RETURN_FALSE;
            }
        }
        return PyBool_FromLong(at == count);
    });
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(conv2d), FAST(gemm), FAST(bitpack), FAST(bitpack_operands), FAST(sequence_run), FAST(unchanged), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module); }
