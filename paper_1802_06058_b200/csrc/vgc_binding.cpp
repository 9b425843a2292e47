// Python binding of the C ABI as a CPython extension module (_vgc_native): unpacks torch tensors, checks them and
// calls the entry points of libvgc.so.
//
// A step of a small network is a dozen calls of a few microseconds of GPU work each, so what a call costs on the host
// is what it costs: with ctypes a call took 6 - 10 us of interpreter time (argument objects, tensor attributes, one
// structure per message: 100 us for the decode of 64 messages), here it takes about 1 us beside the kernel launches.
// Arguments are positional (the Python functions of the package give them names and defaults); status codes are
// returned as integers and turned into exceptions there.  The GIL is released around the library call.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "vgc.h"

namespace {

// a Python exception has been set
struct Raised {};

[[noreturn]] void raise(PyObject *type, const char *fmt, const char *a = "", const char *b = "")
{
    PyErr_Format(type, fmt, a, b);
    throw Raised{};
}

struct Ref {                                             // owned reference
    PyObject *p;
    explicit Ref(PyObject *o) : p(o) { if (!p) throw Raised{}; }
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
};

PyObject *s_words, *s_group_exp, *s_counters, *s_mask, *s_capacity, *s_K, *s_struct, *s_view, *s_cuda_stream;
PyObject *t_message = nullptr, *t_hybrid = nullptr;      // MessageBuffers, HybridMessageBuffers

const at::Tensor &tensor(PyObject *o, const char *name)
{
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "%s must be a CUDA tensor", name);
    return THPVariable_Unpack(o);
}

const char *type_name(at::ScalarType t)
{
    return t == at::kFloat ? "torch.float32" : t == at::kInt ? "torch.int32" : "torch.uint8";
}

void *dev(PyObject *o, at::ScalarType type, const char *name)
{
    const at::Tensor &t = tensor(o, name);
    if (!t.is_cuda()) raise(PyExc_TypeError, "%s must be a CUDA tensor", name);
    if (t.scalar_type() != type) {
        PyErr_Format(PyExc_TypeError, "%s must be %s, got torch.%s", name, type_name(type), c10::toString(t.scalar_type()));
        throw Raised{};
    }
    if (!t.is_contiguous()) raise(PyExc_ValueError, "%s must be contiguous", name);
    return t.data_ptr();
}
float *dev_f(PyObject *o, const char *name) { return static_cast<float *>(dev(o, at::kFloat, name)); }
uint32_t *dev_u(PyObject *o, const char *name) { return static_cast<uint32_t *>(dev(o, at::kInt, name)); }

void *host(PyObject *o, at::ScalarType type, const char *name)
{
    if (THPVariable_Check(o)) {
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.is_cuda() && t.scalar_type() == type && t.is_contiguous()) return t.data_ptr();
    }
    raise(PyExc_TypeError, "%s must be a contiguous CPU tensor of %s", name, type_name(type));
}

void workspace(PyObject *o, void **p, size_t *bytes)
{
    *p = nullptr;
    *bytes = 0;
    if (o == Py_None) return;
    const at::Tensor &t = tensor(o, "workspace");
    if (!t.is_cuda() || !t.is_contiguous()) raise(PyExc_ValueError, "workspace must be a contiguous CUDA tensor");
    *p = t.data_ptr();
    *bytes = (size_t)t.numel() * t.element_size();
}

// whatever float() takes
double number(PyObject *o)
{
    if (PyFloat_CheckExact(o)) return PyFloat_AS_DOUBLE(o);
    Ref f(PyNumber_Float(o));
    return PyFloat_AS_DOUBLE(f.p);
}
long long integer(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
}
int truth(PyObject *o)
{
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw Raised{};
    return v;
}
// None: the current stream of the current device; an object with .cuda_stream; or the handle as a number
vgc_stream_t stream_of(PyObject *o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyLong_Check(o)) return reinterpret_cast<vgc_stream_t>(PyLong_AsVoidPtr(o));
    PyObject *h = PyObject_GetAttr(o, s_cuda_stream);
    if (!h) {
        PyErr_Clear();
        h = PyNumber_Long(o);
    }
    Ref handle(h);
    void *p = PyLong_AsVoidPtr(handle.p);
    if (!p && PyErr_Occurred()) throw Raised{};
    return static_cast<vgc_stream_t>(p);
}

// a pair (rows, columns) of integers
void pair(PyObject *o, int *a, int *b)
{
    Ref seq(PySequence_Fast(o, "a pair of integers is wanted"));
    if (PySequence_Fast_GET_SIZE(seq.p) != 2) raise(PyExc_ValueError, "a pair of integers is wanted");
    *a = (int)integer(PySequence_Fast_GET_ITEM(seq.p, 0));
    *b = (int)integer(PySequence_Fast_GET_ITEM(seq.p, 1));
}

// the bytes of a ctypes structure that a Python object's own struct() / view() made
template <class T>
T from_ctypes(PyObject *owner, PyObject *method)
{
    Ref made(PyObject_CallMethodNoArgs(owner, method));
    Py_buffer buf;
    if (PyObject_GetBuffer(made.p, &buf, PyBUF_SIMPLE)) throw Raised{};
    T v;
    const bool fits = (size_t)buf.len == sizeof(T);
    if (fits) memcpy(&v, buf.buf, sizeof(T));
    PyBuffer_Release(&buf);
    if (!fits) raise(PyExc_TypeError, "unexpected message structure");
    return v;
}

char *data_of(PyObject *owner, PyObject *attr)
{
    Ref t(PyObject_GetAttr(owner, attr));
    return static_cast<char *>(tensor(t.p, "message buffer").data_ptr());
}
long long int_attr(PyObject *owner, PyObject *attr)
{
    Ref v(PyObject_GetAttr(owner, attr));
    return integer(v.p);
}
// optional tensor attribute: its address and number of elements
char *optional_data(PyObject *owner, PyObject *attr, int64_t *numel)
{
    Ref t(PyObject_GetAttr(owner, attr));
    *numel = -1;
    if (t.p == Py_None) return nullptr;
    const at::Tensor &x = tensor(t.p, "mask");
    *numel = x.numel();
    return static_cast<char *>(x.data_ptr());
}

vgc_message message_of(PyObject *o)
{
    if (Py_TYPE(o) != reinterpret_cast<PyTypeObject *>(t_message)) return from_ctypes<vgc_message>(o, s_struct);
    int64_t ignored;
    char *c = data_of(o, s_counters);
    vgc_message m;
    m.words = reinterpret_cast<uint32_t *>(data_of(o, s_words));
    m.capacity = (uint32_t)int_attr(o, s_capacity);
    m.group_exp = reinterpret_cast<int32_t *>(data_of(o, s_group_exp));
    m.nnz = reinterpret_cast<uint32_t *>(c);
    m.n_criterion = reinterpret_cast<uint32_t *>(c + 4);
    m.n_dropped = reinterpret_cast<uint32_t *>(c + 8);
    m.mask = reinterpret_cast<uint8_t *>(optional_data(o, s_mask, &ignored));
    m.dev_status = reinterpret_cast<uint32_t *>(c + 12);
    return m;
}

vgc_hybrid_message hybrid_message_of(PyObject *o)
{
    if (Py_TYPE(o) != reinterpret_cast<PyTypeObject *>(t_hybrid)) return from_ctypes<vgc_hybrid_message>(o, s_struct);
    int64_t ignored;
    char *c = data_of(o, s_counters);
    vgc_hybrid_message m;
    m.words = reinterpret_cast<uint32_t *>(data_of(o, s_words));
    m.capacity = (uint32_t)int_attr(o, s_capacity);
    m.nnz = reinterpret_cast<uint32_t *>(c);
    m.mask = reinterpret_cast<uint8_t *>(optional_data(o, s_mask, &ignored));
    m.dev_status = reinterpret_cast<uint32_t *>(c + 4);
    return m;
}

// W message views: buffers objects, or tuples (words, nnz[, group_exp]) of tensors
void views_of(PyObject *messages, bool hybrid, std::vector<vgc_message_view> &views)
{
    Ref seq(PySequence_Fast(messages, "messages must be a sequence"));
    const Py_ssize_t W = PySequence_Fast_GET_SIZE(seq.p);
    views.resize((size_t)(W > 0 ? W : 1));
    PyTypeObject *type = reinterpret_cast<PyTypeObject *>(hybrid ? t_hybrid : t_message);
    for (Py_ssize_t w = 0; w < W; ++w) {
        PyObject *m = PySequence_Fast_GET_ITEM(seq.p, w);
        vgc_message_view &v = views[(size_t)w];
        if (Py_TYPE(m) == type) {
            Ref t(PyObject_GetAttr(m, s_words));
            const at::Tensor &words = tensor(t.p, "words");
            const long long cap = int_attr(m, s_capacity), have = words.numel();
            v.words = static_cast<const uint32_t *>(words.data_ptr());
            v.max_words = (uint32_t)(cap < have ? cap : have);
            v.nnz = reinterpret_cast<const uint32_t *>(data_of(m, s_counters));
            v.group_exp = hybrid ? nullptr : reinterpret_cast<const int32_t *>(data_of(m, s_group_exp));
        } else if (PyObject_TypeCheck(m, type)) {
            v = from_ctypes<vgc_message_view>(m, s_view);
        } else {
            Ref parts(PySequence_Fast(m, "a message is a buffers object or a tuple of tensors"));
            if (PySequence_Fast_GET_SIZE(parts.p) != (hybrid ? 2 : 3))
                raise(PyExc_ValueError, hybrid ? "a message is (words, nnz)" : "a message is (words, nnz, group_exp)");
            PyObject *words = PySequence_Fast_GET_ITEM(parts.p, 0);
            v.words = dev_u(words, "words");
            v.nnz = dev_u(PySequence_Fast_GET_ITEM(parts.p, 1), "nnz");
            v.group_exp = hybrid ? nullptr
                                 : reinterpret_cast<const int32_t *>(dev_u(PySequence_Fast_GET_ITEM(parts.p, 2), "group_exp"));
            v.max_words = (uint32_t)THPVariable_Unpack(words).numel();
        }
    }
    views.resize((size_t)W);
}

PyObject *status_object(int st) { return PyLong_FromLong(st); }

#define VGC_CALL(expr)                  \
    int st_;                            \
    Py_BEGIN_ALLOW_THREADS st_ = (expr); \
    Py_END_ALLOW_THREADS return status_object(st_)

typedef PyObject *const *Args;

// x, delta, scale, S, accumulate, ws, stream
PyObject *sqgrad_linear(Args a)
{
    const at::Tensor &x = tensor(a[0], "x"), &d = tensor(a[1], "delta"), &S = tensor(a[3], "S");
    if (x.dim() != 2 || d.dim() != 2) raise(PyExc_ValueError, "x and delta must have two dimensions");
    const int64_t B = x.size(0), in = x.size(1), out = d.size(1);
    if (B != d.size(0) || S.numel() != in * out) raise(PyExc_ValueError, "shape mismatch");
    void *ws;
    size_t wsb;
    workspace(a[5], &ws, &wsb);
    const float *xp = dev_f(a[0], "x"), *dp = dev_f(a[1], "delta");
    const float scale = (float)number(a[2]);
    const int acc = truth(a[4]);
    float *Sp = dev_f(a[3], "S");
    vgc_stream_t st = stream_of(a[6]);
    VGC_CALL(vgc_sqgrad_linear(xp, dp, (int)B, (int)in, (int)out, scale, acc, Sp, ws, wsb, st));
}

struct ConvShape {
    int B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw;
    int64_t Ho, Wo;
};
ConvShape conv_shape(const at::Tensor &x, const at::Tensor &d, PyObject *kernel, PyObject *stride, PyObject *padding)
{
    if (x.dim() != 4 || d.dim() != 4) raise(PyExc_ValueError, "x and delta must have four dimensions");
    ConvShape c;
    c.B = (int)x.size(0); c.C = (int)x.size(1); c.H = (int)x.size(2); c.W = (int)x.size(3);
    c.Cout = (int)d.size(1); c.Ho = d.size(2); c.Wo = d.size(3);
    pair(kernel, &c.Kh, &c.Kw);
    pair(stride, &c.sh, &c.sw);
    pair(padding, &c.ph, &c.pw);
    return c;
}
// Python's floor division, so that impossible geometries (kernel larger than the image) are refused alike
int64_t out_size(int64_t in, int64_t pad, int64_t k, int64_t stride)
{
    if (stride == 0) raise(PyExc_ZeroDivisionError, "integer division or modulo by zero");
    const int64_t n = in + 2 * pad - k;
    int64_t q = n / stride;
    if (n % stride != 0 && ((n < 0) != (stride < 0))) --q;
    return q + 1;
}
bool geometry_fits(const ConvShape &c)
{
    return c.Ho == out_size(c.H, c.ph, c.Kh, c.sh) && c.Wo == out_size(c.W, c.pw, c.Kw, c.sw);
}

// x, delta, kernel, stride, padding, scale, S, accumulate, ws, stream, exact
PyObject *sqgrad_conv(Args a)
{
    const at::Tensor &x = tensor(a[0], "x"), &d = tensor(a[1], "delta"), &S = tensor(a[6], "S");
    const ConvShape c = conv_shape(x, d, a[2], a[3], a[4]);
    if (c.B != d.size(0) || S.numel() != (int64_t)c.Cout * c.C * c.Kh * c.Kw) raise(PyExc_ValueError, "shape mismatch");
    if (!geometry_fits(c)) raise(PyExc_ValueError, "delta spatial shape does not match the convolution geometry");
    void *ws;
    size_t wsb;
    workspace(a[8], &ws, &wsb);
    const float *xp = dev_f(a[0], "x"), *dp = dev_f(a[1], "delta");
    const float scale = (float)number(a[5]);
    const int acc = truth(a[7]);
    float *Sp = dev_f(a[6], "S");
    vgc_stream_t st = stream_of(a[9]);
    const auto fn = truth(a[10]) ? vgc_sqgrad_conv_exact : vgc_sqgrad_conv;
    VGC_CALL(fn(xp, dp, c.B, c.C, c.H, c.W, c.Cout, c.Kh, c.Kw, c.sh, c.sw, c.ph, c.pw, scale, acc, Sp, ws, wsb, st));
}

// xs, deltas, kernel, stride, padding, scale, Ss, accumulate, ws, stream, exact; the lists are not empty
PyObject *sqgrad_conv_batch(Args a)
{
    Ref xs(PySequence_Fast(a[0], "xs must be a sequence")), ds(PySequence_Fast(a[1], "deltas must be a sequence")),
        Ss(PySequence_Fast(a[6], "Ss must be a sequence"));
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(xs.p);
    if (PySequence_Fast_GET_SIZE(ds.p) != n || PySequence_Fast_GET_SIZE(Ss.p) != n)
        raise(PyExc_ValueError, "xs, deltas, Ss must have the same length");
    PyObject *const *xo = PySequence_Fast_ITEMS(xs.p), *const *po = PySequence_Fast_ITEMS(ds.p),
                    *const *so = PySequence_Fast_ITEMS(Ss.p);
    const at::Tensor &x0 = tensor(xo[0], "x"), &d0 = tensor(po[0], "delta");
    const ConvShape c = conv_shape(x0, d0, a[2], a[3], a[4]);
    if (c.B != d0.size(0) || !geometry_fits(c)) raise(PyExc_ValueError, "delta shape does not match the convolution geometry");
    std::vector<const float *> xp((size_t)n), dp((size_t)n);
    std::vector<float *> sp((size_t)n);
    for (Py_ssize_t l = 0; l < n; ++l) {
        const at::Tensor &x = tensor(xo[l], "x"), &d = tensor(po[l], "delta"), &S = tensor(so[l], "S");
        if (x.sizes() != x0.sizes() || d.sizes() != d0.sizes() || S.numel() != (int64_t)c.Cout * c.C * c.Kh * c.Kw)
            raise(PyExc_ValueError, "all layers of a batch must have the same shapes");
    }
    for (Py_ssize_t l = 0; l < n; ++l) {
        xp[(size_t)l] = dev_f(xo[l], "x");
        dp[(size_t)l] = dev_f(po[l], "delta");
        sp[(size_t)l] = dev_f(so[l], "S");
    }
    void *ws;
    size_t wsb;
    workspace(a[8], &ws, &wsb);
    const float scale = (float)number(a[5]);
    const int acc = truth(a[7]);
    vgc_stream_t st = stream_of(a[9]);
    const auto fn = truth(a[10]) ? vgc_sqgrad_conv_exact_batch : vgc_sqgrad_conv_batch;
    VGC_CALL(fn((int)n, xp.data(), dp.data(), sp.data(), c.B, c.C, c.H, c.W, c.Cout, c.Kh, c.Kw, c.sh, c.sw, c.ph, c.pw,
                scale, acc, ws, wsb, st));
}

void same_length(PyObject *g, PyObject *s, PyObject *r, PyObject *v, int64_t *n)
{
    *n = tensor(g, "g").numel();
    if ((s != Py_None && tensor(s, "s").numel() != *n) || tensor(r, "r").numel() != *n || tensor(v, "v").numel() != *n)
        raise(PyExc_ValueError, "g, s, r, v must have the same length");
}

void check_mask(PyObject *out, int64_t n)
{
    int64_t numel;
    optional_data(out, s_mask, &numel);
    if (numel >= 0 && numel != n) raise(PyExc_ValueError, "mask length");
}

// g, s, r, v, group_offsets, alpha, zeta, out, ws, stream
PyObject *compress(Args a)
{
    int64_t n;
    same_length(a[0], a[1], a[2], a[3], &n);
    const int64_t K = tensor(a[4], "group_offsets").numel() - 1;
    if (int_attr(a[7], s_K) != K) raise(PyExc_ValueError, "message buffers were made for a different number of groups");
    check_mask(a[7], n);
    void *ws;
    size_t wsb;
    workspace(a[8], &ws, &wsb);
    const vgc_message msg = message_of(a[7]);
    const float *g = dev_f(a[0], "g"), *s = a[1] == Py_None ? nullptr : dev_f(a[1], "s");
    float *r = dev_f(a[2], "r"), *v = dev_f(a[3], "v");
    const uint32_t *offs = dev_u(a[4], "group_offsets");
    const float alpha = (float)number(a[5]), zeta = (float)number(a[6]);
    vgc_stream_t st = stream_of(a[9]);
    VGC_CALL(vgc_compress(g, s, r, v, (size_t)n, offs, (int)K, alpha, zeta, &msg, ws, wsb, st));
}

// g, s, r, v, group_offsets, alpha, zeta, out, stream
PyObject *compress_static(Args a)
{
    int64_t n;
    if (a[1] == Py_None) raise(PyExc_TypeError, "%s must be a CUDA tensor", "s");
    same_length(a[0], a[1], a[2], a[3], &n);
    const int64_t K = tensor(a[4], "group_offsets").numel() - 1;
    if (int_attr(a[7], s_K) != K) raise(PyExc_ValueError, "message buffers were made for a different number of groups");
    const vgc_message msg = message_of(a[7]);
    const float *g = dev_f(a[0], "g"), *s = dev_f(a[1], "s");
    float *r = dev_f(a[2], "r"), *v = dev_f(a[3], "v");
    const uint32_t *offs = dev_u(a[4], "group_offsets");
    const float alpha = (float)number(a[5]), zeta = (float)number(a[6]);
    vgc_stream_t st = stream_of(a[8]);
    VGC_CALL(vgc_compress_static(g, s, r, v, (size_t)n, offs, (int)K, alpha, zeta, &msg, st));
}

// g, s, r, v, alpha, zeta, tau, correction_from_updated_r, out, ws, stream
PyObject *compress_hybrid(Args a)
{
    int64_t n;
    same_length(a[0], a[1], a[2], a[3], &n);
    check_mask(a[8], n);
    void *ws;
    size_t wsb;
    workspace(a[9], &ws, &wsb);
    const vgc_hybrid_message msg = hybrid_message_of(a[8]);
    const float *g = dev_f(a[0], "g"), *s = a[1] == Py_None ? nullptr : dev_f(a[1], "s");
    float *r = dev_f(a[2], "r"), *v = dev_f(a[3], "v");
    const float alpha = (float)number(a[4]), zeta = (float)number(a[5]), tau = (float)number(a[6]);
    const int updated = truth(a[7]);
    vgc_stream_t st = stream_of(a[10]);
    VGC_CALL(vgc_compress_hybrid(g, s, r, v, (size_t)n, alpha, zeta, tau, updated, &msg, ws, wsb, st));
}

// messages, group_offsets, scale, u, dev_status, stream, overwrite
PyObject *decode(Args a)
{
    std::vector<vgc_message_view> views;
    views_of(a[0], false, views);
    const int64_t K = tensor(a[1], "group_offsets").numel() - 1;
    const uint32_t *offs = dev_u(a[1], "group_offsets");
    const float scale = (float)number(a[2]);
    float *u = dev_f(a[3], "u");
    const size_t n = (size_t)THPVariable_Unpack(a[3]).numel();
    uint32_t *status = dev_u(a[4], "dev_status");
    vgc_stream_t st = stream_of(a[5]);
    const auto fn = truth(a[6]) ? vgc_decode_sum : vgc_decode_accumulate;
    VGC_CALL(fn(views.data(), (int)views.size(), offs, (int)K, scale, u, n, status, st));
}

// messages, tau, scale, u, dev_status, stream, overwrite
PyObject *decode_hybrid(Args a)
{
    std::vector<vgc_message_view> views;
    views_of(a[0], true, views);
    const float tau = (float)number(a[1]), scale = (float)number(a[2]);
    float *u = dev_f(a[3], "u");
    const size_t n = (size_t)THPVariable_Unpack(a[3]).numel();
    uint32_t *status = dev_u(a[4], "dev_status");
    vgc_stream_t st = stream_of(a[5]);
    const auto fn = truth(a[6]) ? vgc_decode_sum_hybrid : vgc_decode_accumulate_hybrid;
    VGC_CALL(fn(views.data(), (int)views.size(), tau, scale, u, n, status, st));
}

// words, nnz, packed, packed_bytes, dev_status, ws, stream
PyObject *pack_indices(Args a)
{
    void *ws;
    size_t wsb;
    workspace(a[5], &ws, &wsb);
    const uint32_t *words = dev_u(a[0], "words"), *nnz = dev_u(a[1], "nnz");
    const uint32_t max_words = (uint32_t)THPVariable_Unpack(a[0]).numel();
    uint8_t *packed = static_cast<uint8_t *>(dev(a[2], at::kByte, "packed"));
    const size_t capacity = (size_t)THPVariable_Unpack(a[2]).numel();
    uint32_t *bytes = dev_u(a[3], "packed_bytes"), *status = dev_u(a[4], "dev_status");
    vgc_stream_t st = stream_of(a[6]);
    VGC_CALL(vgc_pack_indices(words, nnz, max_words, packed, capacity, bytes, status, ws, wsb, st));
}

// packed, nnz, words, dev_status, stream
PyObject *unpack_indices(Args a)
{
    const uint8_t *packed = static_cast<const uint8_t *>(dev(a[0], at::kByte, "packed"));
    const uint32_t *nnz = dev_u(a[1], "nnz");
    uint32_t *words = dev_u(a[2], "words");
    const uint32_t max_words = (uint32_t)THPVariable_Unpack(a[2]).numel();
    uint32_t *status = dev_u(a[3], "dev_status");
    vgc_stream_t st = stream_of(a[4]);
    VGC_CALL(vgc_unpack_indices(packed, nnz, max_words, words, status, st));
}

long long layer_int(PyObject *layer, const char *key)
{
    Ref v(PyMapping_GetItemString(layer, key));
    return integer(v.p);
}
// layer.get(key, missing)
long long layer_int(PyObject *layer, const char *key, int missing)
{
    Ref v(PyObject_CallMethod(layer, "get", "si", key, missing));
    return integer(v.p);
}

// layers, g_host, g_dev, s_dev, r, v, group_offsets, alpha, zeta, scale, out, words_host, counters_host, ws_sqgrad,
// ws_compress, stream
PyObject *step_host(Args a)
{
    Ref seq(PySequence_Fast(a[0], "layers must be a sequence"));
    const Py_ssize_t n_layers = PySequence_Fast_GET_SIZE(seq.p);
    std::vector<vgc_layer_host> layers((size_t)(n_layers > 0 ? n_layers : 1));
    for (Py_ssize_t k = 0; k < n_layers; ++k) {
        PyObject *L = PySequence_Fast_GET_ITEM(seq.p, k);
        vgc_layer_host &o = layers[(size_t)k];
        Ref conv(PyMapping_GetItemString(L, "is_conv"));
        Ref conv_number(PyNumber_Long(conv.p));                          // (whatever int() takes)
        o.is_conv = truth(conv_number.p);
        o.B = (int)layer_int(L, "B");
        o.C = (int)layer_int(L, "C");
        o.H = (int)layer_int(L, "H", 1);
        o.W = (int)layer_int(L, "W", 1);
        o.Cout = (int)layer_int(L, "Cout");
        o.Kh = (int)layer_int(L, "Kh", 1);
        o.Kw = (int)layer_int(L, "Kw", 1);
        o.stride_h = o.stride_w = (int)layer_int(L, "stride", 1);
        o.pad_h = o.pad_w = (int)layer_int(L, "pad", 0);
        Ref xh(PyMapping_GetItemString(L, "x_host")), dh(PyMapping_GetItemString(L, "delta_host")),
            xd(PyMapping_GetItemString(L, "x_dev")), dd(PyMapping_GetItemString(L, "delta_dev"));
        o.x_host = static_cast<const float *>(host(xh.p, at::kFloat, "x_host"));
        o.delta_host = static_cast<const float *>(host(dh.p, at::kFloat, "delta_host"));
        o.x_dev = dev_f(xd.p, "x_dev");
        o.delta_dev = dev_f(dd.p, "delta_dev");
    }
    void *wsg, *wsc;
    size_t wsgb, wscb;
    workspace(a[13], &wsg, &wsgb);
    workspace(a[14], &wsc, &wscb);
    const int64_t K = tensor(a[6], "group_offsets").numel() - 1;
    const vgc_message msg = message_of(a[10]);
    const float *g_host = static_cast<const float *>(host(a[1], at::kFloat, "g_host"));
    float *g_dev = dev_f(a[2], "g_dev"), *s_dev = dev_f(a[3], "s_dev"), *r = dev_f(a[4], "r"), *v = dev_f(a[5], "v");
    const size_t n = (size_t)THPVariable_Unpack(a[2]).numel();
    const uint32_t *offs = dev_u(a[6], "group_offsets");
    const float alpha = (float)number(a[7]), zeta = (float)number(a[8]), scale = (float)number(a[9]);
    uint32_t *words_host = static_cast<uint32_t *>(host(a[11], at::kInt, "words_host"));
    uint32_t *counters_host = static_cast<uint32_t *>(host(a[12], at::kInt, "counters_host"));
    vgc_stream_t st = stream_of(a[15]);
    VGC_CALL(vgc_step_host(layers.data(), (int)n_layers, g_host, g_dev, s_dev, r, v, n, offs, (int)K, alpha, zeta, scale, &msg,
                           words_host, counters_host, wsg, wsgb, wsc, wscb, st));
}

// MessageBuffers, HybridMessageBuffers: the classes whose attributes are read directly
PyObject *use_classes(Args a)
{
    Py_INCREF(a[0]);
    Py_INCREF(a[1]);
    Py_XDECREF(t_message);
    Py_XDECREF(t_hybrid);
    t_message = a[0];
    t_hybrid = a[1];
    Py_RETURN_NONE;
}

template <PyObject *(*Fn)(Args), int kArgs>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != kArgs) {
        PyErr_Format(PyExc_TypeError, "%d arguments are wanted, got %zd", kArgs, n);
        return nullptr;
    }
    try {
        return Fn(args);
    } catch (const Raised &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <PyObject *(*Fn)(Args), int kArgs>
PyCFunction method()
{
    return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<Fn, kArgs>));
}

PyMethodDef methods[] = {
    {"sqgrad_linear", method<sqgrad_linear, 7>(), METH_FASTCALL, nullptr},
    {"sqgrad_conv", method<sqgrad_conv, 11>(), METH_FASTCALL, nullptr},
    {"sqgrad_conv_batch", method<sqgrad_conv_batch, 11>(), METH_FASTCALL, nullptr},
    {"compress", method<compress, 10>(), METH_FASTCALL, nullptr},
    {"compress_static", method<compress_static, 9>(), METH_FASTCALL, nullptr},
    {"compress_hybrid", method<compress_hybrid, 11>(), METH_FASTCALL, nullptr},
    {"decode", method<decode, 7>(), METH_FASTCALL, nullptr},
    {"decode_hybrid", method<decode_hybrid, 7>(), METH_FASTCALL, nullptr},
    {"pack_indices", method<pack_indices, 7>(), METH_FASTCALL, nullptr},
    {"unpack_indices", method<unpack_indices, 5>(), METH_FASTCALL, nullptr},
    {"step_host", method<step_host, 16>(), METH_FASTCALL, nullptr},
    {"use_classes", method<use_classes, 2>(), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_vgc_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__vgc_native()
{
    s_words = PyUnicode_InternFromString("words");
    s_group_exp = PyUnicode_InternFromString("group_exp");
    s_counters = PyUnicode_InternFromString("counters");
    s_mask = PyUnicode_InternFromString("mask");
    s_capacity = PyUnicode_InternFromString("capacity");
    s_K = PyUnicode_InternFromString("K");
    s_struct = PyUnicode_InternFromString("struct");
    s_view = PyUnicode_InternFromString("view");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
