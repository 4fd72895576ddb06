// CPython entry points over the C ABI of flashbev.h for callers with torch tensors: argument checks, allocation of the result
// and of the scratch, current stream, parameter struct, call.  Marshalling only, no arithmetic of the operator.
//
// Why native: a call on a coarse grid is 8 us of GPU work, and the same marshalling in Python (about forty ctypes field
// assignments, a device context, tensor attributes) took 16 us per call.  Every function returns the result tensor, or the
// library's status as an int when the call was refused (the Python wrapper raises for it).
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <vector>

#include "flashbev.h"

namespace {

struct Bad {};  // a Python error has been set

[[noreturn]] void value_error(const char *what)
{
    PyErr_SetString(PyExc_ValueError, what);
    throw Bad();
}

const at::Tensor &tensor(PyObject *o, const char *what)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a tensor, not %.100s", what, Py_TYPE(o)->tp_name);
        throw Bad();
    }
    return THPVariable_Unpack(o);
}

int64_t integer(PyObject *o)
{
    PyObject *i = PyNumber_Index(o);
    if (!i) throw Bad();
    const long long v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Bad();
    return v;
}

int32_t narrow(int64_t v)
{
    if (v != (int32_t)v) {
        PyErr_SetString(PyExc_OverflowError, "argument does not fit 32 bits");
        throw Bad();
    }
    return (int32_t)v;
}

int32_t integer32(PyObject *o) { return narrow(integer(o)); }

// int(o): numbers of any kind, cut to whole ones
int32_t cut_integer32(PyObject *o)
{
    PyObject *i = PyNumber_Long(o);
    if (!i) throw Bad();
    const long long v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Bad();
    return narrow(v);
}

// float(o)
double real(PyObject *o)
{
    PyObject *f = PyNumber_Float(o);
    if (!f) throw Bad();
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return v;
}

// The n items of a sequence, handed to `f(index, item)`
template <typename F>
void items(PyObject *o, Py_ssize_t n, const char *what, F f)
{
    PyObject *seq = PySequence_Fast(o, what);
    if (!seq) throw Bad();
    const bool ok = PySequence_Fast_GET_SIZE(seq) == n;
    try {
        if (!ok) value_error(what);
        for (Py_ssize_t i = 0; i < n; ++i) f(i, PySequence_Fast_GET_ITEM(seq, i));
    } catch (...) {
        Py_DECREF(seq);
        throw;
    }
    Py_DECREF(seq);
}

// Geometry fields shared by the parameter structs: image size, ranges, bins
template <typename P>
void geometry(P &p, PyObject *img_hw, PyObject *bev_range)
{
    int32_t hw[2];
    items(img_hw, 2, "img_hw must be (height, width)", [&](Py_ssize_t i, PyObject *v) { hw[i] = integer32(v); });
    p.img_h = hw[0], p.img_w = hw[1];
    double r[6];
    items(bev_range, 6, "bev_range must have six numbers", [&](Py_ssize_t i, PyObject *v) { r[i] = real(v); });
    p.x_min = r[0], p.x_max = r[1], p.y_min = r[2], p.y_max = r[3], p.z_min = r[4], p.z_max = r[5];
}

void tune(int32_t (&t)[4], PyObject *o)
{
    PyObject *seq = PySequence_Fast(o, "tune must be a sequence");
    if (!seq) throw Bad();
    try {
        if (PySequence_Fast_GET_SIZE(seq) > 4) value_error("tune has at most four entries");
        for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(seq); ++i) t[i] = cut_integer32(PySequence_Fast_GET_ITEM(seq, i));
    } catch (...) {
        Py_DECREF(seq);
        throw;
    }
    Py_DECREF(seq);
}

// The stream argument: None for the current one, or a cudaStream_t as an integer
struct StreamArg {
    bool current;
    void *raw;
    explicit StreamArg(PyObject *o)
        : current(o == Py_None), raw(current ? nullptr : reinterpret_cast<void *>(static_cast<uintptr_t>(integer(o))))
    {
    }
};

// A call's device and stream.  A stream that the caller names is the current one while this object lives, so that the allocator
// hands out memory that belongs to it: scratch is free again when the call returns, and only later work of the same stream may
// get it, and what an earlier owner still does on another stream is not written over.  (Memory of the current stream, written
// on another one, was open to both.)
class Place {
    const c10::cuda::CUDAGuard device_;
    c10::cuda::OptionalCUDAStreamGuard named_;
    void *stream_;
    c10::cuda::CUDAStream caller_;

public:
    Place(const at::Tensor &t, const StreamArg &s)
        : device_(t.device()), stream_(s.raw), caller_(c10::cuda::getCurrentCUDAStream(t.get_device()))
    {
        if (s.current) stream_ = caller_.stream();
        if (stream_ == caller_.stream()) return;
        // (the legacy stream has a handle of its own beside NULL)
        const cudaStream_t raw = static_cast<cudaStream_t>(stream_);
        named_.reset_stream(raw == cudaStreamLegacy ? c10::cuda::getDefaultCUDAStream(t.get_device())
                                                    : c10::cuda::getStreamFromExternal(raw, t.get_device()));
    }
    void *stream() const { return stream_; }

    // A result: the caller goes on with it on the stream that was current, and drops it at any time.
    at::Tensor result(at::Tensor t) const
    {
        if (stream_ != caller_.stream()) t.record_stream(caller_.unwrap());
        return t;
    }
};

int32_t feature_dtype(const at::Tensor &t)
{
    if (t.scalar_type() == at::kFloat) return FLASHBEV_F32;
    if (t.scalar_type() == at::kBFloat16) return FLASHBEV_BF16;
    value_error("features must be float32 or bfloat16");
}

at::Tensor empty(std::initializer_list<int64_t> shape, at::ScalarType type, const at::Tensor &like)
{
    return at::empty(shape, at::TensorOptions().dtype(type).device(like.device()));
}

// `body` without the interpreter lock: an allocation, a launch into a full queue or the memset of the backward may wait, and
// the process's other Python threads go on meanwhile.  `body` touches no Python object.
template <typename F>
flashbev_status unlocked(F body)
{
    struct Unlock {
        PyThreadState *state = PyEval_SaveThread();
        ~Unlock() { PyEval_RestoreThread(state); }
    } unlock;
    return body();
}

PyObject *status(flashbev_status st) { return PyLong_FromLong(st); }

void need_args(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
    throw Bad();
}

// `body` with C++ exceptions turned into the Python errors that PyTorch's own functions raise for them: a failed allocation is
// torch.OutOfMemoryError (callers catch it, free memory and try again), a missing dimension IndexError.
template <typename F>
PyObject *guarded(F body)
{
    try {
        return body();
    } catch (const Bad &) {
        return nullptr;
    } catch (...) {
        torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
}

// features, lidar2img, img_hw, bev_range, grid, reduce, out, valid_count, kernel, tune, stream, layout, out_dtype, workspace
PyObject *py_sampling_vt(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        need_args(n, 14);
        const at::Tensor &f = tensor(a[0], "features"), &m = tensor(a[1], "lidar2img");
        if (!f.is_cuda() || !m.is_cuda()) value_error("sampling_vt needs CUDA tensors; there is no CPU path");
        if (!f.is_contiguous() || !m.is_contiguous()) value_error("features and lidar2img must be contiguous");
        flashbev_vt_params p = {};
        p.struct_size = sizeof(p);
        p.feat_dtype = feature_dtype(f);
        if (m.scalar_type() != at::kFloat) value_error("lidar2img must be float32");
        if (f.dim() != 5) value_error("features must have five dimensions");
        p.layout = integer32(a[11]);
        const bool nhwc = p.layout == FLASHBEV_NHWC;
        p.B = (int32_t)f.size(0), p.N = (int32_t)f.size(1), p.C = (int32_t)f.size(nhwc ? 4 : 2);
        p.feat_h = (int32_t)f.size(nhwc ? 2 : 3), p.feat_w = (int32_t)f.size(nhwc ? 3 : 4);
        geometry(p, a[2], a[3]);
        int32_t *const axis[3] = {&p.X, &p.Y, &p.Z};
        items(a[4], 3, "grid must be (X, Y, Z)", [&](Py_ssize_t i, PyObject *v) { *axis[i] = integer32(v); });
        p.reduce = integer32(a[5]), p.kernel = integer32(a[8]), p.out_dtype = integer32(a[12]);
        tune(p.tune, a[9]);
        const StreamArg stream(a[10]);
        at::Tensor out, scratch;
        if (a[6] != Py_None) out = tensor(a[6], "out");
        if (a[7] != Py_None) p.valid_count_out = static_cast<int32_t *>(tensor(a[7], "valid_count").data_ptr());
        const bool lend = a[13] != Py_False && a[13] != Py_None, own_scratch = a[13] == Py_True;
        if (lend && !own_scratch && THPVariable_Check(a[13])) scratch = THPVariable_Unpack(a[13]);
        const flashbev_status st = unlocked([&] {
            const Place place(f, stream);
            const auto type = p.out_dtype == FLASHBEV_F32 ? at::kFloat : at::kBFloat16;
            if (!out.defined())
                out = place.result(nhwc ? empty({p.B, p.X, p.Y, p.C}, type, f) : empty({p.B, p.C, p.X, p.Y}, type, f));
            p.features = f.data_ptr(), p.lidar2img = static_cast<const float *>(m.data_ptr()), p.out = out.data_ptr();
            const size_t need = lend ? flashbev_workspace_bytes(&p) : 0;
            if (need) {
                if (own_scratch) scratch = empty({(int64_t)need}, at::kByte, f);
                TORCH_CHECK_TYPE(scratch.defined(), "workspace must be True, False, None or a tensor");
                p.workspace = scratch.data_ptr(), p.workspace_bytes = (size_t)scratch.numel() * scratch.element_size();
            }
            return flashbev_sampling_vt(&p, place.stream());
        });
        return st == FLASHBEV_OK ? THPVariable_Wrap(std::move(out)) : status(st);
    });
}

// grad_out, lidar2img, feat_hw, img_hw, bev_range, grid, reduce, grad_features, tune, stream
PyObject *py_sampling_vt_backward(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        need_args(n, 10);
        const at::Tensor &g = tensor(a[0], "grad_out"), &m = tensor(a[1], "lidar2img");
        if (!g.is_cuda() || g.scalar_type() != at::kFloat || !g.is_contiguous())
            value_error("grad_out must be a contiguous CUDA float32 tensor");
        if (!m.is_cuda() || m.scalar_type() != at::kFloat || !m.is_contiguous())
            value_error("lidar2img must be a contiguous CUDA float32 tensor");
        if (g.dim() != 4) value_error("grad_out must have four dimensions");
        flashbev_vt_backward_params p = {};
        p.struct_size = sizeof(p);
        p.B = (int32_t)g.size(0), p.X = (int32_t)g.size(1), p.Y = (int32_t)g.size(2), p.C = (int32_t)g.size(3);
        p.N = (int32_t)m.size(1);
        items(a[2], 2, "feat_hw must be (height, width)", [&](Py_ssize_t i, PyObject *v) { (i ? p.feat_w : p.feat_h) = integer32(v); });
        geometry(p, a[3], a[4]);
        PyObject *z = PySequence_GetItem(a[5], 2);  // X and Y are those of grad_out
        if (!z) throw Bad();
        try {
            p.Z = integer32(z);
        } catch (...) {
            Py_DECREF(z);
            throw;
        }
        Py_DECREF(z);
        p.reduce = integer32(a[6]);
        tune(p.tune, a[8]);
        const StreamArg stream(a[9]);
        at::Tensor out;
        if (a[7] != Py_None) out = tensor(a[7], "grad_features");
        const flashbev_status st = unlocked([&] {
            const Place place(g, stream);
            if (!out.defined()) out = place.result(empty({p.B, p.N, p.feat_h, p.feat_w, p.C}, at::kFloat, g));
            p.grad_out = static_cast<const float *>(g.data_ptr()), p.lidar2img = static_cast<const float *>(m.data_ptr());
            p.grad_features = static_cast<float *>(out.data_ptr());
            return flashbev_sampling_vt_backward(&p, place.stream());
        });
        return st == FLASHBEV_OK ? THPVariable_Wrap(std::move(out)) : status(st);
    });
}

// features (sequence), lidar2img, img_hw, bev_range, grid, reduce, out, valid_count, kernel, tune, stream, layout
PyObject *py_sampling_vt_multires(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        need_args(n, 12);
        const Py_ssize_t levels = PySequence_Size(a[0]);
        if (levels < 0) throw Bad();
        if (levels < 1) value_error("at least one level is needed");
        std::vector<at::Tensor> maps;
        items(a[0], levels, "features must be a sequence of tensors",
              [&](Py_ssize_t, PyObject *v) { maps.push_back(tensor(v, "features")); });
        const at::Tensor &f0 = maps[0], &m = tensor(a[1], "lidar2img");
        for (const at::Tensor &f : maps)
            if (!f.is_cuda() || !f.is_contiguous() || f.dtype() != f0.dtype() || f.dim() != 5)
                value_error("every level must be a contiguous CUDA tensor of the same dtype");
        flashbev_vt_params p = {};
        p.struct_size = sizeof(p);
        p.feat_dtype = feature_dtype(f0);
        if (!m.is_cuda() || m.scalar_type() != at::kFloat || !m.is_contiguous())
            value_error("lidar2img must be a contiguous CUDA float32 tensor");
        p.layout = integer32(a[11]);
        const bool nhwc = p.layout == FLASHBEV_NHWC;
        p.B = (int32_t)f0.size(0), p.N = (int32_t)f0.size(1), p.C = (int32_t)f0.size(nhwc ? 4 : 2);
        geometry(p, a[2], a[3]);
        int32_t *const axis[3] = {&p.X, &p.Y, &p.Z};
        items(a[4], 3, "grid must be (X, Y, Z)", [&](Py_ssize_t i, PyObject *v) { *axis[i] = integer32(v); });
        p.reduce = integer32(a[5]), p.kernel = integer32(a[8]), p.out_dtype = FLASHBEV_F32;
        tune(p.tune, a[9]);
        const StreamArg stream(a[10]);
        at::Tensor out, scratch;
        if (a[6] != Py_None) out = tensor(a[6], "out");
        if (a[7] != Py_None) p.valid_count_out = static_cast<int32_t *>(tensor(a[7], "valid_count").data_ptr());
        const flashbev_status st = unlocked([&] {
            const Place place(f0, stream);
            if (!out.defined())
                out = place.result(nhwc ? empty({p.B, p.X, p.Y, p.C}, at::kFloat, f0) : empty({p.B, p.C, p.X, p.Y}, at::kFloat, f0));
            p.lidar2img = static_cast<const float *>(m.data_ptr()), p.out = out.data_ptr();
            // planar tensors and ragged channel counts: lend the scratch of the largest level (the levels run one after another)
            std::vector<const void *> ptrs;
            std::vector<int32_t> hw;
            size_t need = 0;
            for (const at::Tensor &f : maps) {
                ptrs.push_back(f.data_ptr());
                hw.push_back((int32_t)f.size(nhwc ? 2 : 3)), hw.push_back((int32_t)f.size(nhwc ? 3 : 4));
                p.features = ptrs.back(), p.feat_h = hw[hw.size() - 2], p.feat_w = hw.back();
                need = std::max(need, flashbev_workspace_bytes(&p));
            }
            p.features = ptrs[0], p.feat_h = hw[0], p.feat_w = hw[1];
            if (need) {
                scratch = empty({(int64_t)need}, at::kByte, f0);
                p.workspace = scratch.data_ptr(), p.workspace_bytes = need;
            }
            flashbev_vt_multires_params q = {};
            q.struct_size = sizeof(q), q.base = &p, q.levels = (int32_t)levels, q.features = ptrs.data(), q.feat_hw = hw.data();
            return flashbev_sampling_vt_multires(&q, place.stream());
        });
        return st == FLASHBEV_OK ? THPVariable_Wrap(std::move(out)) : status(st);
    });
}

// value, level_hw, lidar2img, offsets, weights, img_hw, bev_range, grid, out, hits, stream, chunk_records
PyObject *py_sca(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        need_args(n, 12);
        const at::Tensor &v = tensor(a[0], "value"), &m = tensor(a[2], "lidar2img");
        const at::Tensor &o = tensor(a[3], "offsets"), &w = tensor(a[4], "weights");
        for (const at::Tensor *t : {&m, &o, &w})
            if (!t->is_cuda() || t->scalar_type() != at::kFloat || !t->is_contiguous())
                value_error("sca needs contiguous CUDA float32 tensors");
        if (!v.is_cuda() || !v.is_contiguous() || (v.scalar_type() != at::kFloat && v.scalar_type() != at::kBFloat16))
            value_error("value must be a contiguous CUDA float32 or bfloat16 tensor");
        if (v.dim() != 5 || w.dim() != 5) value_error("value and weights must have five dimensions");
        flashbev_sca_params p = {};
        p.struct_size = sizeof(p);
        p.value_dtype = v.scalar_type() == at::kFloat ? FLASHBEV_F32 : FLASHBEV_BF16;
        p.B = (int32_t)v.size(0), p.N = (int32_t)v.size(1), p.heads = (int32_t)v.size(3), p.head_dim = (int32_t)v.size(4);
        p.L = (int32_t)w.size(3), p.P = (int32_t)w.size(4);
        const Py_ssize_t levels = PyObject_Size(a[1]);
        if (levels < 0) throw Bad();
        std::vector<int32_t> hw;  // (height, width) pairs, or the same numbers one after another
        items(a[1], levels, "level_hw must be a sequence of (height, width)", [&](Py_ssize_t, PyObject *l) {
            const auto put = [&](Py_ssize_t, PyObject *x) { hw.push_back(cut_integer32(x)); };
            const bool row = PyObject_Size(l) >= 0;
            PyErr_Clear();  // (a number has none)
            if (row) items(l, 2, "level_hw must be a sequence of (height, width)", put);
            else put(0, l);
        });
        if (hw.size() < 2 * (size_t)p.L) value_error("level_hw must have an entry per level");
        geometry(p, a[5], a[6]);
        int32_t *const axis[3] = {&p.X, &p.Y, &p.Zref};
        items(a[7], 3, "grid must be (X, Y, Zref)", [&](Py_ssize_t i, PyObject *x) { *axis[i] = integer32(x); });
        p.chunk_records = cut_integer32(a[11]);
        const StreamArg stream(a[10]);
        at::Tensor out;
        if (a[8] != Py_None) out = tensor(a[8], "out");
        if (a[9] != Py_None) p.hits_out = static_cast<int32_t *>(tensor(a[9], "hits").data_ptr());
        const flashbev_status st = unlocked([&] {
            const Place place(v, stream);
            if (!out.defined()) out = place.result(empty({p.B, (int64_t)p.X * p.Y, (int64_t)p.heads * p.head_dim}, at::kFloat, v));
            p.value = v.data_ptr(), p.level_hw = hw.data(), p.lidar2img = static_cast<const float *>(m.data_ptr());
            p.offsets = static_cast<const float *>(o.data_ptr()), p.weights = static_cast<const float *>(w.data_ptr());
            p.out = static_cast<float *>(out.data_ptr());
            return flashbev_sca(&p, place.stream());
        });
        return st == FLASHBEV_OK ? THPVariable_Wrap(std::move(out)) : status(st);
    });
}

PyMethodDef methods[] = {
    {"sampling_vt", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(py_sampling_vt)), METH_FASTCALL, nullptr},
    {"sampling_vt_backward", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(py_sampling_vt_backward)), METH_FASTCALL, nullptr},
    {"sampling_vt_multires", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(py_sampling_vt_multires)), METH_FASTCALL, nullptr},
    {"sca", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(py_sca)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
