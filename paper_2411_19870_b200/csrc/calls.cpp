// The per-step calls of binding.py without Python between the tensors and the library: a call whose tensors have the layout that the
// library assumes (number, type, shape, device, contiguous: looked at in every call, wherever they lie) takes the current stream and enters
// the library; anything else returns None, and binding.py takes its own way, which says what is wrong.
//
// What it saves is host time, which is all that a step of small tensors costs (one attribute look-up and method call per tensor and list,
// the checks in Python, ctypes' conversion of the arguments, the device and stream queries).  Without it -> with it, tensors where the call
// before had them / tensors elsewhere, whose pointers the library copies to the device: compress of one matrix 5.6 -> 3.0 / 15.5 -> 9.6 us,
// of 50 matrices and 12 vectors (two launches) 16.3 -> 7.1 / 93 -> 20, decode of the same set 12.2 -> 6.4 / 48 -> 9.8, of 64 payloads
// 28.4 -> 8.1 / 38.4 -> 11.6.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <c10/util/SmallVector.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <memory>
#include <vector>

namespace {

// A reference that is given up at the end of the scope.
struct Ref {
    PyObject *p;
    explicit Ref(PyObject *o) : p(o) {}
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
    explicit operator bool() const { return p != nullptr; }
};

// data_ptr() of a tensor; false with a Python error set.  Subclasses of Tensor are asked through their own method.
bool data_pointer(PyObject *t, std::uintptr_t *out)
{
    if (THPVariable_CheckExact(t)) {
        *out = reinterpret_cast<std::uintptr_t>(THPVariable_Unpack(t).data_ptr());
        return true;
    }
    Ref v(PyObject_CallMethod(t, "data_ptr", nullptr));
    if (!v) return false;
    *out = reinterpret_cast<std::uintptr_t>(PyLong_AsVoidPtr(v.p));
    return !PyErr_Occurred();
}

enum class Found { error, no, yes };

// What the library assumes of a list of tensors: contiguous, of one type, on one device (-1: any), of these shapes.
struct Layouts {
    at::ScalarType dtype;
    int device;
    std::vector<std::int64_t> dims;         // shape after shape
    std::vector<std::size_t> starts = {0};  // of the shapes, and the end
    Py_ssize_t size() const { return (Py_ssize_t)starts.size() - 1; }
    bool placed(const at::Tensor &t) const { return device < 0 || t.device() == at::Device(at::kCUDA, (at::DeviceIndex)device); }
    bool fits(const at::Tensor &t, Py_ssize_t i) const  // (i < size())
    {
        return t.scalar_type() == dtype && t.sizes() == at::IntArrayRef(dims.data() + starts[i], starts[i + 1] - starts[i]) && t.is_contiguous() &&
               placed(t);
    }
};
constexpr const char *LAYOUTS = "paper_2411_19870_b200.layouts";
void free_layouts(PyObject *capsule) { delete static_cast<Layouts *>(PyCapsule_GetPointer(capsule, LAYOUTS)); }

// layouts(dtype, device index or -1, sequence of shapes): the third part of a cache entry, against which every call's tensors are held
PyObject *make_layouts(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    if (n != 3 || !THPDtype_Check(a[0])) return PyErr_Format(PyExc_TypeError, "layouts: a dtype, a device index and shapes");
    auto l = std::make_unique<Layouts>();
    l->dtype = reinterpret_cast<THPDtype *>(a[0])->scalar_type;
    l->device = (int)PyLong_AsLong(a[1]);
    Ref shapes(PySequence_Fast(a[2], "layouts: shapes"));
    if (!shapes || PyErr_Occurred()) return nullptr;
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(shapes.p); ++i) {
        Ref shape(PySequence_Fast(PySequence_Fast_GET_ITEM(shapes.p, i), "layouts: a shape"));
        if (!shape) return nullptr;
        for (Py_ssize_t d = 0; d < PySequence_Fast_GET_SIZE(shape.p); ++d)
            l->dims.push_back(PyLong_AsLongLong(PySequence_Fast_GET_ITEM(shape.p, d)));
        l->starts.push_back(l->dims.size());
    }
    if (PyErr_Occurred()) return nullptr;
    PyObject *capsule = PyCapsule_New(l.get(), LAYOUTS, free_layouts);
    if (capsule) l.release();
    return capsule;
    END_HANDLE_TH_ERRORS
}

// The pointers of a list of tensors, and the cache entry that they were held against.
struct Array {
    PyObject *entry = nullptr;
    const Layouts *layouts = nullptr;
    c10::SmallVector<void *, 64> pointers;
    Py_buffer view{};
    ~Array()
    {
        if (view.obj) PyBuffer_Release(&view);
        Py_XDECREF(entry);
    }
    void **data() { return pointers.data(); }
};
// cache[key] = (list, array of pointers, layouts).  Tensors proper are held against the layouts.  A subclass answers for itself, in Python:
// it has to lie where it lay when binding.py asked it last, which is what the array says.  (So does everything under an entry without layouts.)
Found lookup(PyObject *cache, PyObject *key, PyObject *tensors, Array *array)
{
    PyObject *hit = PyDict_GetItemWithError(cache, key);  // (borrowed; kept by `array` below)
    if (!hit) return PyErr_Occurred() ? Found::error : Found::no;
    if (!PyTuple_Check(hit) || PyTuple_GET_SIZE(hit) < 2 || PyTuple_GET_SIZE(hit) > 3) return Found::no;
    array->entry = Py_NewRef(hit);
    if (PyTuple_GET_SIZE(hit) == 3) {
        array->layouts = static_cast<const Layouts *>(PyCapsule_GetPointer(PyTuple_GET_ITEM(hit, 2), LAYOUTS));
        if (!array->layouts) return Found::error;
    }
    const Layouts *l = array->layouts;
    if (!PyList_Check(tensors) && !PyTuple_Check(tensors)) return Found::no;  // (an iterator is left to binding.py)
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(tensors);
    if (l && l->size() != n) return Found::no;
    auto known = [&]() {  // the array, asked for once; null with a Python error set
        if (!array->view.obj && PyObject_GetBuffer(PyTuple_GET_ITEM(array->entry, 1), &array->view, PyBUF_SIMPLE) != 0) return false;
        return true;
    };
    if (!l) {
        if (!known()) return Found::error;
        if (array->view.len != n * (Py_ssize_t)sizeof(void *)) return Found::no;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (i >= PySequence_Fast_GET_SIZE(tensors)) return Found::no;  // (a subclass's data_ptr may have changed the list)
        PyObject *t = PySequence_Fast_GET_ITEM(tensors, i);
        if (l && THPVariable_CheckExact(t)) {
            const at::Tensor &v = THPVariable_Unpack(t);
            if (!l->fits(v, i)) return Found::no;
            array->pointers.push_back(v.data_ptr());
            continue;
        }
        Ref hold(Py_NewRef(t));
        std::uintptr_t p;
        if (l && (!THPVariable_Check(t) || !l->fits(THPVariable_Unpack(t), i))) return Found::no;
        if (!known() || !data_pointer(t, &p)) return Found::error;
        if ((i + 1) * (Py_ssize_t)sizeof(void *) > array->view.len || static_cast<std::uintptr_t *>(array->view.buf)[i] != p) return Found::no;
        array->pointers.push_back(reinterpret_cast<void *>(p));
    }
    return Found::yes;
}

// Whether a payload is bytes end to end, on the tensors' device, and its (data pointer, size) among those that were checked.
Found payload_known(PyObject *known, PyObject *payload, const Layouts *tensors, std::uintptr_t *ptr)
{
    if (!THPVariable_CheckExact(payload)) return Found::no;
    const at::Tensor &t = THPVariable_Unpack(payload);
    if (t.scalar_type() != at::kByte || !t.is_contiguous() || (tensors && !tensors->placed(t))) return Found::no;
    *ptr = reinterpret_cast<std::uintptr_t>(t.data_ptr());
    Ref key(Py_BuildValue("(KL)", (unsigned long long)*ptr, (long long)t.numel()));
    if (!key) return Found::error;
    const int in = PySet_Contains(known, key.p);
    return in < 0 ? Found::error : in ? Found::yes : Found::no;
}

bool stream_of(PyObject *stream, void **out)
{
    if (stream == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    *out = PyLong_AsVoidPtr(stream);
    return !PyErr_Occurred();
}

PyObject *slow(Found f)
{
    if (f == Found::error) return nullptr;
    Py_RETURN_NONE;
}

using CompressFn = int (*)(void *, std::int32_t, void **, void **, void *, void *);
using DecodeFn = int (*)(void *, void **, std::int32_t, void **, void *);
using ApplyFn = int (*)(void *, void **, void **, void *);

// compress(function, context, cache, known payloads, worker, key of grads, grads, key of momentum, momentum, payload, stream or None)
PyObject *compress(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    if (n != 11) return PyErr_Format(PyExc_TypeError, "compress: 11 arguments");
    void *fn = PyLong_AsVoidPtr(a[0]), *ctx = PyLong_AsVoidPtr(a[1]), *stream = nullptr;
    const long worker = PyLong_AsLong(a[4]);
    if (PyErr_Occurred()) return nullptr;
    std::uintptr_t payload = 0;
    Array g, m;
    Found f = lookup(a[2], a[5], a[6], &g);
    if (f == Found::yes) f = lookup(a[2], a[7], a[8], &m);
    if (f == Found::yes) f = payload_known(a[3], a[9], g.layouts, &payload);
    if (f != Found::yes) return slow(f);
    if (!stream_of(a[10], &stream)) return nullptr;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = reinterpret_cast<CompressFn>(fn)(ctx, (std::int32_t)worker, g.data(), m.data(), reinterpret_cast<void *>(payload), stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
    END_HANDLE_TH_ERRORS
}

// decode(function, context, cache, known payloads, payloads, key of tensors, tensors, stream or None)
PyObject *decode(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    if (n != 8) return PyErr_Format(PyExc_TypeError, "decode: 8 arguments");
    void *fn = PyLong_AsVoidPtr(a[0]), *ctx = PyLong_AsVoidPtr(a[1]), *stream = nullptr;
    if (PyErr_Occurred()) return nullptr;
    if (!PyList_Check(a[4]) && !PyTuple_Check(a[4])) Py_RETURN_NONE;
    Array x;
    c10::SmallVector<void *, 64> p;
    Found f = lookup(a[2], a[5], a[6], &x);
    for (Py_ssize_t i = 0; f == Found::yes && i < PySequence_Fast_GET_SIZE(a[4]); ++i) {
        std::uintptr_t ptr;
        f = payload_known(a[3], PySequence_Fast_GET_ITEM(a[4], i), x.layouts, &ptr);
        if (f == Found::yes) p.push_back(reinterpret_cast<void *>(ptr));
    }
    if (f != Found::yes) return slow(f);
    if (!stream_of(a[7], &stream)) return nullptr;
    const std::int32_t count = (std::int32_t)p.size();
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = reinterpret_cast<DecodeFn>(fn)(ctx, p.data(), count, x.data(), stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
    END_HANDLE_TH_ERRORS
}

// apply_signs(function, context, cache, signs, params, stream or None)
PyObject *apply_signs(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    if (n != 6) return PyErr_Format(PyExc_TypeError, "apply_signs: 6 arguments");
    void *fn = PyLong_AsVoidPtr(a[0]), *ctx = PyLong_AsVoidPtr(a[1]), *stream = nullptr;
    if (PyErr_Occurred()) return nullptr;
    static PyObject *const key_s = PyUnicode_InternFromString("s"), *const key_x = PyUnicode_InternFromString("x");
    if (!key_s || !key_x) return nullptr;
    Array s, x;
    Found f = lookup(a[2], key_s, a[3], &s);
    if (f == Found::yes) f = lookup(a[2], key_x, a[4], &x);
    if (f != Found::yes) return slow(f);
    if (!stream_of(a[5], &stream)) return nullptr;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = reinterpret_cast<ApplyFn>(fn)(ctx, s.data(), x.data(), stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"layouts", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(make_layouts)), METH_FASTCALL, nullptr},
    {"compress", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(compress)), METH_FASTCALL, nullptr},
    {"decode", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(decode)), METH_FASTCALL, nullptr},
    {"apply_signs", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(apply_signs)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&module); }
