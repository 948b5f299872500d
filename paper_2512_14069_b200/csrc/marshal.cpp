// Argument marshalling of the ctypes-free call path: fills an argument struct of radar.h from a dictionary of Python
// objects and calls the library.  A step makes a dozen calls of thirty arguments each, and where the draft model runs
// between them nothing hides their host time: filled field by field from Python a call took 25 us, of which the library
// and its launches are 5.  RADAR_BUILT_FOR names the torch and Python it is compiled against.  Nothing is kept between calls: every tensor is checked and its address taken each time.
#include <Python.h>

#include <torch/csrc/autograd/python_variable.h>

#include <climits>
#include <cstring>
#include <exception>
#include <vector>

namespace {

enum Kind : int { kInt = 0, kInt64 = 1, kFloat = 2, kPointer = 3 };

struct Field {
    Py_ssize_t offset;
    int kind;
    int dtype;          // c10::ScalarType a tensor must have, -1: any
    bool required;
    bool address;       // a pointer field that may also be given as a plain address
};

struct Filler {
    PyObject_HEAD
    Py_ssize_t size;
    PyObject* index;                    // {name: position in fields}
    std::vector<Field>* fields;
    Py_ssize_t n_required;
};

constexpr Py_ssize_t kMaxStruct = 1024;

// Writes one argument; false with a Python error set.
bool fill(const Field& f, PyObject* name, PyObject* v, unsigned char* out) {
    unsigned char* to = out + f.offset;
    switch (f.kind) {
        case kInt: {
            const long x = PyLong_AsLong(v);
            if (x == -1 && PyErr_Occurred()) return false;
            if (x < INT_MIN || x > INT_MAX) { PyErr_Format(PyExc_OverflowError, "%U does not fit an int", name); return false; }
            const int y = static_cast<int>(x);
            std::memcpy(to, &y, sizeof y);
            return true;
        }
        case kInt64: {
            const long long x = PyLong_AsLongLong(v);
            if (x == -1 && PyErr_Occurred()) return false;
            std::memcpy(to, &x, sizeof x);
            return true;
        }
        case kFloat: {
            const double x = PyFloat_AsDouble(v);
            if (x == -1.0 && PyErr_Occurred()) return false;
            const float y = static_cast<float>(x);
            std::memcpy(to, &y, sizeof y);
            return true;
        }
        default: {
            void* p = nullptr;
            if (v == Py_None) {
            } else if (THPVariable_Check(v)) {
                try {
                    const at::Tensor& t = THPVariable_Unpack(v);
                    if (!t.is_cuda() || !t.is_contiguous()) { PyErr_Format(PyExc_ValueError, "%U: expected a contiguous CUDA tensor", name); return false; }
                    if (f.dtype >= 0 && static_cast<int>(t.scalar_type()) != f.dtype) {
                        PyErr_Format(PyExc_ValueError, "%U: expected dtype %s, got %s", name, c10::toString(static_cast<c10::ScalarType>(f.dtype)),
                                     c10::toString(t.scalar_type()));
                        return false;
                    }
                    p = t.data_ptr();
                } catch (const std::exception& e) {
                    PyErr_SetString(PyExc_RuntimeError, e.what());
                    return false;
                }
            } else if (f.address) {
                p = PyLong_AsVoidPtr(v);
                if (p == nullptr && PyErr_Occurred()) return false;
            } else {
                PyErr_Format(PyExc_TypeError, "%U: expected a tensor or None, got %s", name, Py_TYPE(v)->tp_name);
                return false;
            }
            std::memcpy(to, &p, sizeof p);
            return true;
        }
    }
}

// filler(function address, context handle, stream handle, {name: value}) -> status
PyObject* filler_call(PyObject* self_, PyObject* args, PyObject* kwargs) {
    Filler* self = reinterpret_cast<Filler*>(self_);
    if (kwargs != nullptr && PyDict_GET_SIZE(kwargs) != 0) { PyErr_SetString(PyExc_TypeError, "positional arguments only"); return nullptr; }
    PyObject *fn, *ctx, *stream, *dict;
    if (!PyArg_UnpackTuple(args, "call", 4, 4, &fn, &ctx, &stream, &dict)) return nullptr;
    if (!PyDict_Check(dict)) { PyErr_SetString(PyExc_TypeError, "expected a dictionary"); return nullptr; }
    void* const f = PyLong_AsVoidPtr(fn);
    if (f == nullptr) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null function"); return nullptr; }
    void* const c = PyLong_AsVoidPtr(ctx);
    if (c == nullptr && PyErr_Occurred()) return nullptr;
    void* const s = PyLong_AsVoidPtr(stream);
    if (s == nullptr && PyErr_Occurred()) return nullptr;
    alignas(16) unsigned char buf[kMaxStruct];
    std::memset(buf, 0, static_cast<size_t>(self->size));
    Py_ssize_t pos = 0, required = 0;
    PyObject *key, *value;
    while (PyDict_Next(dict, &pos, &key, &value)) {
        PyObject* at = PyDict_GetItemWithError(self->index, key);
        if (at == nullptr) {
            if (!PyErr_Occurred()) PyErr_Format(PyExc_TypeError, "unexpected keyword argument '%S'", key);
            return nullptr;
        }
        const Field& fld = (*self->fields)[static_cast<size_t>(PyLong_AsSsize_t(at))];
        if (!fill(fld, key, value, buf)) return nullptr;
        required += fld.required ? 1 : 0;
    }
    if (required != self->n_required) {
        PyObject *name, *at;
        for (pos = 0; PyDict_Next(self->index, &pos, &name, &at);)
            if ((*self->fields)[static_cast<size_t>(PyLong_AsSsize_t(at))].required && PyDict_GetItemWithError(dict, name) == nullptr) {
                PyErr_Format(PyExc_TypeError, "missing required keyword argument '%S'", name);
                return nullptr;
            }
    }
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = reinterpret_cast<int (*)(void*, const void*, void*)>(f)(c, buf, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

// Filler(struct size, [(name, offset, kind, dtype, required, address), ...]); dtype: a tensor of the type, or None
PyObject* filler_new(PyTypeObject* type, PyObject* args, PyObject*) {
    Py_ssize_t size;
    PyObject* list;
    if (!PyArg_ParseTuple(args, "nO!", &size, &PyList_Type, &list)) return nullptr;
    if (size <= 0 || size > kMaxStruct) { PyErr_SetString(PyExc_ValueError, "struct size out of range"); return nullptr; }
    Filler* self = reinterpret_cast<Filler*>(type->tp_alloc(type, 0));
    if (self == nullptr) return nullptr;
    self->size = size;
    self->n_required = 0;
    self->index = PyDict_New();
    self->fields = new std::vector<Field>;
    for (Py_ssize_t i = 0; i < PyList_GET_SIZE(list); ++i) {
        PyObject *name, *dtype;
        Py_ssize_t offset;
        int kind, required, address;
        if (!PyArg_ParseTuple(PyList_GET_ITEM(list, i), "O!niOpp", &PyUnicode_Type, &name, &offset, &kind, &dtype, &required, &address)) { Py_DECREF(self); return nullptr; }
        const Py_ssize_t bytes = kind == kInt || kind == kFloat ? 4 : 8;
        if (kind < kInt || kind > kPointer || offset < 0 || offset + bytes > size) { Py_DECREF(self); PyErr_SetString(PyExc_ValueError, "bad field"); return nullptr; }
        Field f{offset, kind, -1, required != 0, address != 0};
        if (dtype != Py_None) {
            if (!THPVariable_Check(dtype)) { Py_DECREF(self); PyErr_SetString(PyExc_TypeError, "dtype: a tensor of the type, or None"); return nullptr; }
            f.dtype = static_cast<int>(THPVariable_Unpack(dtype).scalar_type());
        }
        PyObject* at = PyLong_FromSsize_t(static_cast<Py_ssize_t>(self->fields->size()));
        self->fields->push_back(f);
        self->n_required += f.required ? 1 : 0;
        const int rc = at == nullptr ? -1 : PyDict_SetItem(self->index, name, at);
        Py_XDECREF(at);
        if (rc != 0) { Py_DECREF(self); return nullptr; }
    }
    return reinterpret_cast<PyObject*>(self);
}

void filler_dealloc(PyObject* self_) {
    Filler* self = reinterpret_cast<Filler*>(self_);
    Py_XDECREF(self->index);
    delete self->fields;
    PyTypeObject* type = Py_TYPE(self_);
    type->tp_free(self_);
    Py_DECREF(type);
}

PyType_Slot filler_slots[] = {{Py_tp_new, reinterpret_cast<void*>(filler_new)},
                              {Py_tp_call, reinterpret_cast<void*>(filler_call)},
                              {Py_tp_dealloc, reinterpret_cast<void*>(filler_dealloc)},
                              {0, nullptr}};
PyType_Spec filler_spec = {"_marshal.Filler", sizeof(Filler), 0, Py_TPFLAGS_DEFAULT, filler_slots};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, nullptr, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
    PyObject* m = PyModule_Create(&module_def);
    if (m == nullptr) return nullptr;
    PyObject* type = PyType_FromSpec(&filler_spec);
    if (type == nullptr || PyModule_AddStringConstant(m, "BUILT_FOR", RADAR_BUILT_FOR) != 0 || PyModule_AddObject(m, "Filler", type) != 0) {
        Py_XDECREF(type);
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
