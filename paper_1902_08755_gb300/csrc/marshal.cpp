// marshal.cpp -- the binding's argument marshalling for lists of images: fills
// the C ABI's descriptor arrays from the Python objects.
//
// A compositing call over n images needs about a dozen attribute reads and
// checks per image; done in Python they take 3.4 us per image, and 7.6 with a
// gradient buffer (64 tiles: 213 us around a 21 us kernel; 128 layers with
// gradients: 980 us).  Here both calls are as long as their kernels.
//
// These functions take only the plain forms: exact torch.Tensor objects with
// storage, in the accepted layouts, on the context's device, and rectangles
// that are tuples or lists of Python ints.  Anything else makes them return
// "not taken" without side effects; the caller then runs its own checks, which
// report what is wrong or accept the rarer forms.  Nothing is kept between
// calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/ec.h"

namespace {

PyObject *s_color, *s_depth, *s_pvp, *s_roi;

// New reference, or nullptr (no exception set).
struct Ref {
    PyObject* p;
    explicit Ref(PyObject* o) : p(o) { if (!p) PyErr_Clear(); }
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
};

// Item i of a list or tuple (nullptr past its end), held: reading an attribute
// may run Python code, which may take the item out of the list.
PyObject* item_of(PyObject* seq, Py_ssize_t i)
{
    if (i >= PySequence_Fast_GET_SIZE(seq)) return nullptr;
    PyObject* o = PySequence_Fast_GET_ITEM(seq, i);
    Py_INCREF(o);
    return o;
}

const at::Tensor* tensor_of(PyObject* o)
{
    if (!o || !THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || t.layout() != at::kStrided || !t.has_storage()) return nullptr;
    return &t;
}

bool on_device(const at::Tensor& t, int dev) { return t.is_cuda() && t.device().index() == dev; }

struct Layout {
    int fmt;
    int64_t pitch, w, h;
};

// The layouts of a colour tensor (see api.pixel_layout).
bool layout_of(const at::Tensor& t, Layout* l)
{
    const auto sz = t.sizes(), st = t.strides();
    const auto ty = t.scalar_type();
    if (sz.size() == 2 && (ty == at::kUInt32 || ty == at::kInt)) {
        if (st[1] != 1) return false;
        *l = Layout{EC_RGBA8, st[0], sz[1], sz[0]};
    } else if (sz.size() == 3 && sz[2] == 4 && (ty == at::kFloat || ty == at::kHalf)) {
        if (st[2] != 1 || st[1] != 4 || st[0] % 4) return false;
        *l = Layout{ty == at::kFloat ? EC_RGBA32F : EC_RGBA16F, st[0] / 4, sz[1], sz[0]};
    } else {
        return false;
    }
    return l->pitch >= 0 && l->pitch <= INT32_MAX && l->w <= INT32_MAX && l->h <= INT32_MAX;
}

// A rectangle given as a tuple or list of four ints; None is `none`.
bool rect_of(PyObject* o, const ec_rect& none, ec_rect* r)
{
    if (o == Py_None) { *r = none; return true; }
    const bool tup = PyTuple_CheckExact(o);
    if (!tup && !PyList_CheckExact(o)) return false;
    if ((tup ? PyTuple_GET_SIZE(o) : PyList_GET_SIZE(o)) != 4) return false;
    int32_t v[4];
    for (int k = 0; k < 4; ++k) {
        PyObject* e = tup ? PyTuple_GET_ITEM(o, k) : PyList_GET_ITEM(o, k);
        if (!PyLong_CheckExact(e)) return false;
        int over = 0;
        const long long x = PyLong_AsLongLongAndOverflow(e, &over);
        if (over || x < INT32_MIN || x > INT32_MAX) return false;
        v[k] = (int32_t)x;
    }
    *r = ec_rect{v[0], v[1], v[2], v[3]};
    return true;
}

// float32 [>= h][>= w] with unit column stride and the colour's pitch.
const at::Tensor* depth_of(PyObject* o, int dev, const Layout& l, int64_t w, int64_t h)
{
    const at::Tensor* t = tensor_of(o);
    if (!t || !on_device(*t, dev) || t->scalar_type() != at::kFloat || t->dim() != 2) return nullptr;
    if (t->stride(1) != 1 || t->stride(0) != l.pitch || t->size(0) < h || t->size(1) < w) return nullptr;
    return t;
}

enum { kNoDepth = 0, kDepth = 1, kAnyDepth = 2 };

bool image_of(PyObject* o, int dev, int need, ec_image* im, Layout* l)
{
    const Ref color(PyObject_GetAttr(o, s_color)), pvp(PyObject_GetAttr(o, s_pvp)), roi(PyObject_GetAttr(o, s_roi));
    const at::Tensor* t = tensor_of(color.p);
    if (!t || !pvp.p || !roi.p || !on_device(*t, dev) || !layout_of(*t, l)) return false;
    if (!rect_of(pvp.p, ec_rect{0, 0, (int32_t)l->w, (int32_t)l->h}, &im->pvp)) return false;
    if (!rect_of(roi.p, im->pvp, &im->roi)) return false;
    if (im->pvp.w > l->w || im->pvp.h > l->h) return false;
    im->pitch = (int32_t)l->pitch;
    im->format = l->fmt;
    im->color = t->data_ptr();
    im->depth = nullptr;
    if (need != kNoDepth) {
        const Ref depth(PyObject_GetAttr(o, s_depth));
        if (!depth.p) return false;
        if (depth.p != Py_None) {
            const at::Tensor* d = depth_of(depth.p, dev, *l, im->pvp.w, im->pvp.h);
            if (!d) return false;
            im->depth = static_cast<float*>(d->data_ptr());
        } else if (need == kDepth) {
            return false;
        }
    }
    return true;
}

// Runs f (which returns a Python object) with C++ exceptions turned into "not taken".
template <class F>
PyObject* taken(F f)
{
    try {
        return f();
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_FALSE;
    }
}

// images(seq, dev, need_depth, address): the ec_image array at address, one per
// image of the list or tuple; False if one is not plain.
PyObject* images(PyObject*, PyObject* args)
{
    PyObject* seq;
    int dev, need;
    unsigned long long at;
    if (!PyArg_ParseTuple(args, "OiiK", &seq, &dev, &need, &at)) return nullptr;
    if (!PyList_CheckExact(seq) && !PyTuple_CheckExact(seq)) Py_RETURN_FALSE;
    return taken([&]() -> PyObject* {
        ec_image* out = reinterpret_cast<ec_image*>((uintptr_t)at);
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
        Layout l;
        for (Py_ssize_t i = 0; i < n; ++i) {
            const Ref im(item_of(seq, i));
            if (!im.p || !image_of(im.p, dev, need, &out[i], &l)) Py_RETURN_FALSE;
        }
        Py_RETURN_TRUE;
    });
}

// gradients(grads, images, dev, address): checks one gradient buffer per image
// against its image's layout and writes the pointers; returns the shared
// format, or False.
PyObject* gradients(PyObject*, PyObject* args)
{
    PyObject *seq, *imgs;
    int dev;
    unsigned long long at;
    if (!PyArg_ParseTuple(args, "OOiK", &seq, &imgs, &dev, &at)) return nullptr;
    if (!(PyList_CheckExact(seq) || PyTuple_CheckExact(seq)) || !(PyList_CheckExact(imgs) || PyTuple_CheckExact(imgs)))
        Py_RETURN_FALSE;
    return taken([&]() -> PyObject* {
        void** out = reinterpret_cast<void**>((uintptr_t)at);
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
        if (n == 0 || n != PySequence_Fast_GET_SIZE(imgs)) Py_RETURN_FALSE;
        int fmt = -1;
        for (Py_ssize_t i = 0; i < n; ++i) {
            const Ref grad(item_of(seq, i)), im(item_of(imgs, i));
            if (!grad.p || !im.p) Py_RETURN_FALSE;
            const at::Tensor* g = tensor_of(grad.p);
            const Ref color(PyObject_GetAttr(im.p, s_color));
            const at::Tensor* c = tensor_of(color.p);
            Layout lg, lc;
            if (!g || !c || !on_device(*g, dev) || !layout_of(*g, &lg) || !layout_of(*c, &lc)) Py_RETURN_FALSE;
            if (lg.fmt == EC_RGBA8 || lg.pitch != lc.pitch || lg.w != lc.w || lg.h != lc.h) Py_RETURN_FALSE;
            if (fmt >= 0 && lg.fmt != fmt) Py_RETURN_FALSE;
            fmt = lg.fmt;
            out[i] = g->data_ptr();
        }
        return PyLong_FromLong(fmt);
    });
}

// target(color, depth or None, pvp or None, dev, address): the ec_target.
PyObject* target(PyObject*, PyObject* args)
{
    PyObject *color, *depth, *pvp;
    int dev;
    unsigned long long at;
    if (!PyArg_ParseTuple(args, "OOOiK", &color, &depth, &pvp, &dev, &at)) return nullptr;
    return taken([&]() -> PyObject* {
        ec_target* out = reinterpret_cast<ec_target*>((uintptr_t)at);
        const at::Tensor* t = tensor_of(color);
        Layout l;
        if (!t || !on_device(*t, dev) || !layout_of(*t, &l)) Py_RETURN_FALSE;
        if (!rect_of(pvp, ec_rect{0, 0, (int32_t)l.w, (int32_t)l.h}, &out->pvp)) Py_RETURN_FALSE;
        if (out->pvp.w > l.w || out->pvp.h > l.h) Py_RETURN_FALSE;
        out->pitch = (int32_t)l.pitch;
        out->format = l.fmt;
        out->color = t->data_ptr();
        out->depth = nullptr;
        if (depth != Py_None) {
            const at::Tensor* d = depth_of(depth, dev, l, out->pvp.w, out->pvp.h);
            if (!d) Py_RETURN_FALSE;
            out->depth = static_cast<float*>(d->data_ptr());
        }
        Py_RETURN_TRUE;
    });
}

// order(seq, n, address): n int32 values; False if one is not an int32.
PyObject* order(PyObject*, PyObject* args)
{
    PyObject* seq;
    Py_ssize_t n;
    unsigned long long at;
    if (!PyArg_ParseTuple(args, "OnK", &seq, &n, &at)) return nullptr;
    if (!PyList_CheckExact(seq) && !PyTuple_CheckExact(seq)) Py_RETURN_FALSE;
    if (PySequence_Fast_GET_SIZE(seq) != n) Py_RETURN_FALSE;
    int32_t* out = reinterpret_cast<int32_t*>((uintptr_t)at);
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject* e = PySequence_Fast_GET_ITEM(seq, i);
        if (!PyLong_CheckExact(e)) Py_RETURN_FALSE;
        int over = 0;
        const long long x = PyLong_AsLongLongAndOverflow(e, &over);
        if (over || x < INT32_MIN || x > INT32_MAX) Py_RETURN_FALSE;
        out[i] = (int32_t)x;
    }
    Py_RETURN_TRUE;
}

PyMethodDef methods[] = {{"images", images, METH_VARARGS, nullptr},
                         {"gradients", gradients, METH_VARARGS, nullptr},
                         {"target", target, METH_VARARGS, nullptr},
                         {"order", order, METH_VARARGS, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal()
{
    s_color = PyUnicode_InternFromString("color");
    s_depth = PyUnicode_InternFromString("depth");
    s_pvp = PyUnicode_InternFromString("pvp");
    s_roi = PyUnicode_InternFromString("roi");
    if (!s_color || !s_depth || !s_pvp || !s_roi) return nullptr;
    return PyModule_Create(&module);
}
