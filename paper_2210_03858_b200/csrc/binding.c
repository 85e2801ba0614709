/* CPython entry points for the calls a training step or a decode loop makes (see include/bcq.h).
 *
 * The GPU side of such a call can be as short as 3 us, so the way to it counts: a ctypes call with 15
 * arguments costs 2.3 us of the host, one of these 0.4 us (four decode calls of a small layer: 26 us
 * with ctypes, limited by the host; 13 us is what the GPU needs).  Arguments are integers (pointers
 * among them, None = NULL) and floats, in the order of the C functions; the result is the status.
 * load() resolves the functions from the library that is already loaded in the process. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <stddef.h>
#include <stdint.h>

typedef int (*fwd_fn)(int, int, int, int, int, const void*, size_t, const void*, const void*, const void*, void*, size_t, int, void*,
                      size_t, void*);
typedef int (*packed_fn)(int, int, int, int, int, const void*, size_t, void*, const void*, void*, size_t, int, void*, size_t, void*);
typedef int (*bwd_x_fn)(int, int, int, int, int, const void*, size_t, const void*, const void*, void*, size_t, int, void*, size_t,
                        void*);
typedef int (*bwd_alpha_fn)(int, int, int, int, int, const void*, size_t, const void*, size_t, const void*, uint32_t, float, int,
                            void*, void*, size_t, void*);
typedef int (*quantize_fn)(int, int, int, int, const void*, size_t, int, void*, void*, void*, void*);
typedef int (*adamw_fn)(long long, int, const void*, const void*, const void*, void*, const void*, void*, void*, long long, float,
                        float, float, float, float, float, void*);
typedef float (*lr_fn)(float, long long, long long, long long);
typedef int (*gather_fn)(long long, int, const void*, const void*, void*, void*, void*);

static fwd_fn f_fwd, f_fwd_prepared, f_decode;
static packed_fn f_packed;
static bwd_x_fn f_bwd_x, f_bwd_x_prepared;
static bwd_alpha_fn f_bwd_alpha;
static quantize_fn f_quantize;
static adamw_fn f_adamw;
static gather_fn f_pack, f_unpack;
static lr_fn f_lr;

static inline long long as_int(PyObject* o) { return o == Py_None ? 0 : PyLong_AsLongLong(o); }
static inline void* as_ptr(PyObject* o) { return o == Py_None ? NULL : PyLong_AsVoidPtr(o); }

#define I(k) (int)a_[k]
#define L(k) a_[k]
#define Z(k) (size_t)a_[k]
#define P(k) p_[k]

/* Bit k of `ptrs`: argument k is a pointer; of `floats`: a float; the others are integers. */
static int parse(PyObject* const* args, Py_ssize_t n, Py_ssize_t want, uint32_t ptrs, uint32_t floats, long long* a, void** p,
                 float* f) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
        return 0;
    }
    for (Py_ssize_t k = 0; k < n; ++k) {
        if ((ptrs >> k) & 1u) p[k] = as_ptr(args[k]);
        else if ((floats >> k) & 1u) f[k] = (float)PyFloat_AsDouble(args[k]);
        else a[k] = as_int(args[k]);
    }
    return PyErr_Occurred() == NULL;
}

#define BEGIN(want, ptrs, floats)                                                                \
    (void)self;                                                                                  \
    long long a_[want];                                                                          \
    void* p_[want];                                                                              \
    float f_[want];                                                                              \
    int st_;                                                                                     \
    if (!parse(args, n, want, ptrs, floats, a_, p_, f_)) return NULL;                            \
    Py_BEGIN_ALLOW_THREADS
#define END                                                                                      \
    Py_END_ALLOW_THREADS                                                                         \
    (void)a_; (void)p_; (void)f_;                                                                \
    return PyLong_FromLong(st_);

#define FWD(name)                                                                                \
    static PyObject* py_##name(PyObject* self, PyObject* const* args, Py_ssize_t n) {            \
        BEGIN(16, 0xA7A0u, 0u)                                                                   \
        st_ = f_##name(I(0), I(1), I(2), I(3), I(4), P(5), Z(6), P(7), P(8), P(9), P(10), Z(11), I(12), P(13), Z(14), P(15)); \
        END                                                                                      \
    }
FWD(fwd)
FWD(fwd_prepared)
FWD(decode)

static PyObject* py_packed(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    BEGIN(15, 0x53A0u, 0u)
    st_ = f_packed(I(0), I(1), I(2), I(3), I(4), P(5), Z(6), P(7), P(8), P(9), Z(10), I(11), P(12), Z(13), P(14));
    END
}

#define BWD_X(name)                                                                              \
    static PyObject* py_##name(PyObject* self, PyObject* const* args, Py_ssize_t n) {            \
        BEGIN(15, 0x53A0u, 0u)                                                                   \
        st_ = f_##name(I(0), I(1), I(2), I(3), I(4), P(5), Z(6), P(7), P(8), P(9), Z(10), I(11), P(12), Z(13), P(14)); \
        END                                                                                      \
    }
BWD_X(bwd_x)
BWD_X(bwd_x_prepared)

static PyObject* py_bwd_alpha(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    BEGIN(17, 0x162A0u, 0x800u)
    st_ = f_bwd_alpha(I(0), I(1), I(2), I(3), I(4), P(5), Z(6), P(7), Z(8), P(9), (uint32_t)L(10), f_[11], I(12), P(13), P(14),
                      Z(15), P(16));
    END
}

static PyObject* py_quantize(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    BEGIN(11, 0x790u, 0u)
    st_ = f_quantize(I(0), I(1), I(2), I(3), P(4), Z(5), I(6), P(7), P(8), P(9), P(10));
    END
}

static PyObject* py_adamw(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    BEGIN(17, 0x101FCu, 0xFC00u)
    st_ = f_adamw(L(0), I(1), P(2), P(3), P(4), P(5), P(6), P(7), P(8), L(9), f_[10], f_[11], f_[12], f_[13], f_[14], f_[15], P(16));
    END
}

#define GATHER(name)                                                                             \
    static PyObject* py_##name(PyObject* self, PyObject* const* args, Py_ssize_t n) {            \
        BEGIN(7, 0x7Cu, 0u)                                                                      \
        st_ = f_##name(L(0), I(1), P(2), P(3), P(4), P(5), P(6));                                \
        END                                                                                      \
    }
GATHER(pack)
GATHER(unpack)

/* The learning rate of a step (one call per optimiser step; through ctypes 1.1 us, here 0.1).  Steps have to be integers. */
static PyObject* py_lr_linear_decay(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    if (n != 4 || !PyLong_Check(args[1]) || !PyLong_Check(args[2]) || !PyLong_Check(args[3])) {
        PyErr_SetString(PyExc_TypeError, "a float and three integers expected");
        return NULL;
    }
    const float lr0 = (float)PyFloat_AsDouble(args[0]);
    long long k[3];
    for (int i = 0; i < 3; ++i) k[i] = PyLong_AsLongLong(args[1 + i]);
    if (PyErr_Occurred() != NULL) return NULL;
    return PyFloat_FromDouble((double)f_lr(lr0, k[0], k[1], k[2]));
}

static PyObject* py_load(PyObject* self, PyObject* path) {
    (void)self;
    const char* file = PyUnicode_AsUTF8(path);
    if (file == NULL) return NULL;
    void* h = dlopen(file, RTLD_NOW);
    if (h == NULL) {
        PyErr_SetString(PyExc_RuntimeError, dlerror());
        return NULL;
    }
    const struct { const char* name; void* slot; } table[] = {
        {"bcq_linear_fwd", &f_fwd}, {"bcq_linear_fwd_prepared", &f_fwd_prepared}, {"bcq_linear_decode", &f_decode},
        {"bcq_linear_decode_packed", &f_packed}, {"bcq_linear_bwd_x", &f_bwd_x},
        {"bcq_linear_bwd_x_prepared", &f_bwd_x_prepared}, {"bcq_linear_bwd_alpha", &f_bwd_alpha},
        {"bcq_quantize", &f_quantize}, {"bcq_alpha_adamw", &f_adamw}, {"bcq_alpha_pack", &f_pack},
        {"bcq_alpha_unpack", &f_unpack}, {"bcq_lr_linear_decay", &f_lr},
    };
    for (size_t k = 0; k < sizeof(table) / sizeof(table[0]); ++k) {
        void* sym = dlsym(h, table[k].name);
        if (sym == NULL) {
            PyErr_Format(PyExc_RuntimeError, "%s is missing from %s", table[k].name, file);
            return NULL;
        }
        *(void**)table[k].slot = sym;
    }
    Py_RETURN_NONE;
}

#define M(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    M(fwd), M(fwd_prepared), M(decode), M(packed), M(bwd_x), M(bwd_x_prepared), M(bwd_alpha), M(quantize), M(adamw), M(pack),
    M(unpack), M(lr_linear_decay), {"load", py_load, METH_O, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_bcq_call", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__bcq_call(void) { return PyModule_Create(&module); }
