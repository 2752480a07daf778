/* CPython extension of the binding: walks grammar and sketch models and fills the C descriptors of include/xp.h.
 *
 * A batch load marshals thousands of productions and holes; done field by field through ctypes that took longer than the
 * GPU's part of the load (1024 small sketches: 40 ms); so do Python-level constructors, finalisers and ctypes calls per
 * object (1024 grammars, loads and results: 21.7 -> 18.8 ms).  Nothing here evaluates, counts or ranks candidates.
 *
 *   grammar(g)                         -> (address of an xp_grammar_desc, owner)
 *   sketches(list, conv, coords, specs) -> (address of the xp_sketch_desc array, owner, holes per sketch, device tensors per sketch)
 *   code(list)                         -> bytes of xp_instr
 *   grammar_create(create, destroy, class, g), loaded(destroy, addresses, class, grammars, holes, tensors),
 *   hole_results(get, class, fields, result, first, n)  -> instances of the binding's classes, made without running Python code;
 *                                         the functions of the library are passed as addresses
 *   handle(destroy, address), free_all(destroy, addresses, n)
 *
 * The owner object frees the memory behind the address; it also holds the arrays the descriptors point into.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdlib.h>
#include <string.h>

#include "xp.h"

static PyObject *s_variables, *s_name, *s_lo, *s_hi, *s_n_nonterminals, *s_productions, *s_lhs, *s_kind, *s_var, *s_op, *s_left, *s_right, *s_value,
    *s_holes, *s_coords, *s_start_nt, *s_max_size, *s_ctx, *s_spec_expr, *s_spec_table, *s_data_ptr, *s_is_cuda, *s_shape,
    *s_dtype, *s_own, *s_handle, *s_model, *s_grammar, *s_n_holes, *s_keep;

/* What a marshalled description owns: one block of memory and a list of the objects it points into. */
typedef struct { PyObject_HEAD void* mem; PyObject* held; } Owner;

static void owner_dealloc(Owner* o) {
    free(o->mem);
    Py_XDECREF(o->held);
    Py_TYPE(o)->tp_free((PyObject*)o);
}

static PyTypeObject OwnerType = {
    PyVarObject_HEAD_INIT(NULL, 0).tp_name = "_marshal.Owner", .tp_basicsize = sizeof(Owner), .tp_flags = Py_TPFLAGS_DEFAULT,
    .tp_dealloc = (destructor)owner_dealloc, .tp_doc = "Memory of a marshalled description.",
};

static Owner* new_owner(size_t bytes) {
    Owner* o = PyObject_New(Owner, &OwnerType);
    if (!o) return NULL;
    o->mem = calloc(1, bytes ? bytes : 1);
    o->held = PyList_New(0);
    if (!o->mem || !o->held) {
        Py_DECREF(o);
        PyErr_NoMemory();
        return NULL;
    }
    return o;
}

/* An integer (int, numpy integer, anything with __index__; no floats, no texts) between -2^63 and 2^64 - 1 as 64 bits: an unsigned
 * constant wraps, as it does in the C structures.  Returns -1 with an exception set on failure. */
static inline int as_int64(PyObject* v, long long* out) {
    if (PyLong_CheckExact(v)) {
        int over = 0;
        *out = PyLong_AsLongLongAndOverflow(v, &over);
        if (over == 0) return 0;
    }
    PyObject* i = PyNumber_Index(v);
    if (!i) return -1;
    int over = 0;
    long long r = PyLong_AsLongLongAndOverflow(i, &over);
    if (over > 0) r = (long long)PyLong_AsUnsignedLongLong(i);
    else if (over < 0) PyErr_SetString(PyExc_OverflowError, "an integer below -2^63");
    Py_DECREF(i);
    *out = r;
    return PyErr_Occurred() ? -1 : 0;
}

static inline int get_int64(PyObject* obj, PyObject* name, int64_t* out) {
    PyObject* v = PyObject_GetAttr(obj, name);
    long long r = 0;
    const int rc = v ? as_int64(v, &r) : -1;
    Py_XDECREF(v);
    *out = r;
    return rc;
}

static inline int get_int32(PyObject* obj, PyObject* name, int32_t* out) {      /* (the low 32 bits: as the C structures take an int) */
    int64_t r = 0;
    const int rc = get_int64(obj, name, &r);
    *out = (int32_t)r;
    return rc;
}

static int fill_instrs(PyObject* seq, xp_instr* out, Py_ssize_t n) {
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject* t = PySequence_Fast(PySequence_Fast_GET_ITEM(seq, i), "an instruction is a (kind, arg, value) tuple");
        if (!t) return -1;
        if (PySequence_Fast_GET_SIZE(t) != 3) {
            Py_DECREF(t);
            PyErr_SetString(PyExc_ValueError, "an instruction is a (kind, arg, value) tuple");
            return -1;
        }
        long long v[3] = {0, 0, 0};
        int rc = 0;
        for (int k = 0; k < 3 && rc == 0; ++k) rc = as_int64(PySequence_Fast_GET_ITEM(t, k), &v[k]);
        Py_DECREF(t);
        if (rc < 0) return -1;
        out[i].kind = (int32_t)v[0];
        out[i].arg = (int32_t)v[1];
        out[i].value = v[2];
    }
    return 0;
}

static PyObject* m_code(PyObject* self, PyObject* arg) {
    (void)self;
    PyObject* seq = PySequence_Fast(arg, "postfix code is a list");
    if (!seq) return NULL;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    PyObject* out = PyBytes_FromStringAndSize(NULL, (Py_ssize_t)sizeof(xp_instr) * n);
    if (out && fill_instrs(seq, (xp_instr*)PyBytes_AS_STRING(out), n) < 0) Py_CLEAR(out);
    Py_DECREF(seq);
    return out;
}

/* A grammar model's lists, and its descriptor in memory that follows them: sizes first, then the fields. */
typedef struct { PyObject *vars, *prods; Py_ssize_t nv, np; } GrammarLists;

static int grammar_lists(PyObject* g, GrammarLists* l) {
    l->vars = l->prods = NULL;
    for (int k = 0; k < 2; ++k) {
        PyObject* tmp = PyObject_GetAttr(g, k ? s_productions : s_variables);
        if (!tmp) return -1;
        PyObject* f = PySequence_Fast(tmp, k ? "productions is a list" : "variables is a list");
        Py_DECREF(tmp);
        if (!f) return -1;
        if (k) l->prods = f;
        else l->vars = f;
    }
    l->nv = PySequence_Fast_GET_SIZE(l->vars);
    l->np = PySequence_Fast_GET_SIZE(l->prods);
    return 0;
}

static size_t grammar_bytes(const GrammarLists* l) {
    return sizeof(xp_grammar_desc) + sizeof(xp_production) * (size_t)l->np + (sizeof(xp_variable) + sizeof(PyObject*)) * (size_t)l->nv;
}

/* Fills `mem` (zeroed).  names[i] receives the name object that vars[i].name points into. */
static int fill_grammar(PyObject* g, const GrammarLists* l, void* mem, PyObject*** names_out) {
    xp_grammar_desc* d = (xp_grammar_desc*)mem;
    xp_production* p = (xp_production*)(d + 1);
    xp_variable* v = (xp_variable*)(p + l->np);
    PyObject** names = (PyObject**)(v + l->nv);
    *names_out = names;
    d->n_vars = (int32_t)l->nv;
    d->vars = v;
    if (get_int32(g, s_n_nonterminals, &d->n_nonterminals) < 0) return -1;
    d->n_productions = (int32_t)l->np;
    d->productions = p;
    for (Py_ssize_t i = 0; i < l->nv; ++i) {
        PyObject* x = PySequence_Fast_GET_ITEM(l->vars, i);
        names[i] = PyObject_GetAttr(x, s_name);
        if (names[i] && !PyUnicode_Check(names[i])) PyErr_SetString(PyExc_TypeError, "a variable's name is a string");
        v[i].name = names[i] && PyUnicode_Check(names[i]) ? PyUnicode_AsUTF8(names[i]) : NULL;
        if (!v[i].name || get_int64(x, s_lo, &v[i].lo) < 0 || get_int64(x, s_hi, &v[i].hi) < 0) return -1;
    }
    for (Py_ssize_t i = 0; i < l->np; ++i) {
        PyObject* x = PySequence_Fast_GET_ITEM(l->prods, i);
        if (get_int32(x, s_kind, &p[i].kind) < 0 || get_int32(x, s_lhs, &p[i].lhs) < 0) return -1;
        const int rc = p[i].kind == XP_PROD_CONST ? get_int64(x, s_value, &p[i].value)      /* (each kind reads its own fields) */
                     : p[i].kind == XP_PROD_VAR ? get_int32(x, s_var, &p[i].var)
                     : get_int32(x, s_op, &p[i].op) < 0 || get_int32(x, s_left, &p[i].left) < 0 ? -1 : get_int32(x, s_right, &p[i].right);
        if (rc < 0) return -1;
    }
    return 0;
}

static PyObject* m_grammar(PyObject* self, PyObject* g) {
    (void)self;
    PyObject *ret = NULL, **names = NULL;
    GrammarLists l;
    Owner* o = grammar_lists(g, &l) == 0 ? new_owner(grammar_bytes(&l)) : NULL;
    if (o) {
        int rc = fill_grammar(g, &l, o->mem, &names);
        for (Py_ssize_t i = 0; i < l.nv; ++i) {
            if (names[i] && PyList_Append(o->held, names[i]) < 0) rc = -1;
            Py_XDECREF(names[i]);                        /* (the list holds it) */
        }
        if (rc == 0) ret = Py_BuildValue("(KO)", (unsigned long long)(size_t)o->mem, (PyObject*)o);
    }
    Py_XDECREF((PyObject*)o);
    Py_XDECREF(l.vars);
    Py_XDECREF(l.prods);
    return ret;
}

/* Something the library made: destroyed with this object. */
typedef struct { PyObject_HEAD void (*destroy)(void*); void* at; } Handle;

static void handle_dealloc(Handle* h) {
    void (*destroy)(void*) = h->destroy;
    void* at = h->at;
    Py_TYPE(h)->tp_free((PyObject*)h);
    if (!at || !destroy) return;
    Py_BEGIN_ALLOW_THREADS
    destroy(at);
    Py_END_ALLOW_THREADS
}

static PyTypeObject HandleType = {
    PyVarObject_HEAD_INIT(NULL, 0).tp_name = "_marshal.Handle", .tp_basicsize = sizeof(Handle), .tp_flags = Py_TPFLAGS_DEFAULT,
    .tp_dealloc = (destructor)handle_dealloc, .tp_doc = "Something the library made; destroyed with this object.",
};

static PyObject* new_handle(unsigned long long destroy, void* at) {
    Handle* h = PyObject_New(Handle, &HandleType);
    if (!h) return NULL;
    h->destroy = (void (*)(void*))(size_t)destroy;
    h->at = at;
    return (PyObject*)h;
}

static PyObject* m_handle(PyObject* self, PyObject* args) {
    (void)self;
    unsigned long long destroy, at;
    if (!PyArg_ParseTuple(args, "KK", &destroy, &at)) return NULL;
    return new_handle(destroy, (void*)(size_t)at);
}

/* obj.name = value; takes the reference (NULL: an exception is set). */
static int put(PyObject* obj, PyObject* name, PyObject* value) {
    const int rc = value ? PyObject_SetAttr(obj, name, value) : -1;
    Py_XDECREF(value);
    return rc;
}

/* An instance of `cls` without a call of its __init__. */
static PyObject* blank(PyObject* cls) {
    PyObject* none = PyTuple_New(0);
    PyObject* obj = none ? ((PyTypeObject*)cls)->tp_new((PyTypeObject*)cls, none, NULL) : NULL;
    Py_XDECREF(none);
    return obj;
}

/* A new instance of the Python class `cls` that owns the library object `at`. */
static PyObject* owning(PyObject* cls, unsigned long long destroy, void* at) {
    PyObject* own = new_handle(destroy, at);             /* (first: whatever fails from here on, `at` is destroyed) */
    if (!own) return NULL;
    PyObject* obj = blank(cls);
    if (!obj) { Py_DECREF(own); return NULL; }
    if (put(obj, s_own, own) < 0 || put(obj, s_handle, PyLong_FromVoidPtr(at)) < 0) Py_CLEAR(obj);
    return obj;
}

static PyObject* m_grammar_create(PyObject* self, PyObject* args) {
    (void)self;
    unsigned long long create, destroy;
    PyObject *cls, *g, *ret = NULL, **names = NULL;
    if (!PyArg_ParseTuple(args, "KKO!O", &create, &destroy, &PyType_Type, &cls, &g)) return NULL;
    GrammarLists l;
    _Alignas(16) char room[4096];                        /* (most grammars fit) */
    void* mem = NULL;
    if (grammar_lists(g, &l) == 0) {
        const size_t bytes = grammar_bytes(&l);
        mem = bytes <= sizeof(room) ? memset(room, 0, bytes) : calloc(1, bytes);
        if (!mem) PyErr_NoMemory();
        else {
            void* at = NULL;
            if (fill_grammar(g, &l, mem, &names) == 0) {
                int st;
                Py_BEGIN_ALLOW_THREADS                   /* (what `mem` points into is held by `names`) */
                st = ((int (*)(const xp_grammar_desc*, void**))(size_t)create)((const xp_grammar_desc*)mem, &at);
                Py_END_ALLOW_THREADS
                if (st != 0) ret = PyLong_FromLong(st);
                else {
                    ret = owning(cls, destroy, at);
                    if (ret && put(ret, s_model, Py_NewRef(g)) < 0) Py_CLEAR(ret);
                }
            }
            for (Py_ssize_t i = 0; i < l.nv; ++i) Py_XDECREF(names[i]);
            if (mem != (void*)room) free(mem);
        }
    }
    Py_XDECREF(l.vars);
    Py_XDECREF(l.prods);
    return ret;
}

/* Instances of `cls` for n loaded sketches. */
static PyObject* m_loaded(PyObject* self, PyObject* args) {
    (void)self;
    unsigned long long destroy, address;
    PyObject *cls, *grs, *nhs, *keeps;
    if (!PyArg_ParseTuple(args, "KKO!OO!O!", &destroy, &address, &PyType_Type, &cls, &grs, &PyList_Type, &nhs, &PyList_Type, &keeps)) return NULL;
    void** at = (void**)(size_t)address;
    const Py_ssize_t n = PyList_GET_SIZE(nhs);
    PyObject* seq = PySequence_Fast(grs, "grammars is a list");
    PyObject* out = seq ? PyList_New(n) : NULL;
    int rc = out ? 0 : -1;
    if (rc == 0 && (PySequence_Fast_GET_SIZE(seq) != n || PyList_GET_SIZE(keeps) != n)) {
        PyErr_SetString(PyExc_ValueError, "lists of one length were expected");
        rc = -1;
    }
    for (Py_ssize_t i = 0; out && i < n; ++i) {
        PyObject* obj = owning(cls, destroy, at[i]);     /* (also after a failure: every sketch gets its owner) */
        if (!obj) { rc = -1; continue; }
        PyList_SET_ITEM(out, i, obj);
        if (rc < 0) continue;
        if (put(obj, s_grammar, Py_NewRef(PySequence_Fast_GET_ITEM(seq, i))) < 0 || put(obj, s_n_holes, Py_NewRef(PyList_GET_ITEM(nhs, i))) < 0 ||
            put(obj, s_keep, Py_NewRef(PyList_GET_ITEM(keeps, i))) < 0) rc = -1;
    }
    Py_XDECREF(seq);
    if (rc < 0) Py_CLEAR(out);
    return out;
}

/* destroy(address[0 .. n)) */
static PyObject* m_free_all(PyObject* self, PyObject* args) {
    (void)self;
    unsigned long long destroy, address;
    Py_ssize_t n;
    if (!PyArg_ParseTuple(args, "KKn", &destroy, &address, &n)) return NULL;
    void** at = (void**)(size_t)address;
    Py_BEGIN_ALLOW_THREADS
    for (Py_ssize_t i = 0; i < n; ++i) ((void (*)(void*))(size_t)destroy)(at[i]);
    Py_END_ALLOW_THREADS
    Py_RETURN_NONE;
}

/* Address and row count of an array with `itemsize`-byte integers; *held receives the object that has to stay alive.
 * A host array goes by the buffer protocol (conv(array, itemsize) first when it is not contiguous or of another type);
 * anything else is a torch tensor. */
static int array_at(PyObject* a, Py_ssize_t itemsize, PyObject* conv, const void** ptr, int32_t* on_device, long long* rows, PyObject** held) {
    Py_buffer b;
    *on_device = 0;
    static PyTypeObject* array_type = NULL;              /* the type seen last that is an array and not just any buffer */
    if (Py_TYPE(a) != array_type && PyObject_CheckBuffer(a) && PyObject_HasAttr(a, s_dtype)) array_type = (PyTypeObject*)Py_NewRef(Py_TYPE(a));
    if (Py_TYPE(a) == array_type) {
        Py_INCREF(a);
        for (int tries = 0; tries < 2; ++tries) {
            if (PyObject_GetBuffer(a, &b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) == 0) {
                const char* f = b.format ? b.format : "B";
                if (*f == '<' || *f == '=' || *f == '@') ++f;
                const int ok = b.itemsize == itemsize && (*f == 'i' || *f == 'l' || *f == 'q') && f[1] == 0 && b.ndim >= 1;
                if (ok) {
                    *ptr = b.buf;
                    *rows = (long long)b.shape[0];
                    PyBuffer_Release(&b);
                    *held = a;
                    return 0;
                }
                PyBuffer_Release(&b);
            } else PyErr_Clear();
            PyObject* c = tries == 0 ? PyObject_CallFunction(conv, "On", a, itemsize) : NULL;
            Py_DECREF(a);
            if (!c) {
                if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "cannot use this array");
                return -1;
            }
            a = c;
        }
        Py_DECREF(a);
        return -1;
    }
    PyObject* p = PyObject_CallMethodNoArgs(a, s_data_ptr);
    PyObject* c = p ? PyObject_GetAttr(a, s_is_cuda) : NULL;
    PyObject* s = c ? PyObject_GetAttr(a, s_shape) : NULL;
    PyObject* r = s ? PySequence_GetItem(s, 0) : NULL;
    if (r) {
        *ptr = (const void*)(size_t)PyLong_AsUnsignedLongLong(p);
        *on_device = PyObject_IsTrue(c);
        *rows = PyLong_AsLongLong(r);
    }
    Py_XDECREF(p);
    Py_XDECREF(c);
    Py_XDECREF(s);
    Py_XDECREF(r);
    if (!r || PyErr_Occurred()) return -1;
    Py_INCREF(a);
    *held = a;
    return 0;
}

static PyObject* get_list(PyObject* obj, PyObject* name, int may_be_none) {       /* obj.name as a fast sequence (None, where it may be: empty) */
    PyObject* v = PyObject_GetAttr(obj, name);
    if (!v) return NULL;
    if (v == Py_None && may_be_none) {
        Py_DECREF(v);
        return PyList_New(0);
    }
    PyObject* f = PySequence_Fast(v, "a list was expected");
    Py_DECREF(v);
    return f;
}

static PyObject* m_sketches(PyObject* self, PyObject* args) {
    (void)self;
    PyObject *list, *conv, *coords_arg, *specs_arg;
    if (!PyArg_ParseTuple(args, "OOOO", &list, &conv, &coords_arg, &specs_arg)) return NULL;
    PyObject* seq = PySequence_Fast(list, "sketches is a list");
    if (!seq) return NULL;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    PyObject *ret = NULL, *nhs = NULL, *devs = NULL;
    Owner* o = NULL;
    /* first walk: how many holes and instructions */
    size_t n_holes = 0, n_instr = 0;
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject* holes = get_list(PySequence_Fast_GET_ITEM(seq, i), s_holes, 0);
        if (!holes) goto done;
        const Py_ssize_t nh = PySequence_Fast_GET_SIZE(holes);
        n_holes += (size_t)nh;
        for (Py_ssize_t h = 0; h < nh; ++h)
            for (int k = 0; k < 2; ++k) {
                PyObject* c = get_list(PySequence_Fast_GET_ITEM(holes, h), k ? s_spec_expr : s_ctx, k);
                if (!c) { Py_DECREF(holes); goto done; }
                n_instr += (size_t)PySequence_Fast_GET_SIZE(c);
                Py_DECREF(c);
            }
        Py_DECREF(holes);
    }
    o = new_owner(sizeof(xp_sketch_desc) * (size_t)n + sizeof(xp_hole_desc) * n_holes + sizeof(xp_instr) * n_instr);
    nhs = PyList_New(n);
    devs = PyList_New(n);
    if (!o || !nhs || !devs) goto done;
    xp_sketch_desc* d = (xp_sketch_desc*)o->mem;
    xp_hole_desc* hd = (xp_hole_desc*)(d + n);
    xp_instr* code = (xp_instr*)(hd + n_holes);
    const xp_instr* code_end = code + n_instr;
    for (Py_ssize_t i = 0; i < n; ++i, ++d) {
        PyObject* sk = PySequence_Fast_GET_ITEM(seq, i);
        PyObject* dev = PyList_New(0);
        if (!dev) goto done;
        PyList_SET_ITEM(devs, i, dev);
        PyObject* holes = get_list(sk, s_holes, 0);
        if (!holes) goto done;
        const Py_ssize_t nh = PySequence_Fast_GET_SIZE(holes);
        PyList_SET_ITEM(nhs, i, PyLong_FromSsize_t(nh));
        d->n_holes = (int32_t)nh;
        d->holes = hd;
        int bad = 0;
        for (Py_ssize_t h = 0; h < nh && !bad; ++h, ++hd) {
            PyObject* ho = PySequence_Fast_GET_ITEM(holes, h);
            if (get_int32(ho, s_start_nt, &hd->start_nt) < 0 || get_int32(ho, s_max_size, &hd->max_size) < 0) { bad = 1; break; }
            PyObject* table = NULL;
            if (specs_arg != Py_None) {
                PyObject* key = PyLong_FromSsize_t(h);
                table = key ? PyObject_GetItem(specs_arg, key) : NULL;
                Py_XDECREF(key);
                if (!table) PyErr_Clear();               /* (not overridden) */
            }
            if (!table) table = PyObject_GetAttr(ho, s_spec_table);
            if (!table) { bad = 1; break; }
            for (int k = 0; k < 2 && !bad; ++k) {
                if (k == 1 && table != Py_None) break;   /* a table: the expression is not looked at */
                PyObject* c = get_list(ho, k ? s_spec_expr : s_ctx, 0);
                const Py_ssize_t len = c ? PySequence_Fast_GET_SIZE(c) : 0;
                if (!c || len > code_end - code || fill_instrs(c, code, len) < 0) bad = 1;
                else if (k) { hd->spec_kind = XP_SPEC_EXPR; hd->spec_len = (int32_t)len; hd->spec_expr = code; }
                else { hd->ctx_len = (int32_t)len; hd->ctx = code; }
                code += len;
                Py_XDECREF(c);
            }
            if (!bad && table != Py_None) {
                const void* ptr = NULL;
                long long rows = 0;
                PyObject* held = NULL;
                hd->spec_kind = XP_SPEC_TABLE;
                if (array_at(table, 8, conv, &ptr, &hd->spec_table_on_device, &rows, &held) < 0) bad = 1;
                else {
                    hd->spec_table = (const int64_t*)ptr;
                    if (PyList_Append(hd->spec_table_on_device ? dev : o->held, held) < 0) bad = 1;
                    Py_DECREF(held);
                }
            }
            Py_DECREF(table);
        }
        Py_DECREF(holes);
        if (bad) goto done;
        PyObject* co = coords_arg != Py_None ? Py_NewRef(coords_arg) : PyObject_GetAttr(sk, s_coords);
        if (!co) goto done;
        if (co != Py_None) {
            const void* ptr = NULL;
            long long rows = 0;
            PyObject* held = NULL;
            int rc = array_at(co, 4, conv, &ptr, &d->coords_on_device, &rows, &held);
            if (rc == 0) {
                d->domain_kind = XP_DOMAIN_TABLE;
                d->n_points = rows;
                d->coords = (const int32_t*)ptr;
                rc = PyList_Append(d->coords_on_device ? dev : o->held, held);
                Py_DECREF(held);
            }
            if (rc < 0) { Py_DECREF(co); goto done; }
        }
        Py_DECREF(co);
    }
    if (PyErr_Occurred()) goto done;
    ret = Py_BuildValue("(KOOO)", (unsigned long long)(size_t)o->mem, (PyObject*)o, nhs, devs);
done:
    if (!ret && !PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "malformed sketch");
    Py_XDECREF((PyObject*)o);
    Py_XDECREF(nhs);
    Py_XDECREF(devs);
    Py_DECREF(seq);
    return ret;
}

/* The results of holes [first, first + n) of a result handle as a list of `cls` (whose fields are `names`); the status where
 * the library refuses one. */
static PyObject* m_hole_results(PyObject* self, PyObject* args) {
    (void)self;
    unsigned long long get, handle;
    PyObject *cls, *names;
    int first, n;
    if (!PyArg_ParseTuple(args, "KO!O!Kii", &get, &PyType_Type, &cls, &PyTuple_Type, &names, &handle, &first, &n)) return NULL;
    PyObject* out = PyList_New(n > 0 ? n : 0);
    for (int h = 0; out && h < n; ++h) {
        xp_result_view v;
        memset(&v, 0, sizeof(v));
        const int st = ((int (*)(void*, int32_t, xp_result_view*))(size_t)get)((void*)(size_t)handle, first + h, &v);
        if (st != 0) {
            Py_DECREF(out);
            return PyLong_FromLong(st);
        }
        const Py_ssize_t K = v.max_size + 1;
        PyObject *cand = PyList_New(K), *match = PyList_New(K), *code = PyList_New(v.least_len);
        for (Py_ssize_t k = 0; cand && match && k < K; ++k) {
            PyList_SET_ITEM(cand, k, PyLong_FromUnsignedLongLong(v.cand_count[k]));
            PyList_SET_ITEM(match, k, PyLong_FromUnsignedLongLong(v.match_count[k]));
        }
        for (Py_ssize_t k = 0; code && k < v.least_len; ++k)
            PyList_SET_ITEM(code, k, Py_BuildValue("(iiL)", (int)v.least_code[k].kind, (int)v.least_code[k].arg, (long long)v.least_code[k].value));
        PyObject* field[] = {PyBool_FromLong(v.solved), cand, match, PyLong_FromLong(v.least_size), PyLong_FromUnsignedLongLong(v.least_rank),
                             PyUnicode_FromString(v.solved ? v.least_text : ""), code, PyLong_FromUnsignedLongLong(v.evals_executed),
                             PyLong_FromUnsignedLongLong(v.filter_survivors), PyLong_FromUnsignedLongLong(v.probe_survivors),
                             PyLong_FromUnsignedLongLong(v.nominal_ops), PyFloat_FromDouble(v.kernel_ms), PyFloat_FromDouble(v.total_ms),
                             PyLong_FromLong(v.n_launches), PyLong_FromUnsignedLongLong(v.filter_tests),
                             PyLong_FromUnsignedLongLong(v.candidates_skipped), PyLong_FromUnsignedLongLong(v.h2d_bytes),
                             PyLong_FromUnsignedLongLong(v.d2h_bytes)};
        const Py_ssize_t nf = (Py_ssize_t)(sizeof(field) / sizeof(field[0]));
        PyObject* obj = PyTuple_GET_SIZE(names) == nf ? blank(cls) : NULL;
        if (!obj && !PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "a hole result has other fields");
        int rc = obj ? 0 : -1;
        for (Py_ssize_t k = 0; k < nf; ++k) {
            if (rc == 0) rc = put(obj, PyTuple_GET_ITEM(names, k), field[k]);
            else Py_XDECREF(field[k]);
        }
        if (rc < 0) {
            Py_XDECREF(obj);
            Py_CLEAR(out);
        } else PyList_SET_ITEM(out, h, obj);
    }
    return out;
}

static PyMethodDef methods[] = {
    {"grammar", m_grammar, METH_O, "Grammar model -> (descriptor address, owner)."},
    {"sketches", m_sketches, METH_VARARGS, "Sketch models -> (descriptors' address, owner, holes per sketch, device tensors per sketch)."},
    {"code", m_code, METH_O, "Postfix list -> xp_instr bytes."},
    {"handle", m_handle, METH_VARARGS, "(address of a destroy function, address) -> owner."},
    {"grammar_create", m_grammar_create, METH_VARARGS, "Grammar model -> instance of a class, or the status of the library's refusal."},
    {"loaded", m_loaded, METH_VARARGS, "Addresses of loaded sketches -> instances of a class."},
    {"free_all", m_free_all, METH_VARARGS, "Destroys an array of library objects."},
    {"hole_results", m_hole_results, METH_VARARGS, "Results of a handle's holes -> instances of a class."},
    {NULL, NULL, 0, NULL},
};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", "Descriptors of include/xp.h from Python models.", -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void) {
    static const struct { PyObject** to; const char* name; } names[] = {
        {&s_variables, "variables"}, {&s_name, "name"}, {&s_lo, "lo"}, {&s_hi, "hi"}, {&s_n_nonterminals, "n_nonterminals"},
        {&s_productions, "productions"}, {&s_lhs, "lhs"}, {&s_kind, "kind"}, {&s_var, "var"}, {&s_op, "op"}, {&s_left, "left"},
        {&s_right, "right"}, {&s_value, "value"}, {&s_holes, "holes"}, {&s_coords, "coords"}, {&s_start_nt, "start_nt"},
        {&s_max_size, "max_size"}, {&s_ctx, "ctx"}, {&s_spec_expr, "spec_expr"}, {&s_spec_table, "spec_table"},
        {&s_data_ptr, "data_ptr"}, {&s_is_cuda, "is_cuda"}, {&s_shape, "shape"}, {&s_dtype, "dtype"}, {&s_own, "_own"},
        {&s_handle, "handle"}, {&s_model, "model"}, {&s_grammar, "grammar"}, {&s_n_holes, "n_holes"}, {&s_keep, "_keep"}};
    for (size_t i = 0; i < sizeof(names) / sizeof(names[0]); ++i) {
        *names[i].to = PyUnicode_InternFromString(names[i].name);
        if (!*names[i].to) return NULL;
    }
    if (PyType_Ready(&OwnerType) < 0 || PyType_Ready(&HandleType) < 0) return NULL;
    return PyModule_Create(&module);
}
