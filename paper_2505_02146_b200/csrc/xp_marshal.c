/* CPython extension of the binding: walks grammar and sketch models and fills the C descriptors of include/xp.h.
 *
 * A batch load marshals thousands of productions and holes; done field by field through ctypes that took longer than the
 * GPU's part of the load (1024 small sketches: 40 ms).  Nothing here evaluates, counts or ranks candidates.
 *
 *   grammar(g)                         -> (address of an xp_grammar_desc, owner)
 *   sketches(list, conv, coords, specs) -> (address of the xp_sketch_desc array, owner, holes per sketch, device tensors per sketch)
 *   code(list)                         -> bytes of xp_instr
 *   hole_result(address of an xp_result_view) -> tuple of a hole result's fields
 *
 * The owner object frees the memory behind the address; it also holds the arrays the descriptors point into.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdlib.h>
#include <string.h>

#include "xp.h"

static PyObject *s_variables, *s_name, *s_lo, *s_hi, *s_n_nonterminals, *s_productions, *s_lhs, *s_kind, *s_var, *s_op, *s_left, *s_right, *s_value,
    *s_holes, *s_coords, *s_start_nt, *s_max_size, *s_ctx, *s_spec_expr, *s_spec_table, *s_data_ptr, *s_is_cuda, *s_shape;

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

/* obj.name as an integer; -1 with an exception set on failure. */
static long long int_attr(PyObject* obj, PyObject* name) {
    PyObject* v = PyObject_GetAttr(obj, name);
    if (!v) return -1;
    const long long r = PyLong_AsLongLong(v);
    if (r == -1 && PyErr_Occurred() && PyErr_ExceptionMatches(PyExc_TypeError)) {      /* numpy integers and the like */
        PyErr_Clear();
        PyObject* w = PyNumber_Long(v);
        Py_DECREF(v);
        if (!w) return -1;
        const long long q = PyLong_AsLongLong(w);
        Py_DECREF(w);
        return q;
    }
    Py_DECREF(v);
    return r;
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
        long long v[3];
        for (int k = 0; k < 3; ++k) {
            PyObject* x = PyNumber_Index(PySequence_Fast_GET_ITEM(t, k));
            v[k] = x ? PyLong_AsLongLong(x) : -1;
            Py_XDECREF(x);
        }
        Py_DECREF(t);
        if (PyErr_Occurred()) return -1;
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

static PyObject* m_grammar(PyObject* self, PyObject* g) {
    (void)self;
    PyObject *vars = NULL, *prods = NULL, *ret = NULL, *tmp;
    Owner* o = NULL;
    tmp = PyObject_GetAttr(g, s_variables);
    if (!tmp) return NULL;
    vars = PySequence_Fast(tmp, "variables is a list");
    Py_DECREF(tmp);
    tmp = vars ? PyObject_GetAttr(g, s_productions) : NULL;
    if (!tmp) goto done;
    prods = PySequence_Fast(tmp, "productions is a list");
    Py_DECREF(tmp);
    if (!prods) goto done;
    const Py_ssize_t nv = PySequence_Fast_GET_SIZE(vars), np = PySequence_Fast_GET_SIZE(prods);
    o = new_owner(sizeof(xp_grammar_desc) + sizeof(xp_variable) * (size_t)nv + sizeof(xp_production) * (size_t)np);
    if (!o) goto done;
    xp_grammar_desc* d = (xp_grammar_desc*)o->mem;
    xp_production* p = (xp_production*)(d + 1);
    xp_variable* v = (xp_variable*)(p + np);
    d->n_vars = (int32_t)nv;
    d->vars = v;
    d->n_nonterminals = (int32_t)int_attr(g, s_n_nonterminals);
    d->n_productions = (int32_t)np;
    d->productions = p;
    for (Py_ssize_t i = 0; i < nv; ++i) {
        PyObject* x = PySequence_Fast_GET_ITEM(vars, i);
        PyObject* name = PyObject_GetAttr(x, s_name);
        PyObject* utf = name ? PyUnicode_AsUTF8String(name) : NULL;
        Py_XDECREF(name);
        if (!utf || PyList_Append(o->held, utf) < 0) { Py_XDECREF(utf); goto done; }
        v[i].name = PyBytes_AS_STRING(utf);
        Py_DECREF(utf);                                  /* (the list holds it) */
        v[i].lo = int_attr(x, s_lo);
        v[i].hi = int_attr(x, s_hi);
    }
    for (Py_ssize_t i = 0; i < np; ++i) {
        PyObject* x = PySequence_Fast_GET_ITEM(prods, i);
        const int32_t kind = (int32_t)int_attr(x, s_kind);
        p[i].kind = kind;
        p[i].lhs = (int32_t)int_attr(x, s_lhs);
        if (kind == XP_PROD_CONST) { p[i].value = int_attr(x, s_value); continue; }      /* (each kind reads its own fields) */
        if (kind == XP_PROD_VAR) { p[i].var = (int32_t)int_attr(x, s_var); continue; }
        p[i].op = (int32_t)int_attr(x, s_op);
        p[i].left = (int32_t)int_attr(x, s_left);
        p[i].right = (int32_t)int_attr(x, s_right);
    }
    if (PyErr_Occurred()) goto done;
    ret = Py_BuildValue("(KO)", (unsigned long long)(size_t)o->mem, (PyObject*)o);
done:
    Py_XDECREF((PyObject*)o);
    Py_XDECREF(vars);
    Py_XDECREF(prods);
    return ret;
}

/* Address and row count of an array with `itemsize`-byte integers; *held receives the object that has to stay alive.
 * A host array goes by the buffer protocol (conv(array, itemsize) first when it is not contiguous or of another type);
 * anything else is a torch tensor. */
static int array_at(PyObject* a, Py_ssize_t itemsize, PyObject* conv, const void** ptr, int32_t* on_device, long long* rows, PyObject** held) {
    Py_buffer b;
    *on_device = 0;
    if (PyObject_CheckBuffer(a)) {
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

static PyObject* get_list(PyObject* obj, PyObject* name) {       /* obj.name as a fast sequence (None: empty) */
    PyObject* v = PyObject_GetAttr(obj, name);
    if (!v) return NULL;
    if (v == Py_None) {
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
        PyObject* holes = get_list(PySequence_Fast_GET_ITEM(seq, i), s_holes);
        if (!holes) goto done;
        const Py_ssize_t nh = PySequence_Fast_GET_SIZE(holes);
        n_holes += (size_t)nh;
        for (Py_ssize_t h = 0; h < nh; ++h)
            for (int k = 0; k < 2; ++k) {
                PyObject* c = get_list(PySequence_Fast_GET_ITEM(holes, h), k ? s_spec_expr : s_ctx);
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
        PyObject* holes = get_list(sk, s_holes);
        if (!holes) goto done;
        const Py_ssize_t nh = PySequence_Fast_GET_SIZE(holes);
        PyList_SET_ITEM(nhs, i, PyLong_FromSsize_t(nh));
        d->n_holes = (int32_t)nh;
        d->holes = hd;
        int bad = 0;
        for (Py_ssize_t h = 0; h < nh && !bad; ++h, ++hd) {
            PyObject* ho = PySequence_Fast_GET_ITEM(holes, h);
            hd->start_nt = (int32_t)int_attr(ho, s_start_nt);
            hd->max_size = (int32_t)int_attr(ho, s_max_size);
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
                PyObject* c = get_list(ho, k ? s_spec_expr : s_ctx);
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

static PyObject* m_hole_result(PyObject* self, PyObject* arg) {
    (void)self;
    const xp_result_view* v = (const xp_result_view*)(size_t)PyLong_AsUnsignedLongLong(arg);
    if (!v) return NULL;
    const Py_ssize_t K = v->max_size + 1;
    PyObject *cand = PyList_New(K), *match = PyList_New(K), *code = PyList_New(v->least_len);
    if (!cand || !match || !code) {
        Py_XDECREF(cand);
        Py_XDECREF(match);
        Py_XDECREF(code);
        return NULL;
    }
    for (Py_ssize_t k = 0; k < K; ++k) {
        PyList_SET_ITEM(cand, k, PyLong_FromUnsignedLongLong(v->cand_count[k]));
        PyList_SET_ITEM(match, k, PyLong_FromUnsignedLongLong(v->match_count[k]));
    }
    for (Py_ssize_t k = 0; k < v->least_len; ++k)
        PyList_SET_ITEM(code, k, Py_BuildValue("(iiL)", (int)v->least_code[k].kind, (int)v->least_code[k].arg, (long long)v->least_code[k].value));
    return Py_BuildValue("(NNNiKsNKKKKddiKKKK)", PyBool_FromLong(v->solved), cand, match, (int)v->least_size, (unsigned long long)v->least_rank,
                         v->solved ? v->least_text : "", code, (unsigned long long)v->evals_executed, (unsigned long long)v->filter_survivors,
                         (unsigned long long)v->probe_survivors, (unsigned long long)v->nominal_ops, v->kernel_ms, v->total_ms, (int)v->n_launches,
                         (unsigned long long)v->filter_tests, (unsigned long long)v->candidates_skipped, (unsigned long long)v->h2d_bytes,
                         (unsigned long long)v->d2h_bytes);
}

static PyMethodDef methods[] = {
    {"grammar", m_grammar, METH_O, "Grammar model -> (descriptor address, owner)."},
    {"sketches", m_sketches, METH_VARARGS, "Sketch models -> (descriptors' address, owner, holes per sketch, device tensors per sketch)."},
    {"code", m_code, METH_O, "Postfix list -> xp_instr bytes."},
    {"hole_result", m_hole_result, METH_O, "Address of an xp_result_view -> tuple."},
    {NULL, NULL, 0, NULL},
};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", "Descriptors of include/xp.h from Python models.", -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void) {
    static const struct { PyObject** to; const char* name; } names[] = {
        {&s_variables, "variables"}, {&s_name, "name"}, {&s_lo, "lo"}, {&s_hi, "hi"}, {&s_n_nonterminals, "n_nonterminals"},
        {&s_productions, "productions"}, {&s_lhs, "lhs"}, {&s_kind, "kind"}, {&s_var, "var"}, {&s_op, "op"}, {&s_left, "left"},
        {&s_right, "right"}, {&s_value, "value"}, {&s_holes, "holes"}, {&s_coords, "coords"}, {&s_start_nt, "start_nt"},
        {&s_max_size, "max_size"}, {&s_ctx, "ctx"}, {&s_spec_expr, "spec_expr"}, {&s_spec_table, "spec_table"},
        {&s_data_ptr, "data_ptr"}, {&s_is_cuda, "is_cuda"}, {&s_shape, "shape"}};
    for (size_t i = 0; i < sizeof(names) / sizeof(names[0]); ++i) {
        *names[i].to = PyUnicode_InternFromString(names[i].name);
        if (!*names[i].to) return NULL;
    }
    if (PyType_Ready(&OwnerType) < 0) return NULL;
    return PyModule_Create(&module);
}
