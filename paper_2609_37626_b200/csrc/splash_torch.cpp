// Python entry points of the library: torch tensors in, one C ABI call, torch tensors out.
//
// The argument marshalling of a decode call is on the critical path of every small one: reading a dozen tensors' sizes,
// strides and pointers through Python attributes, two torch.empty and a ctypes call cost 20 us of host time, more than the
// GPU needs for a small batch.  Here the tensors are read in C++ and the outputs come straight from the CUDA caching
// allocator: about 2 us beside the launches themselves.  The functions have the names, arguments, defaults, results and
// assertions of the Python ones that they replaced; binding.py exports them.
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <map>
#include <string>
#include <utility>

#include "../../include/splash_mla.h"

namespace {

constexpr int64_t kDQK = 576, kDV = 512;

PyObject *g_error_class = nullptr;      // binding.SplashError

// ---- arguments -------------------------------------------------------------------------------------------------------

// Names of a function's arguments; the first `positional` may be given by position, the first `required` (and those the
// function checks itself) must be given.
struct Signature {
    const char *name;
    int positional, required, total;
    const char *const *names;
    PyObject **interned;
};

void intern(Signature &s) {
    s.interned = new PyObject *[s.total];
    for (int k = 0; k < s.total; ++k) s.interned[k] = PyUnicode_InternFromString(s.names[k]);
}

// Borrowed references into v (NULL where an argument was not given); None is kept as given.
bool parse(const Signature &s, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames, PyObject **v) {
    for (int k = 0; k < s.total; ++k) v[k] = nullptr;
    if (nargs > s.positional) {
        PyErr_Format(PyExc_TypeError, "%s() takes %d positional arguments but %zd were given", s.name, s.positional, nargs);
        return false;
    }
    for (Py_ssize_t k = 0; k < nargs; ++k) v[k] = args[k];
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t j = 0; j < nkw; ++j) {
        PyObject *name = PyTuple_GET_ITEM(kwnames, j);
        int k = 0;
        while (k < s.total && s.interned[k] != name) ++k;
        if (k == s.total)
            for (k = 0; k < s.total; ++k)
                if (PyUnicode_Compare(s.interned[k], name) == 0) break;
        if (k == s.total) { PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", s.name, name); return false; }
        if (v[k]) { PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%U'", s.name, name); return false; }
        v[k] = args[nargs + j];
    }
    for (int k = 0; k < s.required; ++k)
        if (!v[k]) { PyErr_Format(PyExc_TypeError, "%s() missing required argument '%s'", s.name, s.names[k]); return false; }
    return true;
}

bool given(PyObject *o) { return o != nullptr && o != Py_None; }

// The argument's tensor, or NULL with an exception set.
const at::Tensor *tensor(PyObject *o, const char *name) {
    if (!THPVariable_Check(o)) { PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor, not %.100s", name, Py_TYPE(o)->tp_name); return nullptr; }
    return &THPVariable_Unpack(o);
}

// Optional tensor: false with an exception set when it is something else.
bool maybe_tensor(PyObject *o, const char *name, const at::Tensor *&t) {
    t = nullptr;
    if (!given(o)) return true;
    t = tensor(o, name);
    return t != nullptr;
}

bool integer(PyObject *o, int64_t if_absent, int64_t &value) {
    if (!given(o)) { value = if_absent; return true; }
    value = PyLong_AsLongLong(o);
    return !(value == -1 && PyErr_Occurred());
}

bool stream_of(PyObject *o, void *&stream) {
    if (!given(o)) { stream = c10::cuda::getCurrentCUDAStream().stream(); return true; }
    PyObject *p = PyObject_GetAttrString(o, "cuda_stream");
    if (!p) return false;
    stream = PyLong_AsVoidPtr(p);
    Py_DECREF(p);
    return !PyErr_Occurred();
}

#define SPLASH_ASSERT(cond)                                                      \
    do {                                                                         \
        if (!(cond)) { PyErr_SetString(PyExc_AssertionError, #cond); return nullptr; } \
    } while (0)

PyObject *raise_status(int rc) {
    std::string msg = std::string(splash_status_string(rc)) + ": " + splash_last_error();
    PyObject *err = g_error_class ? PyObject_CallFunction(g_error_class, "is", rc, msg.c_str()) : nullptr;
    if (err) { PyErr_SetObject(g_error_class, err); Py_DECREF(err); }
    else if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, msg.c_str());
    return nullptr;
}

void *ptr(const at::Tensor *t) { return t ? t->data_ptr() : nullptr; }

// A call into the library without the GIL: with the stream's launch queue full a launch blocks until the GPU has caught up, which may
// itself wait for this process's other threads.  (Given back on every way out; addresses are read from the tensors before, where an
// exception finds the GIL held.)
template <typename F>
int without_gil(F &&call) {
    struct Released {
        PyThreadState *state = PyEval_SaveThread();
        ~Released() { PyEval_RestoreThread(state); }
    } released;
    return call();
}

at::Tensor new_tensor(at::IntArrayRef size, at::ScalarType dtype, const at::Tensor &like) {
    return at::Tensor(at::detail::empty_cuda(size, dtype, like.device(), std::nullopt));
}

// The scratch buffer of calls that bring none: one per device and purpose, as large as the largest call so far.  (Never
// destroyed: the allocator may be gone when static objects are.)  Guarded by the GIL.
std::map<std::pair<int, std::string>, at::Tensor> &workspaces() {
    static auto *m = new std::map<std::pair<int, std::string>, at::Tensor>();
    return *m;
}

at::Tensor &cached_workspace(const at::Tensor &like, size_t nbytes, const char *tag) {
    at::Tensor &ws = workspaces()[{like.device().index(), tag}];
    if (!ws.defined() || (size_t)ws.numel() < nbytes)
        ws = new_tensor({(int64_t)(nbytes > 256 ? nbytes : 256)}, at::kByte, like);
    return ws;
}

PyObject *pair_of(PyObject *a, const at::Tensor &ta, PyObject *b, const at::Tensor &tb) {
    // the caller's own objects come back when it gave them
    PyObject *pa = given(a) ? Py_NewRef(a) : THPVariable_Wrap(ta);
    PyObject *pb = given(b) ? Py_NewRef(b) : THPVariable_Wrap(tb);
    PyObject *t = pa && pb ? PyTuple_Pack(2, pa, pb) : nullptr;
    Py_XDECREF(pa);
    Py_XDECREF(pb);
    return t;
}

// Fills the shape of a decode call; false with an AssertionError set when the tensors do not fit together.
bool fill_shape(splash_mla_shape &s, const at::Tensor &q, const at::Tensor &kv, const at::Tensor &table, const at::Tensor &out,
                const at::Tensor &lse, double scale, int64_t flags) {
    auto fail = [](const char *what) { PyErr_SetString(PyExc_AssertionError, what); return false; };
    s = splash_mla_shape{};
    s.struct_size = sizeof s;
    const bool rows = q.dim() == 4;
    if (rows) {
        const int64_t R = q.size(2);
        if (q.stride(3) != 1 || q.stride(2) != q.size(3) || out.dim() != 4 || out.stride(3) != 1) return fail("q / out rows must be dense");
        if (out.stride(2) != out.size(3) || lse.dim() != 3 || lse.stride(2) != 1 || lse.stride(1) != R) return fail("out / lse rows must be dense");
        s.q_rows = (uint32_t)R;
    } else {
        if (q.dim() != 3) { PyErr_SetString(PyExc_ValueError, "q must have 3 or 4 dimensions"); return false; }
        if (q.stride(2) != 1 || out.stride(2) != 1 || lse.stride(1) != 1) return fail("q, out and lse must be dense in their last dimension");
    }
    s.num_requests = (int32_t)q.size(0);
    s.num_heads = (int32_t)q.size(1);
    s.d_qk = (int32_t)q.size(-1);
    s.d_v = (int32_t)out.size(-1);
    s.page_size = (int32_t)kv.size(1);
    s.num_pool_pages = (int32_t)kv.size(0);
    s.block_table_stride = table.dim() == 2 && s.num_requests > 0 ? (int32_t)table.stride(0) : 0;
    s.kv_dtype = kv.scalar_type() == at::kBFloat16 ? SPLASH_KV_BF16
                 : kv.size(-1) == SPLASH_SPARSE_ROW_BYTES ? SPLASH_KV_E4M3_BLOCK_SCALE_BF16_ROPE : SPLASH_KV_E4M3_TOKEN_SCALE;
    s.softmax_scale = (float)scale;
    s.q_stride_request = q.stride(0);
    s.q_stride_head = q.stride(1);
    s.out_stride_request = out.stride(0);
    s.out_stride_head = out.stride(1);
    s.lse_stride_request = lse.stride(0);
    s.flags = (uint32_t)flags;
    return true;
}

// ---- decode ----------------------------------------------------------------------------------------------------------

const char *const kDecodeNames[] = {"q", "kv_pool", "block_table", "seq_lens", "softmax_scale", "kv_scales", "head_begin", "head_end",
                                    "kv_begin", "kv_end", "out", "lse", "workspace", "stream", "flags", "migrate_job"};
Signature sig_decode{"splash_mla_decode", 4, 5, 16, kDecodeNames, nullptr};

PyObject *mla_decode(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    PyObject *v[16];
    if (!parse(sig_decode, args, nargs, kwnames, v)) return nullptr;
    const at::Tensor *q, *kv, *table, *lens, *scales, *begin, *end, *ws;
    if (!(q = tensor(v[0], "q")) || !(kv = tensor(v[1], "kv_pool")) || !(table = tensor(v[2], "block_table")) || !(lens = tensor(v[3], "seq_lens")))
        return nullptr;
    const double scale = PyFloat_AsDouble(v[4]);
    if (scale == -1.0 && PyErr_Occurred()) return nullptr;
    if (!maybe_tensor(v[5], "kv_scales", scales) || !maybe_tensor(v[8], "kv_begin", begin) || !maybe_tensor(v[9], "kv_end", end) ||
        !maybe_tensor(v[12], "workspace", ws))
        return nullptr;
    SPLASH_ASSERT(q->is_cuda() && q->scalar_type() == at::kBFloat16);
    int64_t first, last, flags;
    if (!integer(v[6], 0, first) || !integer(v[7], q->size(1), last) || !integer(v[14], 0, flags)) return nullptr;
    at::Tensor out, lse;
    const int64_t B = q->size(0), H = q->size(1);
    if (given(v[10])) { const at::Tensor *t = tensor(v[10], "out"); if (!t) return nullptr; out = *t; }
    else if (q->dim() == 4) out = new_tensor({B, H, q->size(2), kDV}, at::kFloat, *q);
    else out = new_tensor({B, H, kDV}, at::kFloat, *q);
    if (given(v[11])) { const at::Tensor *t = tensor(v[11], "lse"); if (!t) return nullptr; lse = *t; }
    else if (q->dim() == 4) lse = new_tensor({B, H, q->size(2)}, at::kFloat, *q);
    else lse = new_tensor({B, H}, at::kFloat, *q);
    SPLASH_ASSERT(table->scalar_type() == at::kInt && lens->scalar_type() == at::kInt);
    splash_mla_shape shape;
    if (!fill_shape(shape, *q, *kv, *table, out, lse, scale, flags)) return nullptr;
    void *stream;
    if (!stream_of(v[13], stream)) return nullptr;
    if (!ws) ws = &cached_workspace(*q, splash_mla_decode_workspace_bytes(&shape, (int32_t)first, (int32_t)last), "decode");
    const at::Tensor keep = *ws;                    // another thread may replace the cached one while the GIL is released
    const size_t ws_bytes = (size_t)keep.numel() * keep.element_size();
    const void *q_at = q->data_ptr(), *kv_at = kv->data_ptr(), *scales_at = ptr(scales), *table_at = table->data_ptr(), *lens_at = lens->data_ptr();
    const void *begin_at = ptr(begin), *end_at = ptr(end);
    void *out_at = out.data_ptr(), *lse_at = lse.data_ptr(), *ws_at = keep.data_ptr();
    auto decode = [&](const splash_migrate_job *job) {
        return without_gil([&] {
            return splash_mla_decode_migrating(&shape, q_at, kv_at, (const float *)scales_at, (const int32_t *)table_at, (const int32_t *)lens_at,
                                               (int32_t)first, (int32_t)last, (const int32_t *)begin_at, (const int32_t *)end_at, (float *)out_at,
                                               (float *)lse_at, ws_at, ws_bytes, stream, job);
        });
    };
    int rc;
    if (given(v[15])) {                             // (splash_migrate_job as a ctypes structure, what keeps it alive)
        PyObject *job = PySequence_GetItem(v[15], 0);
        Py_buffer view;
        if (!job) return nullptr;
        if (PyObject_GetBuffer(job, &view, PyBUF_SIMPLE) != 0) { Py_DECREF(job); return nullptr; }
        rc = (size_t)view.len == sizeof(splash_migrate_job) ? decode((const splash_migrate_job *)view.buf) : SPLASH_INVALID_ARG;
        PyBuffer_Release(&view);
        Py_DECREF(job);
    } else {
        rc = decode(nullptr);
    }
    if (rc != SPLASH_OK) return raise_status(rc);
    return pair_of(v[10], out, v[11], lse);
    END_HANDLE_TH_ERRORS
}

const char *const kSparseNames[] = {"q", "kv_pool", "block_table", "seq_lens", "sel_tokens", "sel_count", "softmax_scale", "max_selected",
                                    "head_begin", "head_end", "out", "lse", "workspace", "stream", "flags"};
Signature sig_sparse{"splash_mla_decode_sparse", 6, 7, 15, kSparseNames, nullptr};

PyObject *mla_decode_sparse(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    PyObject *v[15];
    if (!parse(sig_sparse, args, nargs, kwnames, v)) return nullptr;
    const at::Tensor *q, *kv, *table, *lens, *sel, *count, *ws;
    if (!(q = tensor(v[0], "q")) || !(kv = tensor(v[1], "kv_pool")) || !(table = tensor(v[2], "block_table")) || !(lens = tensor(v[3], "seq_lens")) ||
        !(sel = tensor(v[4], "sel_tokens")) || !(count = tensor(v[5], "sel_count")) || !maybe_tensor(v[12], "workspace", ws))
        return nullptr;
    const double scale = PyFloat_AsDouble(v[6]);
    if (scale == -1.0 && PyErr_Occurred()) return nullptr;
    SPLASH_ASSERT(q->is_cuda() && q->scalar_type() == at::kBFloat16 && q->dim() == 3);
    SPLASH_ASSERT(kv->scalar_type() == at::kByte && kv->size(-1) == SPLASH_SPARSE_ROW_BYTES && kv->is_contiguous());
    SPLASH_ASSERT(sel->scalar_type() == at::kInt && count->scalar_type() == at::kInt && sel->dim() == 2);
    SPLASH_ASSERT(sel->numel() == 0 || sel->stride(1) == 1);
    SPLASH_ASSERT(table->scalar_type() == at::kInt && lens->scalar_type() == at::kInt);
    int64_t most, first, last, flags;
    if (!integer(v[7], sel->size(1), most) || !integer(v[8], 0, first) || !integer(v[9], q->size(1), last) || !integer(v[14], 0, flags)) return nullptr;
    at::Tensor out, lse;
    if (given(v[10])) { const at::Tensor *t = tensor(v[10], "out"); if (!t) return nullptr; out = *t; }
    else out = new_tensor({q->size(0), q->size(1), kDV}, at::kFloat, *q);
    if (given(v[11])) { const at::Tensor *t = tensor(v[11], "lse"); if (!t) return nullptr; lse = *t; }
    else lse = new_tensor({q->size(0), q->size(1)}, at::kFloat, *q);
    splash_mla_shape shape;
    if (!fill_shape(shape, *q, *kv, *table, out, lse, scale, flags)) return nullptr;
    void *stream;
    if (!stream_of(v[13], stream)) return nullptr;
    if (!ws) {
        const size_t need = splash_mla_decode_sparse_workspace_bytes(&shape, (int32_t)most, (int32_t)first, (int32_t)last);
        if (need == 0) return raise_status(SPLASH_INVALID_ARG);
        ws = &cached_workspace(*q, need, "decode");
    }
    const at::Tensor keep = *ws;
    const void *q_at = q->data_ptr(), *kv_at = kv->data_ptr(), *table_at = table->data_ptr(), *lens_at = lens->data_ptr(), *sel_at = sel->data_ptr();
    const void *count_at = count->data_ptr();
    void *out_at = out.data_ptr(), *lse_at = lse.data_ptr(), *ws_at = keep.data_ptr();
    const int64_t sel_stride = q->size(0) > 0 ? sel->stride(0) : 0;
    const size_t ws_bytes = (size_t)keep.numel() * keep.element_size();
    const int rc = without_gil([&] {
        return splash_mla_decode_sparse(&shape, q_at, kv_at, (const int32_t *)table_at, (const int32_t *)lens_at, (const int32_t *)sel_at, sel_stride,
                                        (const int32_t *)count_at, (int32_t)most, (int32_t)first, (int32_t)last, (float *)out_at, (float *)lse_at,
                                        ws_at, ws_bytes, stream);
    });
    if (rc != SPLASH_OK) return raise_status(rc);
    return pair_of(v[10], out, v[11], lse);
    END_HANDLE_TH_ERRORS
}

const char *const kMergeNames[] = {"part_out", "part_lse", "out", "lse", "stream"};
Signature sig_merge{"splash_lse_merge", 5, 2, 5, kMergeNames, nullptr};

PyObject *lse_merge(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    PyObject *v[5];
    if (!parse(sig_merge, args, nargs, kwnames, v)) return nullptr;
    const at::Tensor *po, *pl;
    if (!(po = tensor(v[0], "part_out")) || !(pl = tensor(v[1], "part_lse"))) return nullptr;
    SPLASH_ASSERT(po->is_contiguous() && pl->is_contiguous());
    if (po->dim() != 3) { PyErr_SetString(PyExc_ValueError, "part_out must be [parts][rows][d_v]"); return nullptr; }
    const int64_t parts = po->size(0), rows = po->size(1), dv = po->size(2);
    at::Tensor out, lse;
    if (given(v[2])) { const at::Tensor *t = tensor(v[2], "out"); if (!t) return nullptr; out = *t; }
    else out = new_tensor({rows, dv}, at::kFloat, *po);
    if (given(v[3])) { const at::Tensor *t = tensor(v[3], "lse"); if (!t) return nullptr; lse = *t; }
    else lse = new_tensor({rows}, at::kFloat, *po);
    void *stream;
    if (!stream_of(v[4], stream)) return nullptr;
    const void *po_at = po->data_ptr(), *pl_at = pl->data_ptr();
    void *out_at = out.data_ptr(), *lse_at = lse.data_ptr();
    const int rc = without_gil([&] {
        return splash_lse_merge((int32_t)parts, rows, (int32_t)dv, (const float *)po_at, (const float *)pl_at, (float *)out_at, (float *)lse_at, stream);
    });
    if (rc != SPLASH_OK) return raise_status(rc);
    return pair_of(v[2], out, v[3], lse);
    END_HANDLE_TH_ERRORS
}

// ---- page migration ---------------------------------------------------------------------------------------------------

const char *const kMigrateNames[] = {"src_pool", "dst_pool", "src_page_ids", "dst_page_ids", "block_table", "src_scales", "dst_scales",
                                     "src_id_base", "dst_id_base", "max_page_id", "workspace", "stream"};
Signature sig_migrate{"splash_kv_page_migrate", 5, 5, 12, kMigrateNames, nullptr};
const char *const kMigrateStaticNames[] = {"src_pool", "dst_pool", "src_page_ids", "dst_page_ids", "block_table", "src_scales", "dst_scales",
                                           "src_id_base", "dst_id_base", "max_page_id", "stream"};
Signature sig_migrate_static{"splash_kv_page_migrate_static", 5, 5, 11, kMigrateStaticNames, nullptr};

PyObject *migrate(PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames, bool with_workspace) {
    PyObject *v[12];
    if (!parse(with_workspace ? sig_migrate : sig_migrate_static, args, nargs, kwnames, v)) return nullptr;
    const at::Tensor *src, *dst, *sid, *did, *table, *ss, *ds, *ws = nullptr;
    if (!(src = tensor(v[0], "src_pool")) || !(dst = tensor(v[1], "dst_pool")) || !(sid = tensor(v[2], "src_page_ids")) ||
        !(did = tensor(v[3], "dst_page_ids")) || !(table = tensor(v[4], "block_table")) || !maybe_tensor(v[5], "src_scales", ss) ||
        !maybe_tensor(v[6], "dst_scales", ds) || (with_workspace && !maybe_tensor(v[10], "workspace", ws)))
        return nullptr;
    SPLASH_ASSERT(src->is_contiguous() && dst->is_contiguous() && table->is_contiguous());
    SPLASH_ASSERT(sid->scalar_type() == at::kInt && did->scalar_type() == at::kInt);
    int64_t src_base, dst_base, most;
    if (!integer(v[7], 0, src_base) || !integer(v[8], 0, dst_base)) return nullptr;
    if (!integer(v[9], std::max(src_base + src->size(0), dst_base + dst->size(0)), most)) return nullptr;
    void *stream;
    if (!stream_of(v[with_workspace ? 11 : 10], stream)) return nullptr;
    const int64_t page_bytes = src->size(1) * src->size(2) * src->element_size();
    if (with_workspace && !ws) ws = &cached_workspace(*src, splash_kv_page_migrate_workspace_bytes((int32_t)most), "migrate");
    const at::Tensor keep = with_workspace ? *ws : at::Tensor();
    const void *src_at = src->data_ptr(), *ss_at = ptr(ss), *sid_at = sid->data_ptr(), *did_at = did->data_ptr();
    void *dst_at = dst->data_ptr(), *ds_at = ptr(ds), *table_at = table->data_ptr(), *ws_at = with_workspace ? keep.data_ptr() : nullptr;
    const int64_t n = sid->numel(), entries = table->numel();
    const size_t ws_bytes = with_workspace ? (size_t)keep.numel() : 0;
    const int rc = without_gil([&] {
        return with_workspace
                   ? splash_kv_page_migrate(src_at, (const float *)ss_at, dst_at, (float *)ds_at, page_bytes, (const int32_t *)sid_at,
                                            (const int32_t *)did_at, n, (int32_t)src_base, (int32_t)dst_base, (int32_t)most, (int32_t *)table_at,
                                            entries, ws_at, ws_bytes, stream)
                   : splash_kv_page_migrate_static(src_at, (const float *)ss_at, dst_at, (float *)ds_at, page_bytes, (const int32_t *)sid_at,
                                                   (const int32_t *)did_at, n, (int32_t)src_base, (int32_t)dst_base, (int32_t)most,
                                                   (int32_t *)table_at, entries, stream);
    });
    if (rc != SPLASH_OK) return raise_status(rc);
    Py_RETURN_NONE;
}

PyObject *kv_page_migrate(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    return migrate(args, nargs, kwnames, true);
    END_HANDLE_TH_ERRORS
}

PyObject *kv_page_migrate_static(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    return migrate(args, nargs, kwnames, false);
    END_HANDLE_TH_ERRORS
}

// ---- DOP layout changes -----------------------------------------------------------------------------------------------

const char *const kPackNames[] = {"a", "b", "send_row", "out", "stream"};
Signature sig_pack{"splash_dop_pack_rows", 5, 3, 5, kPackNames, nullptr};

PyObject *dop_pack_rows(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    PyObject *v[5];
    if (!parse(sig_pack, args, nargs, kwnames, v)) return nullptr;
    const at::Tensor *a, *b, *row;
    if (!(a = tensor(v[0], "a")) || !maybe_tensor(v[1], "b", b) || !(row = tensor(v[2], "send_row"))) return nullptr;
    SPLASH_ASSERT(a->dim() == 3 && (a->numel() == 0 || a->stride(2) == 1) && row->scalar_type() == at::kInt);
    SPLASH_ASSERT(row->numel() == 0 || row->is_contiguous());
    const int64_t es = a->element_size(), n = row->numel(), h = a->size(1), da = a->size(2);
    int64_t db = 0;
    if (b) {
        SPLASH_ASSERT(b->dim() == 3 && (b->numel() == 0 || b->stride(2) == 1) && b->scalar_type() == a->scalar_type());
        SPLASH_ASSERT(b->size(0) == a->size(0) && b->size(1) == a->size(1));
        db = b->size(2);
    }
    at::Tensor out;
    if (given(v[3])) { const at::Tensor *t = tensor(v[3], "out"); if (!t) return nullptr; out = *t; }
    else out = new_tensor({n, h, da + db}, a->scalar_type(), *a);
    SPLASH_ASSERT(out.is_contiguous() && out.sizes() == at::IntArrayRef({n, h, da + db}));
    void *stream;
    if (!stream_of(v[4], stream)) return nullptr;
    const void *a_at = a->data_ptr(), *b_at = ptr(b), *row_at = row->data_ptr();
    void *out_at = out.data_ptr();
    const int64_t a_row = a->stride(0) * es, a_head = a->stride(1) * es, b_row = b ? b->stride(0) * es : 0, b_head = b ? b->stride(1) * es : 0;
    const int rc = without_gil([&] {
        return splash_dop_pack_rows(a_at, da * es, a_row, a_head, b_at, db * es, b_row, b_head, (const int32_t *)row_at, n, (int32_t)h, out_at, stream);
    });
    if (rc != SPLASH_OK) return raise_status(rc);
    return given(v[3]) ? Py_NewRef(v[3]) : THPVariable_Wrap(out);
    END_HANDLE_TH_ERRORS
}

const char *const kSwapNames[] = {"x", "out", "stream"};
Signature sig_swap{"splash_dop_swap_outer", 3, 1, 3, kSwapNames, nullptr};

PyObject *dop_swap_outer(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    PyObject *v[3];
    if (!parse(sig_swap, args, nargs, kwnames, v)) return nullptr;
    const at::Tensor *x = tensor(v[0], "x");
    if (!x) return nullptr;
    SPLASH_ASSERT(x->is_contiguous() && x->dim() >= 2);
    int64_t inner = x->element_size();
    for (int64_t k = 2; k < x->dim(); ++k) inner *= x->size(k);
    at::Tensor out;
    if (given(v[1])) {
        const at::Tensor *t = tensor(v[1], "out");
        if (!t) return nullptr;
        out = *t;
    } else {
        at::DimVector size(x->sizes().begin(), x->sizes().end());
        std::swap(size[0], size[1]);
        out = new_tensor(size, x->scalar_type(), *x);
    }
    SPLASH_ASSERT(out.is_contiguous());
    void *stream;
    if (!stream_of(v[2], stream)) return nullptr;
    const void *x_at = x->data_ptr();
    void *out_at = out.data_ptr();
    const int64_t A = x->size(0), Bn = x->size(1);
    const int rc = without_gil([&] { return splash_dop_swap_outer(x_at, A, Bn, inner, out_at, stream); });
    if (rc != SPLASH_OK) return raise_status(rc);
    return given(v[1]) ? Py_NewRef(v[1]) : THPVariable_Wrap(out);
    END_HANDLE_TH_ERRORS
}

const char *const kUnpackNames[] = {"recv", "send_row", "out", "stream"};
Signature sig_unpack{"splash_dop_unpack_rows", 4, 3, 4, kUnpackNames, nullptr};

PyObject *dop_unpack_rows(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    HANDLE_TH_ERRORS
    PyObject *v[4];
    if (!parse(sig_unpack, args, nargs, kwnames, v)) return nullptr;
    const at::Tensor *recv, *row, *out;
    if (!(recv = tensor(v[0], "recv")) || !(row = tensor(v[1], "send_row")) || !(out = tensor(v[2], "out"))) return nullptr;
    SPLASH_ASSERT(recv->is_contiguous() && row->scalar_type() == at::kInt && row->is_contiguous());
    if (out->size(0) > 0) {
        auto of_a_row = [](const at::Tensor &t) { return t.dim() > 0 ? t.sizes().slice(1) : at::IntArrayRef(); };
        SPLASH_ASSERT(of_a_row(*recv) == of_a_row(*out));
        int64_t dense = 1;                          // every row of out is dense (the rows themselves may lie apart, and one without elements is)
        for (int64_t k = out->dim() - 1; k >= 1 && out->numel() > 0; --k) {
            SPLASH_ASSERT(out->size(k) == 1 || out->stride(k) == dense);
            dense *= out->size(k);
        }
    }
    int64_t row_bytes = recv->element_size();
    for (int64_t k = 1; k < recv->dim(); ++k) row_bytes *= recv->size(k);
    void *stream;
    if (!stream_of(v[3], stream)) return nullptr;
    const void *recv_at = recv->data_ptr(), *row_at = row->data_ptr();
    void *out_at = out->data_ptr();
    const int64_t n = row->numel(), pitch = out->stride(0) * out->element_size();
    const int rc = without_gil([&] { return splash_dop_unpack_rows(recv_at, (const int32_t *)row_at, n, row_bytes, out_at, pitch, stream); });
    if (rc != SPLASH_OK) return raise_status(rc);
    return Py_NewRef(v[2]);
    END_HANDLE_TH_ERRORS
}

// ---- module -----------------------------------------------------------------------------------------------------------

PyObject *set_error_class(PyObject *, PyObject *cls) {
    Py_XSETREF(g_error_class, Py_NewRef(cls));
    Py_RETURN_NONE;
}

PyObject *cached(PyObject *, PyObject *args) {
    int device;
    const char *tag;
    if (!PyArg_ParseTuple(args, "is", &device, &tag)) return nullptr;
    auto it = workspaces().find({device, tag});
    if (it == workspaces().end()) Py_RETURN_NONE;
    return THPVariable_Wrap(it->second);
}

#define FAST(f) ((PyCFunction)(void (*)(void))(f))
PyMethodDef kMethods[] = {
    {"splash_mla_decode", FAST(mla_decode), METH_FASTCALL | METH_KEYWORDS,
     "splash_mla_decode(q, kv_pool, block_table, seq_lens, *, softmax_scale, kv_scales=None, head_begin=0, head_end=None, "
     "kv_begin=None, kv_end=None, out=None, lse=None, workspace=None, stream=None, flags=0, migrate_job=None)\n--\n\n"
     "Decode attention of one shard; see splash_mla_decode in include/splash_mla.h.\n"
     "With migrate_job (from make_migrate_job) the call is splash_mla_decode_migrating: the job's pages\n"
     "move while this call decodes.\n\n"
     "q [B][H][576] bf16; kv_pool [P][64][576] bf16, or uint8 / float8_e4m3fn with\n"
     "kv_scales [P][64] fp32; block_table [B][stride] int32; seq_lens, kv_begin, kv_end\n"
     "[B] int32.  out [B][H][512] fp32 and lse [B][H] fp32 are allocated (uninitialised\n"
     "outside the head slice) unless given.  Returns (out, lse).\n"
     "A 4-D q [B][H][R][576] asks for R causal query rows per request (the request's R\n"
     "newest tokens); out is then [B][H][R][512] and lse [B][H][R].\n"},
    {"splash_mla_decode_sparse", FAST(mla_decode_sparse), METH_FASTCALL | METH_KEYWORDS,
     "splash_mla_decode_sparse(q, kv_pool, block_table, seq_lens, sel_tokens, sel_count, *, softmax_scale, max_selected=None, "
     "head_begin=0, head_end=None, out=None, lse=None, workspace=None, stream=None, flags=0)\n--\n\n"
     "Decode attention over a token list per request; see splash_mla_decode_sparse in include/splash_mla.h.\n\n"
     "q [B][H][576] bf16; kv_pool [P][64][656] uint8 (e4m3 latent, four block scales, bf16 rope per row);\n"
     "sel_tokens [B][K] int32 token positions, request i uses the first sel_count[i] (<= max_selected, default K).\n"
     "Returns (out [B][H][512] fp32, lse [B][H] fp32).\n"},
    {"splash_lse_merge", FAST(lse_merge), METH_FASTCALL | METH_KEYWORDS,
     "splash_lse_merge(part_out, part_lse, out=None, lse=None, stream=None)\n--\n\n"
     "Merge [parts][rows][d_v] fp32 partial outputs by their [parts][rows] LSE.\n"},
    {"splash_kv_page_migrate", FAST(kv_page_migrate), METH_FASTCALL | METH_KEYWORDS,
     "splash_kv_page_migrate(src_pool, dst_pool, src_page_ids, dst_page_ids, block_table, *, src_scales=None, dst_scales=None, "
     "src_id_base=0, dst_id_base=0, max_page_id=None, workspace=None, stream=None)\n--\n\n"
     "Copy listed pages pool -> pool and rewrite block_table in place.\n"},
    {"splash_kv_page_migrate_static", FAST(kv_page_migrate_static), METH_FASTCALL | METH_KEYWORDS,
     "splash_kv_page_migrate_static(src_pool, dst_pool, src_page_ids, dst_page_ids, block_table, *, src_scales=None, dst_scales=None, "
     "src_id_base=0, dst_id_base=0, max_page_id=None, stream=None)\n--\n\n"
     "Page migration for callers that cannot allocate device memory: same effect as\n"
     "splash_kv_page_migrate, but the remap table is the library's built-in 1 MiB device\n"
     "array, so this wrapper passes no workspace and creates no tensor.  Page ids must stay\n"
     "below 262,144; calls that could overlap on the GPU must be ordered by the caller.\n"},
    {"splash_dop_pack_rows", FAST(dop_pack_rows), METH_FASTCALL | METH_KEYWORDS,
     "splash_dop_pack_rows(a, b, send_row, out=None, stream=None)\n--\n\n"
     "Send buffer of the DOP forward exchange: out[p][j] = a[send_row[p]][j] ++ b[send_row[p]][j].\n\n"
     "a [N][h][da], b [N][h][db] or None (last dimension contiguous, any row / head strides), send_row [n] int32.\n"
     "Returns out [n][h][da+db] (dense).\n"},
    {"splash_dop_swap_outer", FAST(dop_swap_outer), METH_FASTCALL | METH_KEYWORDS,
     "splash_dop_swap_outer(x, out=None, stream=None)\n--\n\n"
     "[A][B][...] -> [B][A][...] (contiguous in, contiguous out).\n"},
    {"splash_dop_unpack_rows", FAST(dop_unpack_rows), METH_FASTCALL | METH_KEYWORDS,
     "splash_dop_unpack_rows(recv, send_row, out, stream=None)\n--\n\n"
     "out[send_row[p]] = recv[p]; recv [n][...] contiguous, out [N][...] with contiguous rows.\n"},
    {"set_error_class", set_error_class, METH_O, "The exception class of a call that did not succeed."},
    {"cached_workspace", cached, METH_VARARGS, "The scratch buffer that calls without one share on a device, or None."},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_splash_torch", "Native entry points of libsplash_mla.so for torch tensors.", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__splash_torch() {
    for (Signature *s : {&sig_decode, &sig_sparse, &sig_merge, &sig_migrate, &sig_migrate_static, &sig_pack, &sig_swap, &sig_unpack}) intern(*s);
    return PyModule_Create(&kModule);
}
