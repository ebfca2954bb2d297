// CPython module behind binding.py: the calls of the hot path from torch tensors to the C ABI.
//
// A small layer is three to six of these calls, each 4 to 20 us of kernels.  Marshalled in Python through
// ctypes a call cost 8 to 12 us of host time (attribute look-ups, allocations through the dispatcher, 13
// to 25 converted arguments), which is what bound every call below ~4000 tokens; here it is 1 to 2 us
// beside the launches.  Argument checks, results and errors are those binding.py documents.
//
// Arguments are read and results wrapped under the interpreter lock; allocations and the calls of the library run
// without it, so that a call that waits (a full launch queue, a kernel's first load, an allocation) stops no
// other Python thread.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <map>
#include <mutex>
#include <vector>

#include "usv.h"

namespace {

struct ValueErr { const char* what; };       // -> ValueError
struct PyErr {};                             // a Python error is already set
struct Status { int status; const char* where; };   // -> USVError

PyObject* g_raise = nullptr;                 // callable (status, where) that raises USVError

void check(int status, const char* where) {
    if (status != USV_OK) throw Status{status, where};
}
void need(bool ok, const char* what) {
    if (!ok) throw ValueErr{what};
}

bool is_none(PyObject* o) { return o == nullptr || o == Py_None; }

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor");
        throw PyErr();
    }
    return THPVariable_Unpack(o);
}
at::Tensor given(PyObject* o) { return is_none(o) ? at::Tensor() : tensor(o); }   // optional
int64_t integer(PyObject* o) {
    if (PyLong_Check(o)) {
        const long long v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) throw PyErr();
        return v;
    }
    PyObject* n = PyNumber_Long(o);          // what int() does
    if (n == nullptr) throw PyErr();
    const long long v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw PyErr();
    return v;
}
// whole numbers only (what an index takes): a grid of floats is refused
int64_t whole(PyObject* o) {
    if (PyLong_Check(o)) return integer(o);
    PyObject* n = PyNumber_Index(o);
    if (n == nullptr) throw PyErr();
    const long long v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw PyErr();
    return v;
}
// the number of merged sources; beside a given output, whose rows it is compared with, also a float of that value
int64_t merged_count(PyObject* o, bool with_out) {
    if (!with_out || !PyFloat_Check(o)) return whole(o);
    const int64_t v = integer(o);
    need((double)v == PyFloat_AS_DOUBLE(o), "out must be a contiguous bf16 [B,N-r,C] tensor");
    return v;
}
double real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PyErr();
    return v;
}
bool truth(PyObject* o) {
    const int t = PyObject_IsTrue(o);
    if (t < 0) throw PyErr();
    return t != 0;
}

void* ptr(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }
void* stream_of(const at::Tensor& t) { return c10::cuda::getCurrentCUDAStream(t.device().index()).stream(); }

at::Tensor fresh(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) {
    return at::detail::empty_cuda(sizes, type, like.device(), std::nullopt);
}

usv_strides view(const at::Tensor& t, const char* what) {
    need(t.dim() == 4 && t.scalar_type() == at::kBFloat16 && t.is_cuda() && t.stride(3) == 1, what);
    return usv_strides{t.stride(0), t.stride(1), t.stride(2)};
}
#define VIEW_TEXT(name) name " must be a CUDA bf16 [B,H,N,d] view with a contiguous last axis"

// Kept key blocks per head, as the C ABI takes them.
struct Kept {
    std::vector<int32_t> k;
    int most = 0;
    Kept(PyObject* o, int64_t H) {
        PyObject* seq = PySequence_Fast(o, "k_per_head must be a sequence");
        if (seq == nullptr) throw PyErr();
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
        k.resize(n);
        try {
            for (Py_ssize_t i = 0; i < n; ++i) k[i] = (int32_t)integer(PySequence_Fast_GET_ITEM(seq, i));
        } catch (...) {
            Py_DECREF(seq);
            throw;
        }
        Py_DECREF(seq);
        need(n == H && n > 0, "k_per_head needs one entry per head");
        most = k[0];
        for (int32_t v : k) most = v > most ? v : most;
    }
};

// Interpreter lock given up for the lifetime of the object.
struct NoGil {
    PyThreadState* state = PyEval_SaveThread();
    NoGil() = default;
    NoGil(const NoGil&) = delete;
    ~NoGil() { PyEval_RestoreThread(state); }
};

// Grow-only scratch buffer per (device, stream).  Its header (status word) starts at zero and is carried
// over when the buffer grows, so that workspace_status() sees every call.  A Scratch object holds the buffer for
// one call: calls of several threads on one stream put their kernels into it one call after the other.  (Only
// taken without the interpreter lock, which an allocation inside may ask for.)
struct Buffer {
    std::mutex lock;
    at::Tensor mem;
};
class Scratch {
    std::unique_lock<std::mutex> held_;
    at::Tensor mem_;

  public:
    Scratch(at::Device device, size_t bytes) {
        static auto* all = new std::map<std::pair<int, void*>, Buffer>();   // never torn down: outlives the CUDA context
        static std::mutex all_lock;
        c10::cuda::CUDAStream s = c10::cuda::getCurrentCUDAStream(device.index());
        Buffer* buf;
        {
            std::lock_guard<std::mutex> g(all_lock);
            buf = &(*all)[{device.index(), (void*)s.stream()}];   // (entries of a map stay where they are)
        }
        held_ = std::unique_lock<std::mutex>(buf->lock);
        if (!buf->mem.defined() || (size_t)buf->mem.numel() < bytes) {
            const int64_t n = bytes > USV_WS_HEADER ? (int64_t)bytes : USV_WS_HEADER;
            at::Tensor grown = at::detail::empty_cuda({n}, at::kByte, device, std::nullopt);
            if (!buf->mem.defined()) check(usv_workspace_init(grown.data_ptr(), s.stream()), "usv_workspace_init");
            else grown.narrow(0, 0, USV_WS_HEADER).copy_(buf->mem.narrow(0, 0, USV_WS_HEADER));
            buf->mem = grown;
        }
        mem_ = buf->mem;
    }
    void* ptr() const { return mem_.data_ptr(); }
    size_t bytes() const { return (size_t)mem_.numel(); }
    const at::Tensor& mem() const { return mem_; }
};

PyObject* wrap(const at::Tensor& t) {
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}
PyObject* tuple_of(std::initializer_list<at::Tensor> ts) {
    PyObject* out = PyTuple_New((Py_ssize_t)ts.size());
    Py_ssize_t i = 0;
    for (const at::Tensor& t : ts) PyTuple_SET_ITEM(out, i++, wrap(t));
    return out;
}

int blocks(int64_t n) { return (int)((n + USV_BLOCK - 1) / USV_BLOCK); }

// ---- (q, k, Nq, Nk, out)
PyObject* block_scores(PyObject* const* a) {
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]);
    const usv_strides sq = view(q, VIEW_TEXT("q")), sk = view(k, VIEW_TEXT("k"));
    const int B = (int)q.size(0), H = (int)q.size(1), d = (int)q.size(3);
    const int Nq = (int)(is_none(a[2]) ? q.size(2) : integer(a[2])), Nk = (int)(is_none(a[3]) ? k.size(2) : integer(a[3]));
    at::Tensor out = given(a[4]);
    {
        NoGil off;
        if (!out.defined()) out = fresh({B, H, blocks(Nq), blocks(Nk)}, at::kFloat, q);
        Scratch ws(q.device(), usv_block_scores_workspace(B, H, Nq, Nk, d));
        check(usv_block_scores(B, H, Nq, Nk, d, ptr(q), &sq, ptr(k), &sk, (float*)ptr(out), ws.ptr(), ws.bytes(), stream_of(q)),
              "usv_block_scores");
    }
    return wrap(out);
}

void need_scores(const at::Tensor& s, const char* what) {
    need(s.scalar_type() == at::kFloat && s.is_cuda() && s.is_contiguous() && s.dim() == 4, what);
}

// ---- (scores, k_per_head, kmax, out)
PyObject* select_blocks(PyObject* const* a) {
    const at::Tensor& s = tensor(a[0]);
    need_scores(s, "scores must be a contiguous CUDA fp32 tensor");
    const int B = (int)s.size(0), H = (int)s.size(1), NBq = (int)s.size(2), NBk = (int)s.size(3);
    const Kept kept(a[1], H);
    const int kmax = is_none(a[2]) ? kept.most : (int)integer(a[2]);
    at::Tensor out = given(a[3]);
    {
        NoGil off;
        if (!out.defined()) out = fresh({B, H, NBq, kmax > 0 ? kmax : 0}, at::kInt, s);
        check(usv_select_blocks(B, H, NBq, NBk, (const float*)ptr(s), kept.k.data(), kmax, (int32_t*)ptr(out), stream_of(s)),
              "usv_select_blocks");
    }
    return wrap(out);
}

// ---- (scores, exclude)
PyObject* set_own_block(PyObject* const* a) {
    const at::Tensor& s = tensor(a[0]);
    need_scores(s, "scores must be a contiguous CUDA fp32 [B,H,NBq,NBk] tensor");
    const bool out = truth(a[1]);
    {
        NoGil off;
        check((out ? usv_exclude_own_block : usv_force_own_block)((int)s.size(0), (int)s.size(1), (int)s.size(2), (int)s.size(3),
                                                                  (float*)ptr(s), stream_of(s)),
              out ? "usv_exclude_own_block" : "usv_force_own_block");
    }
    return Py_NewRef(a[0]);
}

// optional fp32 output: a given one is checked, and left undefined here where one is wanted but not given
at::Tensor f32_given(bool wanted, PyObject* o, at::IntArrayRef sizes, const char* what) {
    if (!wanted || is_none(o)) return at::Tensor();
    const at::Tensor& t = tensor(o);
    need(t.scalar_type() == at::kFloat && t.is_contiguous() && t.sizes() == sizes, what);
    return t;
}
PyObject* with_optional(const at::Tensor& out, const at::Tensor& f32, const at::Tensor& lse) {
    if (f32.defined()) return lse.defined() ? tuple_of({out, f32, lse}) : tuple_of({out, f32});
    return lse.defined() ? tuple_of({out, lse}) : wrap(out);
}
void need_sel(const at::Tensor& sel) {
    need(sel.scalar_type() == at::kInt && sel.is_contiguous() && sel.is_cuda() && sel.dim() == 4,
         "sel must be a contiguous CUDA int32 tensor");
}

// ---- (q, k, v, sel, k_per_head, N, scale, out, return_f32, return_lse, impl, out_f32, out_lse)
PyObject* sparse_attn_fwd(PyObject* const* a) {
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]), &sel = tensor(a[3]);
    const usv_strides sq = view(q, VIEW_TEXT("q")), sk = view(k, VIEW_TEXT("k")), sv = view(v, VIEW_TEXT("v"));
    const int64_t B = q.size(0), H = q.size(1), n = q.size(2), d = q.size(3);
    const int64_t N = is_none(a[5]) ? n : integer(a[5]);
    need_sel(sel);
    const Kept kept(a[4], H);
    at::Tensor out = given(a[7]);
    usv_strides so = {};
    if (out.defined()) so = view(out, VIEW_TEXT("o"));
    const bool f32 = truth(a[8]), want_lse = truth(a[9]);
    at::Tensor o32 = f32_given(f32, a[11], {B, H, N, d}, "out_f32 must be a contiguous fp32 [B,H,N,d] tensor");
    at::Tensor lse = f32_given(want_lse, a[12], {B, H, N}, "out_lse must be a contiguous fp32 [B,H,N] tensor");
    const int kmax = (int)sel.size(3), impl = (int)integer(a[10]);
    const float scale = (float)real(a[6]);
    {
        NoGil off;
        if (!out.defined()) {
            if (q.is_contiguous()) out = fresh({B, H, n, d}, at::kBFloat16, q);
            else out = fresh({B, n, H, d}, at::kBFloat16, q).permute({0, 2, 1, 3});   // token-major memory
            so = usv_strides{out.stride(0), out.stride(1), out.stride(2)};
        }
        if (f32 && !o32.defined()) o32 = fresh({B, H, N, d}, at::kFloat, q);
        if (want_lse && !lse.defined()) lse = fresh({B, H, N}, at::kFloat, q);
        Scratch ws(q.device(), usv_sparse_attn_workspace((int)B, (int)H, (int)N, (int)d, kmax));
        check(usv_sparse_attn_fwd((int)B, (int)H, (int)N, (int)d, ptr(q), &sq, ptr(k), &sk, ptr(v), &sv, (const int32_t*)ptr(sel),
                                  kept.k.data(), kmax, ptr(out), &so, (float*)ptr(o32), (float*)ptr(lse), scale, impl, ws.ptr(),
                                  ws.bytes(), stream_of(q)),
              "usv_sparse_attn_fwd");
    }
    return with_optional(out, o32, lse);
}

// ---- (o1, lse1, o2, lse2, out, return_f32, return_lse)
PyObject* attn_combine(PyObject* const* a) {
    const at::Tensor &o1 = tensor(a[0]), &l1 = tensor(a[1]), &o2 = tensor(a[2]), &l2 = tensor(a[3]);
    need(o1.scalar_type() == o2.scalar_type() && (o1.scalar_type() == at::kBFloat16 || o1.scalar_type() == at::kFloat),
         "o1 and o2 must both be bf16 or both be fp32");
    for (const at::Tensor* t : {&o1, &o2})
        need(t->dim() == 4 && t->is_cuda() && t->stride(3) == 1,
             "branch outputs must be CUDA [B,H,N,d] views with a contiguous last axis");
    const int64_t B = o1.size(0), H = o1.size(1), N = o1.size(2), d = o1.size(3);
    for (const at::Tensor* l : {&l1, &l2})
        need(l->scalar_type() == at::kFloat && l->is_contiguous() && l->sizes() == at::IntArrayRef({B, H, N}),
             "lse must be a contiguous fp32 [B,H,N] tensor");
    const usv_strides s1{o1.stride(0), o1.stride(1), o1.stride(2)}, s2{o2.stride(0), o2.stride(1), o2.stride(2)};
    at::Tensor out = given(a[4]), o32, lse;
    usv_strides so = {};
    if (out.defined()) so = view(out, VIEW_TEXT("o"));
    const bool f32 = truth(a[5]), want_lse = truth(a[6]);
    {
        NoGil off;
        if (!out.defined()) {
            out = fresh({B, H, N, d}, at::kBFloat16, o1);
            so = usv_strides{out.stride(0), out.stride(1), out.stride(2)};
        }
        if (f32) o32 = fresh({B, H, N, d}, at::kFloat, o1);
        if (want_lse) lse = fresh({B, H, N}, at::kFloat, o1);
        check(usv_attn_combine((int)B, (int)H, (int)N, (int)d, ptr(o1), &s1, (const float*)ptr(l1), ptr(o2), &s2,
                               (const float*)ptr(l2), o1.scalar_type() == at::kFloat ? 1 : 0, ptr(out), &so, (float*)ptr(o32),
                               (float*)ptr(lse), stream_of(o1)),
              "usv_attn_combine");
    }
    return with_optional(out, o32, lse);
}

// ---- (q, k, sel, k_per_head, lse, N, scale)
PyObject* attn_entropy(PyObject* const* a) {
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &sel = tensor(a[2]), &lse = tensor(a[4]);
    const usv_strides sq = view(q, VIEW_TEXT("q")), sk = view(k, VIEW_TEXT("k"));
    const int64_t B = q.size(0), H = q.size(1), d = q.size(3), N = is_none(a[5]) ? q.size(2) : integer(a[5]);
    need_sel(sel);
    need(lse.scalar_type() == at::kFloat && lse.is_contiguous() && lse.sizes() == at::IntArrayRef({B, H, N}),
         "lse must be a contiguous CUDA fp32 [B,H,N] tensor");
    const Kept kept(a[3], H);
    const float scale = (float)real(a[6]);
    at::Tensor marg, ent;
    {
        NoGil off;
        marg = fresh({B, N}, at::kFloat, q);
        ent = fresh({B}, at::kFloat, q);
        Scratch ws(q.device(), usv_attn_entropy_lists_workspace((int)B, (int)H, (int)N, kept.k.data()));
        check(usv_attn_entropy_ws((int)B, (int)H, (int)N, (int)d, ptr(q), &sq, ptr(k), &sk, (const int32_t*)ptr(sel),
                                  kept.k.data(), (int)sel.size(3), (const float*)ptr(lse), scale, (float*)ptr(marg),
                                  (float*)ptr(ent), ws.ptr(), ws.bytes(), stream_of(q)),
              "usv_attn_entropy");
    }
    return tuple_of({marg, ent});
}

struct Triple {
    int v[3] = {0, 0, 0};
    Triple() = default;
    explicit Triple(PyObject* o, int64_t (*read)(PyObject*) = whole) {
        PyObject* seq = PySequence_Fast(o, "expected three numbers");
        if (seq == nullptr) throw PyErr();
        const bool three = PySequence_Fast_GET_SIZE(seq) == 3;
        try {
            need(three, "expected three numbers");
            for (int i = 0; i < 3; ++i) v[i] = (int)read(PySequence_Fast_GET_ITEM(seq, i));
        } catch (...) {
            Py_DECREF(seq);
            throw;
        }
        Py_DECREF(seq);
    }
};

void need_rows(const at::Tensor& x, const char* what) {
    need(x.dim() == 3 && x.scalar_type() == at::kBFloat16 && x.is_cuda() && x.is_contiguous(), what);
}

// ---- (x, metric, grid, part, r, dst_of, pos, debug, window, out) -> (out, dst_of, pos, u, jstar)
PyObject* token_merge(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0]);
    need_rows(x, "x must be a contiguous CUDA bf16 [B,N,C] tensor");
    const int64_t B = x.size(0), N = x.size(1), C = x.size(2);
    const Triple g(a[2]), p(a[3]);
    const int64_t r = merged_count(a[4], !is_none(a[9]));
    at::Tensor dst_of, pos, u, js, metric;
    int Hm = 0, dm = 0;
    bool debug = false;
    if (is_none(a[1])) {
        need(!is_none(a[5]), "either metric or plan is needed");
        dst_of = tensor(a[5]);
        pos = tensor(a[6]);
    } else {
        metric = tensor(a[1]);
        need(metric.dim() == 4 && metric.scalar_type() == at::kBFloat16 && metric.is_contiguous(),
             "metric must be a contiguous CUDA bf16 [B,N,Hm,dm] tensor");
        Hm = (int)metric.size(2);
        dm = (int)metric.size(3);
        debug = truth(a[7]);
    }
    at::Tensor out = given(a[9]);
    need(!out.defined() || (out.scalar_type() == at::kBFloat16 && out.is_contiguous() && out.sizes() == at::IntArrayRef({B, N - r, C})),
         "out must be a contiguous bf16 [B,N-r,C] tensor");
    const bool local = !is_none(a[8]);
    Triple w;
    if (local) w = Triple(a[8], integer);   // (any numbers, as int() takes them)
    {
        NoGil off;
        if (metric.defined()) {
            dst_of = fresh({B, N}, at::kInt, x);
            pos = fresh({B, N}, at::kInt, x);
        }
        if (debug) {
            u = fresh({B, N}, at::kFloat, x);
            js = fresh({B, N}, at::kInt, x);
        }
        if (!out.defined()) out = fresh({B, N > r ? N - r : 0, C}, at::kBFloat16, x);
        Scratch ws(x.device(), usv_token_merge_workspace((int)B, (int)N, (int)C, Hm, dm ? dm : 128));
        if (local) {
            check(usv_token_merge_local((int)B, (int)N, (int)C, ptr(x), Hm, dm, ptr(metric), g.v[0], g.v[1], g.v[2], p.v[0], p.v[1],
                                        p.v[2], w.v[0], w.v[1], w.v[2], (int)r, ptr(out), (int32_t*)ptr(dst_of), (int32_t*)ptr(pos),
                                        (float*)ptr(u), (int32_t*)ptr(js), ws.ptr(), ws.bytes(), stream_of(x)),
                  "usv_token_merge_local");
        } else {
            check(usv_token_merge((int)B, (int)N, (int)C, ptr(x), Hm, dm, ptr(metric), g.v[0], g.v[1], g.v[2], p.v[0], p.v[1], p.v[2],
                                  (int)r, ptr(out), (int32_t*)ptr(dst_of), (int32_t*)ptr(pos), (float*)ptr(u), (int32_t*)ptr(js),
                                  ws.ptr(), ws.bytes(), stream_of(x)),
                  "usv_token_merge");
        }
    }
    return tuple_of({out, dst_of, pos, u, js});
}

// ---- (dst_of, pos, grid, part, r)
PyObject* merge_plan_cache(PyObject* const* a) {
    const at::Tensor &dst_of = tensor(a[0]), &pos = tensor(a[1]);
    const int B = (int)pos.size(0), N = (int)pos.size(1);
    const Triple g(a[2]), p(a[3]);
    const size_t bytes = usv_merge_plan_cache_bytes(B, N);
    const int r = (int)integer(a[4]);
    at::Tensor cache;
    {
        NoGil off;
        cache = fresh({(int64_t)bytes}, at::kByte, pos);
        check(usv_merge_plan_cache(B, N, g.v[0], g.v[1], g.v[2], p.v[0], p.v[1], p.v[2], r, (const int32_t*)ptr(dst_of),
                                   (const int32_t*)ptr(pos), ptr(cache), bytes, stream_of(pos)),
              "usv_merge_plan_cache");
    }
    return wrap(cache);
}

// ---- (x, grid, part, r, cache, out)
PyObject* token_merge_apply(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0]), &cache = tensor(a[4]);
    need_rows(x, "x must be a contiguous CUDA bf16 [B,N,C] tensor");
    const int64_t B = x.size(0), N = x.size(1), C = x.size(2), r = merged_count(a[3], !is_none(a[5]));
    const Triple g(a[1]), p(a[2]);
    need((int64_t)g.v[0] * g.v[1] * g.v[2] != N ||   // (refused below)
             (size_t)cache.numel() * cache.element_size() >= usv_merge_plan_cache_bytes((int)B, (int)N),
         "x has more batch elements than the plan");
    at::Tensor out = given(a[5]);
    {
        NoGil off;
        if (!out.defined()) out = fresh({B, N - r, C}, at::kBFloat16, x);
        check(usv_token_merge_apply((int)B, (int)N, (int)C, ptr(x), g.v[0], g.v[1], g.v[2], p.v[0], p.v[1], p.v[2], (int)r,
                                    ptr(cache), ptr(out), stream_of(x)),
              "usv_token_merge_apply");
    }
    return wrap(out);
}

// ---- (y_merged, pos, out)
PyObject* token_unmerge(PyObject* const* a) {
    const at::Tensor &y = tensor(a[0]), &pos = tensor(a[1]);
    need_rows(y, "y_merged must be a contiguous CUDA bf16 [B,Nm,C] tensor");
    const int64_t B = y.size(0), Nm = y.size(1), C = y.size(2), N = pos.size(1);
    at::Tensor out = given(a[2]);
    {
        NoGil off;
        if (!out.defined()) out = fresh({B, N, C}, at::kBFloat16, y);
        check(usv_token_unmerge((int)B, (int)N, (int)Nm, (int)C, ptr(y), (const int32_t*)ptr(pos), ptr(out), stream_of(y)),
              "usv_token_unmerge");
    }
    return wrap(out);
}

// ---- (device index, bytes): the calling stream's scratch buffer
PyObject* workspace_py(PyObject* const* a) {
    const at::Device device(at::kCUDA, (c10::DeviceIndex)integer(a[0]));
    const size_t bytes = (size_t)integer(a[1]);
    at::Tensor mem;
    {
        NoGil off;
        mem = Scratch(device, bytes).mem();
    }
    return wrap(mem);
}

PyObject* on_error(PyObject* const* a) {
    Py_XDECREF(g_raise);
    g_raise = Py_NewRef(a[0]);
    Py_RETURN_NONE;
}

template <PyObject* (*F)(PyObject* const*), int NARGS>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != NARGS) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", NARGS, n);
        return nullptr;
    }
    HANDLE_TH_ERRORS
    try {
        return F(args);
    } catch (const ValueErr& e) {
        PyErr_SetString(PyExc_ValueError, e.what);
    } catch (const PyErr&) {
    } catch (const Status& s) {
        PyObject* r = g_raise ? PyObject_CallFunction(g_raise, "is", s.status, s.where) : nullptr;
        Py_XDECREF(r);
        if (!::PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, s.where);
    }
    return nullptr;
    END_HANDLE_TH_ERRORS
}

#define FN(name, f, n) {name, (PyCFunction)(void (*)(void))entry<f, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FN("block_scores", block_scores, 5),
                         FN("select_blocks", select_blocks, 4),
                         FN("set_own_block", set_own_block, 2),
                         FN("sparse_attn_fwd", sparse_attn_fwd, 13),
                         FN("attn_combine", attn_combine, 7),
                         FN("attn_entropy", attn_entropy, 7),
                         FN("token_merge", token_merge, 10),
                         FN("merge_plan_cache", merge_plan_cache, 5),
                         FN("token_merge_apply", token_merge_apply, 6),
                         FN("token_unmerge", token_unmerge, 3),
                         FN("workspace", workspace_py, 2),
                         FN("on_error", on_error, 1),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_usv", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__usv(void) { return PyModule_Create(&module); }
