// The binding's frequent calls, from Python objects straight to the C ABI.
//
// A ctypes call of one of these functions spends 10 to 15 us on the host: a Python object per pointer, tensor slices for
// matrix b of a plan, a parameter struct, a Stream object.  The kernels of a decode step take 3 to 9 us, so that was the
// time of the call.  Here tensors are unpacked in C++ (about 1 us in all).  Arguments and error codes are those of the C
// ABI; checks that concern Python arguments raise AssertionError as the Python wrappers do.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "variopath.h"

namespace {

struct Failed {};                       // a Python error has been set

[[noreturn]] void fail(PyObject* type, const char* text) {
    if (!PyErr_Occurred()) PyErr_SetString(type, text);
    throw Failed{};
}

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "a tensor is expected");
    return THPVariable_Unpack(o);
}
void* ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }

long long integer(PyObject* o) {
    if (PyLong_CheckExact(o)) {
        const long long v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) throw Failed{};
        return v;
    }
    PyObject* n = PyNumber_Long(o);
    if (!n) throw Failed{};
    const long long v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    return v;
}

struct Ref {                            // an owned reference
    PyObject* o;
    explicit Ref(PyObject* p) : o(p) { if (!o) throw Failed{}; }
    ~Ref() { Py_DECREF(o); }
    Ref(const Ref&) = delete;
};

#define NAMES(X) X(_h) X(value) X(N) X(lambda_ns) X(granule_bytes) X(k_target) X(n_start) X(i_aa) X(k_max) X(n_steps) X(chan_id) \
    X(lane_dst) X(lane_inst) X(lane_bytes) X(send_off) X(recv_off) X(tau_ns) X(status) X(cuda_stream)
#define DECLARE(n) PyObject* s_##n;
NAMES(DECLARE)

long long attr_int(PyObject* o, PyObject* name) { Ref r(PyObject_GetAttr(o, name)); return integer(r.o); }
void* attr_ptr(PyObject* o, PyObject* name) { Ref r(PyObject_GetAttr(o, name)); return ptr(r.o); }

// Address of row b of a plan array (its first dimension is the batch).
template <typename T>
T* row_of(PyObject* plan, PyObject* name, long long b, long long* last = nullptr) {
    Ref r(PyObject_GetAttr(plan, name));
    const at::Tensor& t = tensor(r.o);
    if (b < 0) b += t.size(0);
    if (b < 0 || b >= t.size(0)) fail(PyExc_IndexError, "matrix index out of range");
    if (last) *last = t.size(t.dim() - 1);
    return (T*)((char*)t.data_ptr() + b * t.stride(0) * (long long)t.element_size());
}

void* stream_of(PyObject* o) {
    if (o == Py_None) return (void*)c10::cuda::getCurrentCUDAStream().stream();
    Ref r(PyObject_GetAttr(o, s_cuda_stream));
    return (void*)(uintptr_t)(unsigned long long)integer(r.o);
}

const vp_catalog* handle_of(PyObject* catalog) {
    Ref h(PyObject_GetAttr(catalog, s__h));
    if (h.o == Py_None) return nullptr;
    Ref v(PyObject_GetAttr(h.o, s_value));
    return v.o == Py_None ? nullptr : (const vp_catalog*)PyLong_AsVoidPtr(v.o);
}

vp_sched_params params_of(PyObject* p, long long N) {
    vp_sched_params q;
    q.lambda_ns = attr_int(p, s_lambda_ns);
    q.granule_bytes = attr_int(p, s_granule_bytes);
    q.k_target = (int32_t)attr_int(p, s_k_target);
    q.n_start = (int32_t)attr_int(p, s_n_start);
    q.i_aa = (int32_t)attr_int(p, s_i_aa);
    const long long k = attr_int(p, s_k_max);
    q.k_max = (int32_t)(k ? k : 8 * N);
    return q;
}

size_t bytes_of(const at::Tensor& t) { return (size_t)t.numel() * t.element_size(); }
bool is_i32(const at::Tensor& t) { return t.is_cuda() && t.scalar_type() == at::kInt && t.is_contiguous(); }
bool on_gpu(const at::Tensor& t) { return t.is_cuda() && t.is_contiguous(); }
void check(bool ok, const char* text) { if (!ok) fail(PyExc_AssertionError, text); }

template <typename F>
PyObject* call(Py_ssize_t n, Py_ssize_t want, F f) {
    if (n != want) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; }
    try {
        return PyLong_FromLong(f());
    } catch (const Failed&) {
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}
#define WITHOUT_GIL(rc, expr) { Py_BEGIN_ALLOW_THREADS rc = (expr); Py_END_ALLOW_THREADS }

// ---- one function per call; argument order as in binding.py ------------------------------------------------------------

using SchedFn = int (*)(const vp_catalog*, const vp_sched_params*, const int64_t*, const int64_t*, int, int32_t*, int32_t*, int16_t*,
                        uint16_t*, int64_t*, int64_t*, int64_t*, int64_t*, int32_t*, void*, size_t, void*);

// (catalog, params, demand, tau_ns_in, plan, workspace, stream)
int schedule(SchedFn fn, PyObject* const* a, bool host) {
    const at::Tensor& demand = tensor(a[2]);
    check((host ? !demand.is_cuda() : demand.is_cuda()) && demand.scalar_type() == at::kLong && demand.is_contiguous(),
          host ? "demand: a contiguous int64 host tensor" : "demand: a contiguous int64 device tensor");
    const long long N = attr_int(a[0], s_N), B = demand.size(0);
    check(host || (demand.dim() == 3 && demand.size(1) == N && demand.size(2) == N), "demand: [B, N, N]");
    const vp_catalog* c = handle_of(a[0]);
    const vp_sched_params p = params_of(a[1], N);
    PyObject* plan = a[4];
    void *n_steps = attr_ptr(plan, s_n_steps), *chan = attr_ptr(plan, s_chan_id), *dst = attr_ptr(plan, s_lane_dst),
         *inst = attr_ptr(plan, s_lane_inst), *bytes = attr_ptr(plan, s_lane_bytes), *so = attr_ptr(plan, s_send_off),
         *ro = attr_ptr(plan, s_recv_off), *tau = attr_ptr(plan, s_tau_ns), *st = attr_ptr(plan, s_status);
    const at::Tensor& ws = tensor(a[5]);
    const int64_t *d = (const int64_t*)demand.data_ptr(), *tin = (const int64_t*)ptr(a[3]);
    void *w = ws.data_ptr(), *stream = stream_of(a[6]);
    const size_t wb = (size_t)ws.numel();
    int rc;
    WITHOUT_GIL(rc, fn(c, &p, d, tin, (int)B, (int32_t*)n_steps, (int32_t*)chan, (int16_t*)dst, (uint16_t*)inst, (int64_t*)bytes,
                       (int64_t*)so, (int64_t*)ro, (int64_t*)tau, (int32_t*)st, w, wb, stream))
    return rc;
}
PyObject* schedule_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 7, [&] { return schedule(vp_schedule_batch, a, false); });
}
PyObject* schedule_batch_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 7, [&] { return schedule(vp_schedule_batch_host, a, true); });
}
PyObject* schedule_batch_host_used(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 7, [&] { return schedule(vp_schedule_batch_host_used, a, true); });
}

// (expert_idx, experts_per_rank, N, row_bytes, src0, out, status, stream)
PyObject* demand_from_routing(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 8, [&] {
        const at::Tensor& idx = tensor(a[0]);
        check(is_i32(idx) && idx.dim() == 3, "expert_idx: a contiguous int32 device tensor [n_src, T, topk]");
        const int epr = (int)integer(a[1]), N = (int)integer(a[2]), src0 = (int)integer(a[4]);
        const int64_t rb = integer(a[3]);
        void *out = ptr(a[5]), *st = ptr(a[6]), *stream = stream_of(a[7]);
        int rc;
        WITHOUT_GIL(rc, vp_demand_from_routing((const int32_t*)idx.data_ptr(), (int)idx.size(0), (int)idx.size(1), (int)idx.size(2), epr, N,
                                               src0, rb, (int64_t*)out, (int32_t*)st, stream))
        return rc;
    });
}

// (plan, b, rank, expert_idx, experts_per_rank, rows, staged, src_map, status, workspace or None for the static form, stream)
PyObject* pack(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 11, [&] {
        const at::Tensor &idx = tensor(a[3]), &rows = tensor(a[5]), &staged = tensor(a[6]);
        check(is_i32(idx), "expert_idx: a contiguous int32 device tensor");
        check(on_gpu(rows) && on_gpu(staged), "rows, staged: contiguous device tensors");
        check(idx.dim() == 2 && rows.dim() >= 2, "expert_idx: [T, topk], rows: [T, H]");
        const long long b = integer(a[1]);
        long long N;
        const int32_t* n_steps = row_of<int32_t>(a[0], s_n_steps, b);
        const int16_t* dst = row_of<int16_t>(a[0], s_lane_dst, b, &N);
        const int64_t *bytes = row_of<int64_t>(a[0], s_lane_bytes, b), *so = row_of<int64_t>(a[0], s_send_off, b);
        const int rank = (int)integer(a[2]), k_max = (int)attr_int(a[0], s_k_max), epr = (int)integer(a[4]);
        const int64_t rb = rows.size(1) * (int64_t)rows.element_size(), cap = (int64_t)bytes_of(staged);
        void *map = ptr(a[7]), *st = ptr(a[8]), *stream = stream_of(a[10]);
        const bool own = a[9] != Py_None;
        void* ws = own ? tensor(a[9]).data_ptr() : nullptr;
        const size_t wb = own ? (size_t)tensor(a[9]).numel() : 0;
        int rc;
        WITHOUT_GIL(rc, own ? vp_pack(n_steps, dst, bytes, so, (int)N, rank, k_max, (const int32_t*)idx.data_ptr(), (int)idx.size(0),
                                      (int)idx.size(1), epr, rows.data_ptr(), rb, staged.data_ptr(), cap, (int32_t*)map, (int32_t*)st, ws, wb, stream)
                            : vp_pack_static(n_steps, dst, bytes, so, (int)N, rank, k_max, (const int32_t*)idx.data_ptr(), (int)idx.size(0),
                                             (int)idx.size(1), epr, rows.data_ptr(), rb, staged.data_ptr(), cap, (int32_t*)map, (int32_t*)st, stream))
        return rc;
    });
}

// (plan, b, rank, staged, recv_bufs, recv_capacity, arrived, status, stream)
PyObject* exchange_put(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 9, [&] {
        const long long b = integer(a[1]);
        long long N;
        const int32_t* n_steps = row_of<int32_t>(a[0], s_n_steps, b);
        const int16_t* dst = row_of<int16_t>(a[0], s_lane_dst, b, &N);
        const int64_t *so = row_of<int64_t>(a[0], s_send_off, b), *ro = row_of<int64_t>(a[0], s_recv_off, b);
        const int rank = (int)integer(a[2]), k_max = (int)attr_int(a[0], s_k_max);
        void *staged = ptr(a[3]), *bufs = ptr(a[4]), *cap = ptr(a[5]), *arrived = ptr(a[6]), *st = ptr(a[7]), *stream = stream_of(a[8]);
        int rc;
        WITHOUT_GIL(rc, vp_exchange_put(n_steps, dst, so, ro, (int)N, rank, k_max, staged, (void* const*)bufs, (const int64_t*)cap,
                                        (uint64_t* const*)arrived, (int32_t*)st, stream))
        return rc;
    });
}

// (plan, b, rank, recv, recv_expert, experts_per_rank, out, expert_off, out_src, out_map, status, workspace, stream)
PyObject* unpack(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 13, [&] {
        const at::Tensor &recv = tensor(a[3]), &ex = tensor(a[4]), &out = tensor(a[6]), &ws = tensor(a[11]);
        check(on_gpu(recv) && recv.dim() == 2 && on_gpu(out), "recv, out: contiguous device tensors, recv [capacity_rows, H]");
        check(is_i32(ex), "recv_expert: a contiguous int32 device tensor");
        check(ex.numel() >= recv.size(0) && bytes_of(out) >= bytes_of(recv), "recv_expert, out: as large as recv");
        const long long b = integer(a[1]);
        long long N;
        const int32_t* n_steps = row_of<int32_t>(a[0], s_n_steps, b);
        const int16_t* dst = row_of<int16_t>(a[0], s_lane_dst, b, &N);
        const int64_t* ro = row_of<int64_t>(a[0], s_recv_off, b);
        const int rank = (int)integer(a[2]), k_max = (int)attr_int(a[0], s_k_max), epr = (int)integer(a[5]);
        const int64_t rb = recv.size(1) * (int64_t)recv.element_size();
        void *off = ptr(a[7]), *src = ptr(a[8]), *map = ptr(a[9]), *st = ptr(a[10]), *stream = stream_of(a[12]);
        int rc;
        WITHOUT_GIL(rc, vp_unpack(n_steps, dst, ro, (int)N, rank, k_max, recv.data_ptr(), rb, recv.size(0), (const int32_t*)ex.data_ptr(), epr,
                                  out.data_ptr(), (int32_t*)off, (int32_t*)src, (int32_t*)map, (int32_t*)st, ws.data_ptr(), (size_t)ws.numel(), stream))
        return rc;
    });
}

// (plan, b, rank, expert_idx, experts_per_rank, recv, out, out_map, status, workspace, stream)
PyObject* unpack_tokens(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call(n, 11, [&] {
        const at::Tensor &idx = tensor(a[3]), &recv = tensor(a[5]), &out = tensor(a[6]), &ws = tensor(a[9]);
        check(is_i32(idx) && idx.dim() == 2, "expert_idx: a contiguous int32 device tensor [T, topk]");
        check(on_gpu(recv) && recv.dim() == 2 && on_gpu(out), "recv, out: contiguous device tensors, recv [capacity_rows, H]");
        const int64_t rb = recv.size(1) * (int64_t)recv.element_size();
        check((int64_t)bytes_of(out) >= idx.numel() * rb, "out: a row per routed copy");
        const long long b = integer(a[1]);
        long long N;
        const int32_t* n_steps = row_of<int32_t>(a[0], s_n_steps, b);
        const int16_t* dst = row_of<int16_t>(a[0], s_lane_dst, b, &N);
        const int64_t *bytes = row_of<int64_t>(a[0], s_lane_bytes, b), *ro = row_of<int64_t>(a[0], s_recv_off, b);
        const int rank = (int)integer(a[2]), k_max = (int)attr_int(a[0], s_k_max), epr = (int)integer(a[4]);
        void *map = ptr(a[7]), *st = ptr(a[8]), *stream = stream_of(a[10]);
        int rc;
        WITHOUT_GIL(rc, vp_unpack_tokens(n_steps, dst, bytes, ro, (int)N, rank, k_max, (const int32_t*)idx.data_ptr(), (int)idx.size(0),
                                         (int)idx.size(1), epr, recv.data_ptr(), rb, recv.size(0), out.data_ptr(), (int32_t*)map, (int32_t*)st,
                                         ws.data_ptr(), (size_t)ws.numel(), stream))
        return rc;
    });
}

#define METHOD(n) {#n, (PyCFunction)(void*)n, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(schedule_batch), METHOD(schedule_batch_host), METHOD(schedule_batch_host_used), METHOD(demand_from_routing),
                         METHOD(pack), METHOD(exchange_put), METHOD(unpack), METHOD(unpack_tokens), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() {
#define INTERN(n) if (!(s_##n = PyUnicode_InternFromString(#n))) return nullptr;
    NAMES(INTERN)
    return PyModule_Create(&module);
}
