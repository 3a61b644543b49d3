// Argument marshalling of the hot calls, from torch tensors to libssd's C entry points.
//
// A decoding step is five calls of a few microseconds of GPU work each; marshalled in Python
// through ctypes they took 52 us of host time, more than the GPU needs for a small batch.  Each
// function here takes what the binding function of the same name takes, with the result buffers
// given and no launch options, and answers the C call's status -- or None, having done nothing,
// for anything that is not plainly fine (another type, a host tensor, a missing buffer, a shape
// the binding refuses): the binding then goes its general way and raises what it always raised.
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>

#include <climits>

#include "../../include/ssd.h"

namespace {

struct Unhandled {};

const at::Tensor &tensor(PyObject *o) {
    if (!o || !THPVariable_Check(o)) throw Unhandled{};
    return THPVariable_Unpack(o);
}
void *address(const at::Tensor &t) {
    if (!t.is_cuda()) throw Unhandled{};
    return t.data_ptr();
}
void *address(PyObject *o) { return address(tensor(o)); }
void *address_or_null(PyObject *o) { return !o || o == Py_None ? nullptr : address(o); }

// the buffer `key` of the dict of results; absent or None where the call allows it
PyObject *entry(PyObject *out, PyObject *key) {
    PyObject *v = PyDict_GetItemWithError(out, key);
    if (!v && PyErr_Occurred()) { PyErr_Clear(); throw Unhandled{}; }
    return v;
}

struct Rows {
    void *p;
    int64_t n, ld, V;
    ssd_dtype dtype;
};
Rows rows(PyObject *o, PyObject *V) {
    const at::Tensor &t = tensor(o);
    if (t.dim() != 2 || t.stride(1) != 1) throw Unhandled{};
    Rows r;
    r.n = t.size(0);
    r.ld = r.n > 1 ? t.stride(0) : std::max(t.stride(0), t.size(1));
    if (t.scalar_type() == at::kFloat) r.dtype = SSD_F32;
    else if (t.scalar_type() == at::kBFloat16) r.dtype = SSD_BF16;
    else throw Unhandled{};
    r.V = t.size(1);
    if (V != Py_None) {
        if (!PyLong_Check(V)) throw Unhandled{};
        int over = 0;
        r.V = PyLong_AsLongLongAndOverflow(V, &over);
        if (over) throw Unhandled{};
    }
    if (r.V < INT_MIN || r.V > INT_MAX) throw Unhandled{};
    r.p = address(t);
    return r;
}
const at::Tensor &typed(PyObject *o, at::ScalarType type) {
    const at::Tensor &t = tensor(o);
    if (t.scalar_type() != type || t.dim() < 1) throw Unhandled{};
    return t;
}
int32_t utterances(const at::Tensor &off) {
    const int64_t B = off.size(0) - 1;
    if (B < 0 || B > INT_MAX) throw Unhandled{};
    return (int32_t)B;
}
int32_t int32(PyObject *o) {
    if (!PyLong_Check(o)) throw Unhandled{};
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over || v < INT_MIN || v > INT_MAX) throw Unhandled{};
    return (int32_t)v;
}
float number(PyObject *o) {
    if (PyFloat_Check(o)) return (float)PyFloat_AS_DOUBLE(o);
    if (!PyLong_Check(o)) throw Unhandled{};
    const double v = PyLong_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) { PyErr_Clear(); throw Unhandled{}; }
    return (float)v;
}
void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

PyObject *K_workspace, *K_frame_entropy, *K_frame_argmax, *K_frame_lse, *K_frame_logprob,
    *K_draft_tokens, *K_draft_frames, *K_draft_len, *K_draft_full_len, *K_utt_max_entropy,
    *K_utt_status, *K_gate_accept, *K_max_entropy, *K_token_logp, *K_row_lse, *K_accepted_len,
    *K_all_accepted, *K_rows_read, *K_final_tokens, *K_final_len, *K_is_final, *K_ar_count, *K_ar_utt,
    *K_ar_resume, *K_next_token, *K_next_logp, *K_row_status;

struct Scratch {
    void *p;
    size_t bytes;
};
Scratch scratch(PyObject *o, bool needed) {
    if (!o || o == Py_None) {
        if (needed) throw Unhandled{};
        return {nullptr, 0};
    }
    const at::Tensor &t = tensor(o);
    return {address(t), (size_t)t.numel()};
}

// Runs `body`, which marshals under the interpreter lock and returns what to call without it.
template <typename Body> PyObject *guarded(Py_ssize_t have, Py_ssize_t want, Body body) {
    try {
        if (have != want) throw Unhandled{};
        auto call = body();
        int32_t rc;
        Py_BEGIN_ALLOW_THREADS
        rc = call();
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (...) {
        // only marshalling throws (the entry points are C): nothing has been enqueued
        Py_RETURN_NONE;
    }
}

// a subclass may answer for its items itself
void need_dict(PyObject *o) { if (!PyDict_CheckExact(o)) throw Unhandled{}; }

// ctc_draft(logits, frame_off, blank_id, max_draft_len, V, out)
PyObject *ctc_draft(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 6, [&] {
        const Rows x = rows(a[0], a[4]);
        const at::Tensor &off = typed(a[1], at::kLong);
        const int32_t B = utterances(off), blank = int32(a[2]), cap = int32(a[3]);
        PyObject *o = a[5];
        need_dict(o);
        const Scratch ws = scratch(entry(o, K_workspace), false);
        auto *fo = (const int64_t *)address(off);
        auto *fe = (float *)address(entry(o, K_frame_entropy));
        auto *fa = (int32_t *)address(entry(o, K_frame_argmax));
        auto *fl = (float *)address_or_null(entry(o, K_frame_lse));
        auto *lp = (float *)address_or_null(entry(o, K_frame_logprob));
        auto *dt = (int32_t *)address(entry(o, K_draft_tokens));
        auto *df = (int32_t *)address_or_null(entry(o, K_draft_frames));
        auto *dl = (int32_t *)address(entry(o, K_draft_len));
        auto *du = (int32_t *)address(entry(o, K_draft_full_len));
        auto *um = (float *)address(entry(o, K_utt_max_entropy));
        auto *us = (uint32_t *)address(entry(o, K_utt_status));
        void *st = stream();
        return [=] {
            return ssd_ctc_draft(x.p, x.dtype, (int32_t)x.V, x.ld, fo, B, x.n, blank, cap, fe, fa, fl,
                                 lp, dt, df, dl, du, um, us, ws.p, ws.bytes, st, nullptr);
        };
    });
}

// gate_from_maxima(utt_max_entropy, utt_status, tau_ctc, out)
PyObject *gate_from_maxima(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 4, [&] {
        const at::Tensor &um = typed(a[0], at::kFloat), &us = typed(a[1], at::kInt);
        const int64_t B64 = um.size(0);
        if (B64 > INT_MAX) throw Unhandled{};
        const int32_t B = (int32_t)B64;
        const float tau = number(a[2]);
        need_dict(a[3]);
        auto *ga = (uint8_t *)address(entry(a[3], K_gate_accept));
        auto *me = (float *)address(entry(a[3], K_max_entropy));
        auto *ump = (const float *)address(um);
        auto *usp = (const uint32_t *)address(us);
        void *st = stream();
        return [=] {
            return ssd_entropy_gate(nullptr, nullptr, B, 0, tau, ga, me, nullptr, ump, usp, st);
        };
    });
}

// what ssd_verify and ssd_verify_early_exit have in common
struct Verify {
    Rows x;
    const int64_t *off;
    const int32_t *ids;
    int32_t B;
    float tau;
    const uint8_t *skip;
    float *logp, *lse;
    int32_t *len;
    uint8_t *all;
    uint32_t *status;
    Scratch ws;
    void *st;
};
// (logits, tok_off, draft_ids, tau_slm, skip, V, out)
Verify verify_args(PyObject *const *a) {
    Verify v;
    v.x = rows(a[0], a[5]);
    const at::Tensor &off = typed(a[1], at::kLong), &ids = typed(a[2], at::kInt);
    v.B = utterances(off);
    v.tau = number(a[3]);
    v.skip = a[4] == Py_None ? nullptr : (const uint8_t *)address(typed(a[4], at::kByte));
    PyObject *o = a[6];
    need_dict(o);
    v.off = (const int64_t *)address(off);
    v.ids = (const int32_t *)address(ids);
    v.logp = (float *)address(entry(o, K_token_logp));
    v.lse = (float *)address_or_null(entry(o, K_row_lse));
    v.len = (int32_t *)address(entry(o, K_accepted_len));
    v.all = (uint8_t *)address(entry(o, K_all_accepted));
    v.status = (uint32_t *)address(entry(o, K_utt_status));
    v.ws = scratch(entry(o, K_workspace), true);
    v.st = stream();
    return v;
}
PyObject *verify(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 7, [&] {
        const Verify v = verify_args(a);
        return [=] {
            return ssd_verify(v.x.p, v.x.dtype, (int32_t)v.x.V, v.x.ld, v.off, v.ids, v.B, v.x.n, v.tau,
                              v.skip, v.logp, v.lse, v.len, v.all, v.status, v.ws.p, v.ws.bytes, v.st,
                              nullptr);
        };
    });
}
PyObject *verify_early_exit(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 7, [&] {
        const Verify v = verify_args(a);
        auto *rr = (int32_t *)address_or_null(entry(a[6], K_rows_read));
        return [=] {
            return ssd_verify_early_exit(v.x.p, v.x.dtype, (int32_t)v.x.V, v.x.ld, v.off, v.ids, v.B,
                                         v.x.n, v.tau, v.skip, v.logp, v.lse, v.len, v.all, v.status,
                                         rr, v.ws.p, v.ws.bytes, v.st, nullptr);
        };
    });
}

// verify_shard(logits, col0, tok_off, draft_ids, skip, V_local, stats, workspace)
PyObject *verify_shard(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 8, [&] {
        const Rows x = rows(a[0], a[5]);
        if (!PyLong_Check(a[1])) throw Unhandled{};
        int over = 0;
        const int64_t col0 = PyLong_AsLongLongAndOverflow(a[1], &over);
        if (over) throw Unhandled{};
        const at::Tensor &off = typed(a[2], at::kLong), &ids = typed(a[3], at::kInt);
        const int32_t B = utterances(off);
        auto *skip = a[4] == Py_None ? nullptr : (const uint8_t *)address(typed(a[4], at::kByte));
        auto *offp = (const int64_t *)address(off);
        auto *idsp = (const int32_t *)address(ids);
        auto *stats = (float *)address(a[6]);
        const Scratch ws = scratch(a[7], true);
        void *st = stream();
        return [=] {
            return ssd_verify_shard(x.p, x.dtype, (int32_t)x.V, x.ld, col0, offp, idsp, B, x.n, skip,
                                    stats, ws.p, ws.bytes, st, nullptr);
        };
    });
}

// verify_combine(stats_all, V_total, tok_off, draft_ids, tau_slm, skip, out)
PyObject *verify_combine(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 7, [&] {
        const at::Tensor &s = typed(a[0], at::kFloat);
        if (s.dim() != 3 || s.size(2) != 3 || !s.is_contiguous() || s.size(0) > INT_MAX) throw Unhandled{};
        const int32_t R = (int32_t)s.size(0);
        const int64_t M = s.size(1);
        if (!PyLong_Check(a[1])) throw Unhandled{};
        int over = 0;
        const int64_t V = PyLong_AsLongLongAndOverflow(a[1], &over);
        if (over) throw Unhandled{};
        const at::Tensor &off = typed(a[2], at::kLong), &ids = typed(a[3], at::kInt);
        const int32_t B = utterances(off);
        const float tau = number(a[4]);
        auto *skip = (const uint8_t *)address_or_null(a[5]);
        PyObject *o = a[6];
        need_dict(o);
        auto *sp = (const float *)address(s);
        auto *offp = (const int64_t *)address(off);
        auto *idsp = (const int32_t *)address(ids);
        auto *logp = (float *)address(entry(o, K_token_logp));
        auto *lse = (float *)address_or_null(entry(o, K_row_lse));
        auto *len = (int32_t *)address(entry(o, K_accepted_len));
        auto *all = (uint8_t *)address(entry(o, K_all_accepted));
        auto *status = (uint32_t *)address(entry(o, K_utt_status));
        void *st = stream();
        return [=] {
            return ssd_verify_combine(sp, R, V, offp, idsp, B, M, tau, skip, logp, lse, len, all, status, st);
        };
    });
}

// assemble(tokens, tok_off, gate_accept, accepted_len, all_accepted, out)
PyObject *assemble(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 6, [&] {
        const at::Tensor &tok = typed(a[0], at::kInt), &off = typed(a[1], at::kLong);
        const at::Tensor &ga = typed(a[2], at::kByte), &len = typed(a[3], at::kInt),
                         &all = typed(a[4], at::kByte);
        const int32_t B = utterances(off);
        const int64_t M = tok.size(0);
        PyObject *o = a[5];
        need_dict(o);
        auto *tokp = (const int32_t *)address(tok);
        auto *offp = (const int64_t *)address(off);
        auto *gap = (const uint8_t *)address(ga);
        auto *lenp = (const int32_t *)address(len);
        auto *allp = (const uint8_t *)address(all);
        auto *ft = (int32_t *)address(entry(o, K_final_tokens));
        auto *fl = (int32_t *)address(entry(o, K_final_len));
        auto *fin = (uint8_t *)address(entry(o, K_is_final));
        auto *ac = (int32_t *)address(entry(o, K_ar_count));
        auto *au = (int32_t *)address(entry(o, K_ar_utt));
        auto *ar = (int32_t *)address(entry(o, K_ar_resume));
        void *st = stream();
        return [=] {
            return ssd_assemble(tokp, offp, B, M, gap, lenp, allp, ft, fl, fin, ac, au, ar, st);
        };
    });
}

// greedy_step(logits, V, out)
PyObject *greedy_step(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 3, [&] {
        const Rows x = rows(a[0], a[1]);
        PyObject *o = a[2];
        need_dict(o);
        auto *nt = (int32_t *)address(entry(o, K_next_token));
        auto *lp = (float *)address_or_null(entry(o, K_next_logp));
        auto *lse = (float *)address_or_null(entry(o, K_row_lse));
        auto *rs = (uint32_t *)address_or_null(entry(o, K_row_status));
        const Scratch ws = scratch(entry(o, K_workspace), true);
        void *st = stream();
        return [=] {
            return ssd_greedy_step(x.p, x.dtype, (int32_t)x.V, x.ld, x.n, nt, lp, lse, rs, ws.p, ws.bytes,
                                   st, nullptr);
        };
    });
}

#define SSD_METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SSD_METHOD(ctc_draft), SSD_METHOD(gate_from_maxima), SSD_METHOD(verify),
                         SSD_METHOD(verify_early_exit), SSD_METHOD(verify_shard),
                         SSD_METHOD(verify_combine), SSD_METHOD(assemble), SSD_METHOD(greedy_step),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_ssd_call", nullptr, -1, methods};
// torch's C++ types change from release to release: the binding compares before the first call
const char kBuiltFor[] = "_ssd_call for " SSD_BUILT_FOR;

}  // namespace

PyMODINIT_FUNC PyInit__ssd_call() {
#define SSD_KEY(k) if (!(K_##k = PyUnicode_InternFromString(#k))) return nullptr;
    SSD_KEY(workspace) SSD_KEY(frame_entropy) SSD_KEY(frame_argmax) SSD_KEY(frame_lse)
    SSD_KEY(frame_logprob) SSD_KEY(draft_tokens) SSD_KEY(draft_frames) SSD_KEY(draft_len)
    SSD_KEY(draft_full_len) SSD_KEY(utt_max_entropy) SSD_KEY(utt_status) SSD_KEY(gate_accept)
    SSD_KEY(max_entropy) SSD_KEY(token_logp) SSD_KEY(row_lse) SSD_KEY(accepted_len)
    SSD_KEY(all_accepted) SSD_KEY(rows_read) SSD_KEY(final_tokens) SSD_KEY(final_len)
    SSD_KEY(is_final) SSD_KEY(ar_count) SSD_KEY(ar_utt) SSD_KEY(ar_resume) SSD_KEY(next_token)
    SSD_KEY(next_logp) SSD_KEY(row_status)
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", kBuiltFor) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
