// Pieces shared by the kernels that stream rows of LLM logits through a ring of shared-memory
// stages (ssd_verify, its early-exit variant, ssd_greedy_step): the stage descriptor, the
// per-thread running sum of exponentials and its once-per-stage range check, the FMA-pipe
// exponential split, the optional running arg max, and the warp-level merge.
#pragma once

#include <limits.h>
#include <math.h>

#include "ssd_common.cuh"

namespace ssd {
namespace stream {

constexpr int kOffCacheMax = 2048;     // utterance offsets kept in shared memory up to this many
constexpr uint32_t kFlagLast = 1u, kFlagEnd = 2u;
constexpr float kSumLimit = 1.0e30f;   // a running sum at or above this (or NaN) is recomputed


struct StageDesc {
    int32_t nchunks;
    uint32_t flags;
    int64_t slot;         // index of this item's first partial
    int32_t elem0;        // row-relative index of the first element of the stage's first chunk
    int32_t gather;       // early-exit variant: byte offset of the draft token's logit, or -1
};

// Running arg max of one thread (the greedy-step variant): the largest value so far, the
// row-relative index of its first occurrence (vidx), and, while a stage is being consumed, the
// stage's chunk in which the maximum last rose (vc, -1: not in this stage).  The chunk loop only
// keeps (vmax, vc) with a predicated select: no branch, since with 32 lanes some lane's maximum
// rises in most steps and a branch would be taken nearly always.  The position inside the chunk
// is looked up once per stage (resolve_arg), while the chunk is still in shared memory.
struct ArgTrack {
    float vmax;
    int vidx, vc;
    __device__ __forceinline__ void reset() { vmax = -INFINITY; vidx = INT_MAX; vc = -1; }
};
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
template <typename T>
__device__ __forceinline__ void resolve_arg(uint32_t a0, int elem0, ArgTrack &a) {
    constexpr int EPC = Elem<T>::kPerChunk;
    if (a.vc >= 0) {
        float x[EPC];
        chunk_unpack<T>(lds128(a0 + (uint32_t)a.vc * 16), x);
        int j = EPC - 1;
#pragma unroll
        for (int k = EPC - 2; k >= 0; --k) if (x[k] == a.vmax) j = k;
        a.vidx = elem0 + a.vc * EPC + j;
        a.vc = -1;
    }
}

// Running sum of exponentials of one thread, relative to a reference logit m that is one of the
// thread's own elements (or -inf while it has seen none).  fp32 keeps full relative precision
// over its whole exponent range, so m need not be the maximum: a thread only has to notice when
// a sum came near overflow (an element far above m), which it does once per stage, and then
// redoes that stage from shared memory with the proper maximum.  The common case therefore
// costs one exponential and no comparison per logit.
struct Online {
    float m, mh;
    float2 Sa, Sb;
    __device__ __forceinline__ void reset() {
        m = -INFINITY; mh = -INFINITY; Sa = Sb = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ float total() const { return (Sa.x + Sa.y) + (Sb.x + Sb.y); }
    __device__ __forceinline__ void raise_to(float nm) {
        const float sc = ex2(fmaf(m, kLog2e, -nm * kLog2e));      // 0 when m is still -inf
        Sa = fmul2(Sa, make_float2(sc, sc));
        Sb = fmul2(Sb, make_float2(sc, sc));
        m = nm; mh = nm * kLog2e;
    }
};

__device__ __forceinline__ float2 exp2_pair(float2 x, float2 scale, float2 nmh) {
    const float2 t = ffma2(x, scale, nmh);
    return make_float2(ex2(t.x), ex2(t.y));
}
__device__ __forceinline__ float2 exp2_pair_fma(float2 x, float2 scale, float2 nmh) {
    return exp2_fma_pair(ffma2(x, scale, nmh));
}

// kF of the 4 pairs of a bf16 chunk take the FMA-pipe exponential: the special-function unit
// (16 results per clock per SM) is what bounds this kernel for bf16 logits, and the FMA pipe
// has slots to spare.
template <typename T, int kF, bool kArg>
__device__ __forceinline__ void add_chunk(const uint4 &w, float nmh, Online &st, int c, ArgTrack &at) {
    const float2 sc = make_float2(kLog2e, kLog2e), nm = make_float2(nmh, nmh);
    if (Elem<T>::kBytes == 4) {
        const float2 x0 = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
        const float2 x1 = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
        if (kArg) {
            const float v = max3f(max3f(at.vmax, x0.x, x0.y), x1.x, x1.y);
            if (v > at.vmax) at.vc = c;
            at.vmax = v;
        }
        st.Sa = fadd2(st.Sa, exp2_pair(x0, sc, nm));
        st.Sb = fadd2(st.Sb, exp2_pair(x1, sc, nm));
    } else {
        const float2 x0 = make_float2(bf16_lo(w.x), bf16_hi(w.x)), x1 = make_float2(bf16_lo(w.y), bf16_hi(w.y));
        const float2 x2 = make_float2(bf16_lo(w.z), bf16_hi(w.z)), x3 = make_float2(bf16_lo(w.w), bf16_hi(w.w));
        if (kArg) {
            const float v = max3f(max3f(max3f(max3f(at.vmax, x0.x, x0.y), x1.x, x1.y), x2.x, x2.y), x3.x, x3.y);
            if (v > at.vmax) at.vc = c;
            at.vmax = v;
        }
        st.Sa = fadd2(st.Sa, kF >= 1 ? exp2_pair_fma(x0, sc, nm) : exp2_pair(x0, sc, nm));
        st.Sb = fadd2(st.Sb, kF >= 3 ? exp2_pair_fma(x1, sc, nm) : exp2_pair(x1, sc, nm));
        st.Sa = fadd2(st.Sa, kF >= 2 ? exp2_pair_fma(x2, sc, nm) : exp2_pair(x2, sc, nm));
        st.Sb = fadd2(st.Sb, exp2_pair(x3, sc, nm));
    }
}

// Adds this thread's chunks (ct, ct + NT, ...) of a stage holding n chunks to its running sum.
// Four chunks are fetched before any is used; the last, partial group of up to three is fetched
// together as well.
// With kArg the running arg max is updated as well.
template <typename T, int kF, bool kArg>
__device__ __forceinline__ void add_chunks(uint32_t a0, int n, int ct, int NT, Online &st,
                                           ArgTrack &at) {
    const float nmh = -st.mh;
    const uint32_t step = (uint32_t)NT * 16;
    uint32_t a = a0 + (uint32_t)ct * 16;
    int c = ct;
    for (; c + 3 * NT < n; c += 4 * NT, a += 4 * step) {
        const uint4 w0 = lds128(a), w1 = lds128(a + step), w2 = lds128(a + 2 * step),
                    w3 = lds128(a + 3 * step);
        add_chunk<T, kF, kArg>(w0, nmh, st, c, at);
        add_chunk<T, kF, kArg>(w1, nmh, st, c + NT, at);
        add_chunk<T, kF, kArg>(w2, nmh, st, c + 2 * NT, at);
        add_chunk<T, kF, kArg>(w3, nmh, st, c + 3 * NT, at);
    }
    if (c < n) {
        const bool h1 = c + NT < n, h2 = c + 2 * NT < n;
        const uint4 w0 = lds128(a);
        uint4 w1 = w0, w2 = w0;
        if (h1) w1 = lds128(a + step);
        if (h2) w2 = lds128(a + 2 * step);
        add_chunk<T, kF, kArg>(w0, nmh, st, c, at);
        if (h1) add_chunk<T, kF, kArg>(w1, nmh, st, c + NT, at);
        if (h2) add_chunk<T, kF, kArg>(w2, nmh, st, c + 2 * NT, at);
    }
}

// The reference that goes with a largest element cm (-inf: still none): never below kNegInit.
// A mask of the type's lowest finite value would otherwise be one, its product with log2e would
// leave fp32's range, and a thread that met nothing else would report its row as not finite.
// Against kNegInit such elements add 0, as they do in the closing kernels' merge.
__device__ __forceinline__ float reference_of(float cm) {
    return cm > -INFINITY ? fmaxf(cm, kNegInit) : cm;
}

template <typename T, int kF, bool kArg>
__device__ __forceinline__ void consume_stage(uint32_t a0, int n, int ct, int NT, Online &st,
                                              int elem0, ArgTrack &at) {
    if (ct >= n) return;
    if (!(st.m > -INFINITY)) {
        // no reference yet (start of a row): the largest element of the first chunk
        const float cm = reference_of(chunk_max<T>(lds128(a0 + (uint32_t)ct * 16)));
        if (cm > -INFINITY) { st.m = cm; st.mh = cm * kLog2e; }
    }
    const Online saved = st;
    add_chunks<T, kF, kArg>(a0, n, ct, NT, st, at);
    if (!(st.total() < kSumLimit)) {
        // an element far above the reference, a NaN or +inf, or only -inf so far: redo the
        // stage relative to the maximum of this thread's chunks
        st = saved;
        float cm = -INFINITY;
        for (int c = ct; c < n; c += NT) cm = fmaxf(cm, chunk_max<T>(lds128(a0 + (uint32_t)c * 16)));
        cm = reference_of(cm);
        if (cm > st.m) st.raise_to(cm);
        if (st.m > -INFINITY) add_chunks<T, kF, kArg>(a0, n, ct, NT, st, at);
    }
    if (kArg) resolve_arg<T>(a0, elem0, at);
}

// Warp-level merge of the lanes' (m, S) into one pair relative to the warp maximum.  Exponents carried
// +ml: it is taken out, with the arg max by a division, after which a logit equal to the warp's maximum
// has added exactly 1 (see greedy_row).
template <bool kArg> __device__ __forceinline__ float2 warp_merge(const Online &st) {
    const float S = st.total();
    const float ml = fmaf(st.m, kLog2e, -st.mh);
    const float M = warp_max(st.m);
    // S == 0 covers lanes that saw nothing (their m is -inf); a NaN sum still propagates
    const float rebased = kArg ? S / ex2(ml) * ex2((st.m - M) * kLog2e) : S * ex2(fmaf(st.m - M, kLog2e, -ml));
    const float Sw = warp_sum(S == 0.f ? 0.f : rebased);
    return make_float2(M, Sw);
}

// ln p of a logit x of a row with maximum Mx and lnS the logarithm of its sum relative to it (not
// x - lse: keeps its accuracy when |x| is large).  NaN, which rejects, for a row with a NaN, a +inf
// or nothing above kNegInit: of such a row's masked logits none is likely.
__device__ __forceinline__ float row_logp(float x, float Mx, float lnS) {
    return fabsf(Mx + lnS) < INFINITY ? (x - Mx) - lnS : __int_as_float(0x7fc00000);
}

// Rows to read before each utterance, in shared memory, for up to 32 * L utterances from b0 on and in
// front of utterance `end`: act[b] is `total` and the rows of the ones before b, shift[b] (where asked for)
// what to add to a count of rows to have the row.  Returns the total with them.  Called by all lanes of a
// warp.  The loads are one round trip, and the L prefix sums go through the warp side by side.  Loops are
// kept rolled here and below: a CTA runs this once, and what it costs is fetching the instructions (400 bf16
// rows of 64 KB behind a gate, 8 utterances: 10.4 us unrolled, 10.0 rolled).
template <int L>
__device__ __forceinline__ int count_turn(const int64_t *tok_off, const uint8_t *skip, int end, int64_t M, int b0,
                                          int total, int32_t *act, int32_t *shift) {
    const int lane = threadIdx.x & 31;
    int64_t i0[L], i1[L];
    int skipped[L], mine[L], incl[L];
#pragma unroll
    for (int j = 0; j < L; ++j) {
        const int b = b0 + 32 * j + lane;
        i0[j] = load_if(b < end, tok_off + b);
        i1[j] = load_if(b < end, tok_off + b + 1);
        skipped[j] = load_if(b < end, skip + b);
    }
#pragma unroll
    for (int j = 0; j < L; ++j)
        incl[j] = mine[j] = i0[j] < 0 || i1[j] < i0[j] || i1[j] > M || skipped[j] ? 0 : (int)(i1[j] - i0[j]);
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int j = 0; j < L; ++j) {
            const int y = __shfl_up_sync(0xffffffffu, incl[j], o);
            if (lane >= o) incl[j] += y;
        }
#pragma unroll
    for (int j = 0; j < L; ++j) {
        const int b = b0 + 32 * j + lane, before = total + incl[j] - mine[j];
        if (b < end) {
            act[b] = before;
            if (shift) shift[b] = (int)i0[j] - before;
        }
        total += __shfl_sync(0xffffffffu, incl[j], 31);
    }
    return total;
}
// Rows to read before each utterance (act[B]: their total, which is returned), in shared memory, and what
// to add to such a count to have the row (shift, where asked for).  Called by all threads of a block;
// warp_tot has a word per warp.
__device__ __forceinline__ int count_rows(const int64_t *tok_off, const uint8_t *skip, int B, int64_t M,
                                          int32_t *act, int32_t *warp_tot, const int warps, int32_t *shift) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int share = 32 * ((B + 32 * warps - 1) / (32 * warps)), b0 = warp * share, end = min(B, b0 + share);
    int mine = 0;                        // rows of this warp's utterances
    if (b0 < B) {
        if (share > 32)
            for (int b = b0; b < end; b += 128) mine = count_turn<4>(tok_off, skip, end, M, b, mine, act, shift);
        else
            mine = count_turn<1>(tok_off, skip, end, M, b0, 0, act, shift);
    }
    if (lane == 0) warp_tot[warp] = mine;
    __syncthreads();
    const int each = lane < warps ? warp_tot[lane] : 0;
    const int before = __reduce_add_sync(0xffffffffu, lane < warp ? each : 0);
    const int total = __reduce_add_sync(0xffffffffu, each);
#pragma unroll 1
    for (int b = b0 + lane; b < end; b += 32) {
        act[b] += before;
        if (shift) shift[b] -= before;
    }
    if (threadIdx.x == 0) act[B] = total;
    __syncthreads();
    return total;
}
// The same by one warp, for itself, of up to 128 utterances; with `rehearse` it reads and counts nothing.
__device__ __forceinline__ int count_rows_by_warp(const int64_t *tok_off, const uint8_t *skip, int B, int64_t M,
                                                  int32_t *act, int32_t *shift, bool rehearse) {
    const int end = rehearse ? 0 : B;
    const int total = B > 32 ? count_turn<4>(tok_off, skip, end, M, 0, 0, act, shift)
                             : count_turn<1>(tok_off, skip, end, M, 0, 0, act, shift);
    if ((threadIdx.x & 31) == 0) act[B] = total;
    __syncwarp();
    return total;
}
// Whether none of the B + 1 offsets is below the one before it.  Called by all lanes of a warp.
__device__ __forceinline__ int offsets_ordered(const int64_t *off, int B) {
    constexpr int L = 4;                 // pairs a lane has in flight
    const int lane = threadIdx.x & 31;
    bool ok = true;
    for (int b0 = 0; b0 < B; b0 += 32 * L) {
        int64_t i0[L], i1[L];
#pragma unroll
        for (int j = 0; j < L; ++j) {
            const int b = min(b0 + 32 * j + lane, B - 1);
            i0[j] = off[b];
            i1[j] = off[b + 1];
        }
#pragma unroll
        for (int j = 0; j < L; ++j) ok = ok && i0[j] <= i1[j];
    }
    return __all_sync(0xffffffffu, ok);
}
// The utterance that has row number `at`, below the total: the last one with no more than that many
// rows before it.
__device__ __forceinline__ int utterance_of_count(const int32_t *act, int B, int at) {
    int lo = 0, hi = B - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (act[mid] <= at) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Greedy step: a row closed by one warp from its P partials (reference, sum, largest logit, an
// index).  The ring's index is that of the logit's first occurrence; the direct-load kernel's (kUnit)
// lies up to one 32-byte unit before it, and the unit is looked through here, once per row instead of
// once per column span.  (The look-up is a dependent load: 400 fp32 rows of 128 KB, which the ring
// reads, 15.3 us with it, 14.3 without; 1,024 of 192 KB 36.5, 35.4.)
struct GreedyRow {
    int token;
    float logp, lse;
    uint32_t status;
};
template <typename T, bool kUnit, typename Get>
__device__ __forceinline__ GreedyRow greedy_row(Get get, int P, const char *row, int V, int lane) {
    // three looks at the partials: held in registers where they are few enough, since in the workspace
    // each look is a round trip (450 rows of 220 KB, 10 partials each: 20.9 us the call, 21.8 with three)
    constexpr int L = 4;
    float4 held[L];
    const bool few = P <= 32 * L;
#pragma unroll
    for (int j = 0; j < L; ++j) {
        held[j] = make_float4(kNegInit, 0.f, -INFINITY, __int_as_float(INT_MAX));
        if (few && 32 * j + lane < P) held[j] = get(32 * j + lane);
    }
    auto each = [&](auto look) {
        if (few) {
#pragma unroll
            for (int j = 0; j < L; ++j) look(held[j]);
        } else {
#pragma unroll 1
            for (int q = lane; q < P; q += 32) look(get(q));
        }
    };
    float Mx = kNegInit, vm = -INFINITY;
    each([&](const float4 &v) {
        Mx = fmaxf(Mx, v.x);
        vm = fmaxf(vm, v.z);
    });
    Mx = warp_max(Mx);
    vm = warp_max(vm);
    // Sums are taken relative to the largest logit, and its own exponential is taken out of the one partial
    // that holds it: what is left beside it is all that the logarithm of a confident row is about.  It is
    // taken in the form that the partial has it: below 4,096 the exponents of both carry what rounding left
    // out of the reference's product with log2e, which the direct loads (kUnit) take out by a product and
    // the ring by a quotient; from there on the direct loads hold differences, and in the ring's quotient the
    // reference itself is 1 (1e10 * log2e is rounded by 440: no such factor is in fp32's range).
    const bool plain = vm > kNegInit;
    const float base = plain ? vm : Mx;
    int vi = INT_MAX;
    float ref = 0.f;                  // of the first partial of this lane that has the largest logit
    each([&](const float4 &v) {
        if (v.z == vm && __float_as_int(v.w) < vi) { vi = __float_as_int(v.w); ref = v.x; }
    });
    const int mine = vi;
    vi = __reduce_min_sync(0xffffffffu, vi);
    const int found = vi;
    float beside = -INFINITY;
    if (kUnit && vi >= 0 && vi < V) {             // on its way while the sums are joined
        const int64_t e = (int64_t)vi + lane;
        if (lane < 32 / Elem<T>::kBytes && e < V) beside = Elem<T>::load(row + e * Elem<T>::kBytes);
    }
    float own = 0.f;                  // in one lane, each partial having its own indexes; once, not for each held
    if (plain && mine == found) {
        const float nmh = -(ref * kLog2e), up = ex2(fmaf(vm, kLog2e, nmh)), carried = fmaf(ref, kLog2e, nmh);
        if (!(fabsf(ref) < 4096.f)) own = ex2((vm - ref) * kLog2e);
        else if (kUnit) own = up * ex2(-carried);
        else own = up / ex2(carried);
    }
    float S = 0.f;
    each([&](const float4 &v) {
        const bool holds = v.z == vm && __float_as_int(v.w) == found;
        S += (v.y - (holds ? own : 0.f)) * ex2((v.x - base) * kLog2e);
    });
    S = warp_sum(S);
    if (kUnit) {
        const unsigned hits = __ballot_sync(0xffffffffu, beside == vm && vm > -INFINITY);
        if (hits) vi += __ffs(hits) - 1;
    }
    GreedyRow g;
    // what is left is not negative but for rounding; a NaN stays one
    const float lnS = plain ? log1pf(S < 0.f ? 0.f : S) : logf(S);
    g.lse = base + lnS;
    g.logp = (vm - base) - lnS;
    g.status = fabsf(g.lse) < INFINITY ? 0u : (uint32_t)SSD_UTT_NONFINITE;
    g.token = (vi < 0 || vi >= V) ? 0 : vi;
    return g;
}

}  // namespace stream
}  // namespace ssd
