// Frame statistics from rows that lie in registers: what ctc_rows_direct is made of.
//
// G lanes share a row and fetch all of it at once, up to U 32-byte units a lane (the same units and
// ragged ends as in ssd_direct.cuh), so a row of up to 4 KB is one round trip and there is no stage to
// wait for, no barrier and no copy through shared memory.  With the whole row at hand its maximum comes
// first: every exponential is taken relative to it, there is nothing to re-base and no range to check.
#pragma once

#include <limits.h>
#include <math.h>

#include "ssd_common.cuh"
#include "ssd_direct.cuh"
#include "ssd_ranges.cuh"

namespace ssd {
namespace ctc {

using direct::Unit;

constexpr int kMostUnits = 4;         // a lane's, 32 bytes each
constexpr float kFloor = -1.0e30f;    // what masked logits, and slots past a row's end, count as

struct RowOut {
    float lse, H;
    int arg;
};

template <int G> __device__ __forceinline__ float group_max(float v) {
    if constexpr (G == 32) {
        return warp_max(v);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    }
}
template <int G> __device__ __forceinline__ int group_min(int v) {
    if constexpr (G == 32) {
        return __reduce_min_sync(0xffffffffu, v);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    }
}
template <int G> __device__ __forceinline__ float group_sum(float v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// A row's results are good: a sum in range, relative to a finite maximum.
__device__ __forceinline__ bool row_is_sound(float m, float S) {
    return S > 0.5f && S < INFINITY && fabsf(m) < INFINITY;      // else NaN / +inf / only -inf
}

// Log-sum-exp and entropy of a row with maximum m from S, the sum of 2^t, and A, that of t * 2^t, with
// t = x * log2e - fl(m * log2e).  What rounding left out of fl(m * log2e) every exponent carries: it
// comes out of the log-sum-exp and cancels in the entropy.
__device__ __forceinline__ void close_row(float m, float S, float A, RowOut &out) {
    const float mh = m * kLog2e, ml = fmaf(m, kLog2e, -mh);
    const float lnS = logf(S);
    out.lse = m + (lnS - ml * kLn2);
    out.H = fmaxf(lnS - kLn2 * (A / S), 0.f);
    if (!row_is_sound(m, S)) out.H = __int_as_float(0x7fc00000);       // flagged downstream
}

// A row with a NaN, a +inf, nothing above the floor, or a maximum so large that an exponent should not
// carry what rounding leaves out of its product with log2e (kMostExact: up to 1/16; from 1.2e7 up it
// reaches 1, from 3e9 fp32's exponent range), element by element and by differences.
constexpr float kMostExact = 1048576.f;
template <typename T, int G>
__device__ __noinline__ RowOut row_by_elements(const char *x, int row_bytes, int sub) {
    constexpr int ES = Elem<T>::kBytes;
    float m = -INFINITY;
    int at = INT_MAX;
    for (int e = sub * ES; e < row_bytes; e += G * ES) {
        const float v = Elem<T>::load(x + e);
        if (v > m) { m = v; at = e / ES; }
    }
    const float top = group_max<G>(m);
    RowOut out;
    out.arg = group_min<G>(m == top ? at : INT_MAX);
    if (out.arg == INT_MAX) out.arg = 0;
    float S = 0.f, A = 0.f;
    for (int e = sub * ES; e < row_bytes; e += G * ES) {
        const float t = (Elem<T>::load(x + e) - top) * kLog2e, p = ex2(t);
        S += p;
        A += p > 0.f ? t * p : 0.f;
    }
    S = group_sum<G>(S);
    A = group_sum<G>(A);
    const float lnS = logf(S);
    out.lse = top + lnS;
    out.H = row_is_sound(top, S) ? fmaxf(lnS - kLn2 * (A / S), 0.f) : __int_as_float(0x7fc00000);
    return out;
}

template <typename T> struct Words;
template <> struct Words<float> {
    static constexpr uint32_t kFloorBits = 0xf149f2cau;
    static __device__ __forceinline__ uint32_t raise(uint32_t w) {
        return __float_as_uint(fmax_nan(__uint_as_float(w), kFloor));
    }
};
template <> struct Words<bf16_t> {
    static constexpr uint32_t kFloorBits = 0xf149f149u;      // a pair of -1.0e30 (rounded)
    static __device__ __forceinline__ uint32_t raise(uint32_t w) { return bf16x2_max_nan(w, kFloorBits); }
};

// S += 2^t, A += t * 2^t for a pair.
__device__ __forceinline__ void add_pair(float2 x, float nmh, float2 &S, float2 &A) {
    const float2 t = ffma2(x, make_float2(kLog2e, kLog2e), make_float2(nmh, nmh));
    const float2 e = make_float2(ex2(t.x), ex2(t.y));
    S = fadd2(S, e);
    A = ffma2(t, e, A);
}
template <typename T> __device__ __forceinline__ void add_unit(const Unit &v, float nmh, float2 &S, float2 &A) {
    float2 sa = make_float2(0.f, 0.f), sb = sa, aa = sa, ab = sa;
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        if (Elem<T>::kBytes == 4) {
            const float2 x = make_float2(__uint_as_float(v.r[k]), __uint_as_float(v.r[k + 1]));
            if (k % 4) add_pair(x, nmh, sb, ab); else add_pair(x, nmh, sa, aa);
        } else {
            add_pair(make_float2(bf16_lo(v.r[k]), bf16_hi(v.r[k])), nmh, sa, aa);
            add_pair(make_float2(bf16_lo(v.r[k + 1]), bf16_hi(v.r[k + 1])), nmh, sb, ab);
        }
    }
    S = fadd2(S, fadd2(sa, sb));
    A = fadd2(A, fadd2(aa, ab));
}

// First element of a unit that equals m (it has one).
template <typename T> __device__ __forceinline__ int find_in_unit(const Unit &v, float m);
template <> __device__ __forceinline__ int find_in_unit<float>(const Unit &v, float m) {
    int at = 0;
#pragma unroll
    for (int k = 7; k >= 0; --k) if (__uint_as_float(v.r[k]) == m) at = k;
    return at;
}
template <> __device__ __forceinline__ int find_in_unit<bf16_t>(const Unit &v, float m) {
    int at = 0;
#pragma unroll
    for (int k = 7; k >= 0; --k) {
        if (bf16_hi(v.r[k]) == m) at = 2 * k + 1;
        if (bf16_lo(v.r[k]) == m) at = 2 * k;
    }
    return at;
}

// What a lane holds of a row: its units and the elements it has of the two ragged ends.
template <typename T, int G, int U> struct Row {
    static constexpr int ES = Elem<T>::kBytes, EPU = 32 / ES;
    static constexpr int NE = (2 * EPU + G - 1) / G;
    Unit v[U];
    float edge[NE];
    int head, units;
    // byte of edge element j, or -1
    __device__ __forceinline__ int edge_at(int j, int row_bytes, int sub) const {
        const int s = sub + j * G;
        if (s < EPU) return s * ES < head ? s * ES : -1;
        const int e = head + units + (s - EPU) * ES;
        return s < 2 * EPU && e < row_bytes ? e : -1;
    }
    __device__ __forceinline__ void load(const char *x, int row_bytes, int sub) {
        const ranges::RowUnits ru = ranges::row_units(reinterpret_cast<uintptr_t>(x), row_bytes);
        head = ru.head;
        units = ru.units;
#pragma unroll
        for (int k = 0; k < U; ++k) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[k].r[j] = Words<T>::kFloorBits;
            if ((sub + k * G) * 32 < units) v[k] = direct::load_unit(x + head + (sub + k * G) * 32);
        }
#pragma unroll
        for (int j = 0; j < NE; ++j) {
            edge[j] = kFloor;
            const int e = edge_at(j, row_bytes, sub);
            if (e >= 0) edge[j] = Elem<T>::load(x + e);
        }
    }
};

// Statistics of the row at x, which `row` holds, by the G lanes of a group (lane `sub` of them); every
// lane of the group has the answer.  All 32 lanes of the warp call it, each group with a row of its
// own.  read() is called when `row` is no longer needed: about a third of the instructions are left.
template <typename T, int G, int U, typename Read>
__device__ __forceinline__ RowOut reduce_row(Row<T, G, U> &row, const char *x, int row_bytes, int sub, Read read) {
    constexpr int ES = Elem<T>::kBytes, NE = Row<T, G, U>::NE;
    Unit (&v)[U] = row.v;
    float (&edge)[NE] = row.edge;
    float um[U], vmax = -INFINITY;
#pragma unroll
    for (int k = 0; k < U; ++k) {
        um[k] = direct::unit_max<T>(v[k]);
        vmax = fmaxf(vmax, um[k]);
    }
#pragma unroll
    for (int j = 0; j < NE; ++j) vmax = fmaxf(vmax, edge[j]);
    const float m = group_max<G>(vmax);
    RowOut out;
    {
        int at = INT_MAX;
        if (vmax == m) {
            Unit f = v[U - 1];
            int k = U - 1;
#pragma unroll
            for (int q = U - 2; q >= 0; --q)
                if (um[q] == m) { f = v[q]; k = q; }
            if (um[U - 1] == m || k < U - 1)
                at = (row.head + (sub + k * G) * 32) / ES + find_in_unit<T>(f, m);
#pragma unroll
            for (int j = 0; j < NE; ++j)
                if (edge[j] == m) at = min(at, row.edge_at(j, row_bytes, sub) / ES);
        }
        out.arg = group_min<G>(at);
    }
    const float nmh = -(m * kLog2e);
    float S, A;
#pragma unroll 1
    for (int again = 0;; ++again) {
        float2 S2 = make_float2(0.f, 0.f), A2 = S2;
#pragma unroll
        for (int k = 0; k < U; ++k) add_unit<T>(v[k], nmh, S2, A2);
#pragma unroll
        for (int j = 0; j < NE; j += 2)
            add_pair(make_float2(edge[j], j + 1 < NE ? edge[j + 1 < NE ? j + 1 : j] : kFloor), nmh, S2, A2);
        S = S2.x + S2.y;
        A = A2.x + A2.y;
        // masked logits (-inf, or a type's lowest value) make t * 2^t a NaN: once more with them raised
        if (again || !__any_sync(0xffffffffu, A != A)) break;
#pragma unroll
        for (int k = 0; k < U; ++k)
#pragma unroll
            for (int j = 0; j < 8; ++j) v[k].r[j] = Words<T>::raise(v[k].r[j]);
#pragma unroll
        for (int j = 0; j < NE; ++j) edge[j] = fmax_nan(edge[j], kFloor);
    }
    read();
    S = group_sum<G>(S);
    A = group_sum<G>(A);
    const bool odd = !(fabsf(m) < kMostExact) || !row_is_sound(m, S);
    if (__any_sync(0xffffffffu, odd)) {
        const RowOut slow = row_by_elements<T, G>(x, row_bytes, sub);
        if (odd) return slow;
    }
    close_row(m, S, A, out);
    return out;
}

}  // namespace ctc
}  // namespace ssd
