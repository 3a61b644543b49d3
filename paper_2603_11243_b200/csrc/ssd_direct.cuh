// verify_rows_direct: the streaming kernel of ssd_verify, ssd_verify_shard and ssd_greedy_step
// (use_direct in ssd_verify.cu says on which sizes and types, and what it measured against the ring
// of verify_rows_tma).
//
// A warp works on one span of columns of one row at a time and reads it with 32-byte loads
// straight into registers: no shared memory, no barriers, no hand-over between warps.  What
// bounds it on long batches is the 1 kW power cap (between events, a kernel that only reads takes 611
// us for 4.4 GB there, the ring 710, this one 665), so what counts is instructions per logit: 4.3 of
// 304 KB rows here, 6.0 of 98 KB rows in the ring (executed instructions as ncu counts them).
// 148 x 32 warps keep two blocks of 1 KB each in flight (one where a span ends: the
// next span's second block is asked for when its first has given the reference), the block loop
// holds nothing but the loads, the sums and a counter, and everything that happens once per span
// (reference, range check, merge of the lanes) is done once for the warp instead of once per
// thread.  More in flight was slower throughout (two units a lane and block: +3 %; 48 warps: +18
// %; bulk prefetch to L2: +3 % and more), and so were blocks interleaved among warps.
#pragma once

#include "ssd_common.cuh"
#include "ssd_ranges.cuh"
#include "ssd_stream.cuh"

namespace ssd {
namespace direct {

using ranges::kDirectBlockBytes;

constexpr int kThreads = 512, kWarps = kThreads / 32, kCtasPerSm = 2;
// A lane's sums are joined to its total every so many blocks (even).  With one logit far above the
// rest in them, sums absorb what each unit adds up to half an ulp: up to 2^-25 of the row's
// probability a term, for every term that is added one by one.  Of 297 blocks (152,064 bf16
// logits in one span) that made 9e-6; 16 and 19 joins make 1e-6, below the 3e-6 of a ring thread
// with its 99 chunks.
constexpr int kGroupBlocks = 16;
using ranges::kSpanSumLimit;

struct DirectParams {
    const char *logits;
    int64_t row_pitch;
    int row_bytes;
    int64_t M;
    Cut cut[kCuts];        // how rows are cut: cut[k] where at most M >> k of them are read
    int pairs;             // pairs per row in `partials`
    const int64_t *tok_off;
    int B;
    const uint8_t *skip;
    int table;             // count the rows to read per utterance in shared memory first
    void *partials;        // [M, pairs] float2 (reference, sum), or float4 with the arg max
};

// One lane's 32-byte piece of a block.
struct Unit {
    uint32_t r[8];
};
__device__ __forceinline__ Unit load_unit(const char *p) {
    Unit v;
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v.r[0]), "=r"(v.r[1]), "=r"(v.r[2]), "=r"(v.r[3]), "=r"(v.r[4]),
                   "=r"(v.r[5]), "=r"(v.r[6]), "=r"(v.r[7])
                 : "l"(p));
    return v;
}

template <typename T> __device__ __forceinline__ float unit_max(const Unit &v) {
    const uint4 a = make_uint4(v.r[0], v.r[1], v.r[2], v.r[3]);
    const uint4 b = make_uint4(v.r[4], v.r[5], v.r[6], v.r[7]);
    if (Elem<T>::kBytes == 4) return fmaxf(chunk_max<float>(a), chunk_max<float>(b));
    const uint32_t h = bf16x2_max(bf16x2_max(bf16x2_max(a.x, a.y), bf16x2_max(a.z, a.w)),
                                  bf16x2_max(bf16x2_max(b.x, b.y), bf16x2_max(b.z, b.w)));
    return fmaxf(bf16_lo(h), bf16_hi(h));
}

// What a span's exponentials are taken relative to: one logit m of the warp's first block, as
// nmh = -fl(m * log2e), and for the FMA-pipe exponential a floor and a ceiling around m (ssd_ranges.cuh)
// as packed bf16 pairs.  |m| < 4096.
struct Reference {
    float m, nmh;
    uint32_t floor2 = 0, ceil2 = 0;
    template <typename T> __device__ __forceinline__ void set(float to) {
        m = to;
        nmh = -(to * kLog2e);
        if (Elem<T>::kBytes == 2) {
            floor2 = ranges::bf16_floor(to) * 0x10001u;
            ceil2 = ranges::bf16_ceiling(to) * 0x10001u;
        }
    }
};

// kF of a bf16 unit's eight pairs take the FMA-pipe exponential.  The unit's terms are summed
// apart and join the lane's sums once: a span with one logit far above the rest leaves large
// values in a sum, and a thousand small terms added to that one by one would each lose the same
// fraction of an ulp.
template <typename T, int kF>
__device__ __forceinline__ void add_unit(const Unit &v, const Reference &ref, float2 &Sa, float2 &Sb) {
    const float2 sc = make_float2(kLog2e, kLog2e), nm = make_float2(ref.nmh, ref.nmh);
    float2 ta, tb;
    if (Elem<T>::kBytes == 4) {
        float2 e[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            e[k] = stream::exp2_pair(make_float2(__uint_as_float(v.r[2 * k]), __uint_as_float(v.r[2 * k + 1])), sc, nm);
        ta = fadd2(e[0], e[2]);
        tb = fadd2(e[1], e[3]);
    } else {
        float2 e[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if ((kF >= 1 && k == 0) || (kF >= 2 && k == 4)) {
                const uint32_t w = bf16x2_min_nan(bf16x2_max_nan(v.r[k], ref.floor2), ref.ceil2);
                e[k] = exp2_fma_pair_inrange(ffma2(make_float2(bf16_lo(w), bf16_hi(w)), sc, nm));
            } else {
                e[k] = stream::exp2_pair(make_float2(bf16_lo(v.r[k]), bf16_hi(v.r[k])), sc, nm);
            }
        }
        ta = fadd2(fadd2(e[0], e[2]), fadd2(e[4], e[6]));
        tb = fadd2(fadd2(e[1], e[3]), fadd2(e[5], e[7]));
    }
    Sa = fadd2(Sa, ta);
    Sb = fadd2(Sb, tb);
}

// A span whose sums left fp32's range, or whose first block holds no logit to refer to (masked
// logits, NaN, +inf, a magnitude beyond 4096), read again with a running maximum per lane: one pass
// in the same 32-byte units.  Masked vocabularies come here, a prefix of 1 KB is enough, so it must
// not cost much more than the fast pass.  (One element a lane and step, and a pass of its own for
// the maximum, took 800 us for 16,000 rows of 98 KB with a masked first half that take 273 unmasked;
// this takes 337, the ring 343 to 417.)
struct SpanResult {
    float m, S, vmax;
    int vidx;
};
// It takes what it needs by value: with the address of the kernel's parameters taken, every thread of
// the kernel began by copying them to local memory (the call on 5,568 rows of 24 KB: 32.3 us, now
// 29.6; the greedy step on 1,024 rows of 304 KB: 54.9, now 51.7).
// (kCaller: a copy for each kernel.  ptxas 12.9 crashes on one called by a kernel with cluster barriers
// and by another.)
template <typename T, bool kArg, int kCaller>
__device__ __noinline__ SpanResult span_running_max(const char *x, int row_bytes, Cut cut, int sp, int lane) {
    constexpr int ES = Elem<T>::kBytes;
    constexpr float kLowest = -3.402823466e38f;      // finite, so that x - m is -inf or 0 for a masked x
    const ranges::RowUnits ru = ranges::row_units(reinterpret_cast<uintptr_t>(x), row_bytes);
    const ranges::UnitSpan us = ranges::unit_span(ru, cut.spans, sp, cut.blocks);
    int rest = us.uhi - us.ulo - lane * 32;
    const char *at = x + us.ulo + lane * 32;
    const int e = lane < 16 ? us.lo + lane * ES : us.uhi + (lane - 16) * ES;
    float edge = -INFINITY;
    if (e < (lane < 16 ? us.ulo : us.hi)) edge = Elem<T>::load(x + e);
    // (x - m) * log2e throughout, not x * log2e - m * log2e: a mask of the type's lowest value would
    // leave fp32's range there
    float m = fmaxf(edge, kLowest), S = ex2((edge - m) * kLog2e), total = 0.f, vmax = -INFINITY;
    int blk = 0, vblk = 0;
    auto add = [&](const Unit &d) {
        const float um = unit_max<T>(d);
        if (kArg && um > vmax) { vmax = um; vblk = blk; }
        if (um > m) {
            const float sc = ex2((m - um) * kLog2e);
            S *= sc;
            total *= sc;
            m = um;
        }
        const float2 nm = make_float2(-m, -m), sc = make_float2(kLog2e, kLog2e);
        float2 t = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            float2 a[2];
            if (ES == 4) {
                a[0] = make_float2(__uint_as_float(d.r[k]), __uint_as_float(d.r[k + 1]));
                a[0] = fmul2(fadd2(a[0], nm), sc);
                t = fadd2(t, make_float2(ex2(a[0].x), ex2(a[0].y)));
            } else {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    a[q] = fmul2(fadd2(make_float2(bf16_lo(d.r[k + q]), bf16_hi(d.r[k + q])), nm), sc);
                    a[q] = make_float2(ex2(a[q].x), ex2(a[q].y));
                }
                t = fadd2(t, fadd2(a[0], a[1]));
            }
        }
        S += t.x + t.y;
        if (++blk % kGroupBlocks == 0) { total += S; S = 0.f; }
    };
#pragma unroll 1
    for (; rest > 0; rest -= kDirectBlockBytes, at += kDirectBlockBytes) add(load_unit(at));
    SpanResult r;
    r.m = warp_max(m);
    r.S = warp_sum((S + total) * ex2((m - r.m) * kLog2e));
    r.vmax = -INFINITY;
    r.vidx = INT_MAX;
    if (kArg) {
        r.vmax = warp_max(fmaxf(vmax, edge));
        int idx = INT_MAX;
        if (edge == r.vmax && edge > -INFINITY) idx = e / ES;
        if (vmax == r.vmax && vmax > -INFINITY)
            idx = min(idx, us.ulo / ES + lane * (32 / ES) + vblk * (kDirectBlockBytes / ES));
        r.vidx = __reduce_min_sync(0xffffffffu, idx);
    }
    return r;
}

inline int row_blocks(int64_t row_bytes) {
    const int64_t nb = (row_bytes + kDirectBlockBytes - 1) / kDirectBlockBytes;
    return nb > 0 ? (int)nb : 1;
}

// Where a warp is in the rows it has to read.  With `skip`, the rows of utterances that are not
// read are left out of the count (act: rows to read before utterance b), so that the others are
// dealt out evenly whatever is skipped; with more utterances or rows than the table takes
// (table_fits), skipped rows are passed over one by one.
struct Cursor {
    int a;             // index among the rows to read
    int sp, b;
    int shift;         // row - a, for the rows of utterance b
    int row;
    bool valid;
};

// Which spans a warp takes: number gw, gw + GW, ... of rows * spans.  Row index a stands for
// row first + a * stride of those to read: of the table's, or of the matrix (then, unless `all`, rows
// of skipped utterances are passed over).
struct Deal {
    unsigned gw, GW;
    int rows, first, stride;
    bool table, all;
};

// Streams the spans dealt to this warp and hands each one's result to emit(row, a, span, result),
// called by all lanes.  opened() is called once, when the first block is on its way.
template <typename T, int kF, bool kArg, int kCaller, typename Opened, typename Emit>
__device__ __forceinline__ void stream_spans(const DirectParams &p, const Cut cut, const Deal deal,
                                             const int32_t *act, Opened opened, Emit emit) {
    constexpr int ES = Elem<T>::kBytes;
    const int lane = threadIdx.x & 31;
    const unsigned ns = (unsigned)cut.spans;
    const int da = (int)(deal.GW / ns), ds = (int)(deal.GW % ns);
    Cursor cur;
    cur.a = (int)(deal.gw / ns);
    cur.sp = (int)(deal.gw % ns);
    cur.b = -1;
    cur.shift = 0;
    int b_end = 0;                       // rows to read up to and with utterance b
    auto step = [&]() {
        cur.a += da; cur.sp += ds;
        if (cur.sp >= cut.spans) { cur.sp -= cut.spans; ++cur.a; }
    };
    auto settle = [&]() {
        if (deal.table) {
            cur.valid = cur.a < deal.rows;
            const int at = deal.first + cur.a * deal.stride;
            if (cur.valid && at >= b_end) {
                b_end = act[++cur.b + 1];
                if (b_end <= at) {               // not the next one: short drafts
                    cur.b = stream::utterance_of_count(act, p.B, at);
                    b_end = act[cur.b + 1];
                }
                cur.shift = (int)p.tok_off[cur.b] - act[cur.b];
            }
            cur.row = at + cur.shift;
            return;
        }
        for (;;) {
            cur.valid = cur.a < deal.rows;
            cur.row = deal.first + cur.a * deal.stride;
            if (!cur.valid || deal.all) return;
            const int b = utterance_of_row(p.tok_off, p.B, cur.row);
            if (b < 0 || !p.skip[b]) return;
            step();
        }
    };
    settle();
    if (!cur.valid) { opened(); return; }

    // the span the cursor stands on: this lane's address in its first block, blocks, bytes of
    // the last block from this lane's unit on, the element this lane has of the row's two edges
    const char *at;
    int blocks, rest, edge_idx = 0, unit_elem = 0;
    float edge;
    auto open = [&]() {
        const char *x = p.logits + (int64_t)cur.row * p.row_pitch;
        const ranges::RowUnits ru = ranges::row_units(reinterpret_cast<uintptr_t>(x), p.row_bytes);
        const ranges::UnitSpan us = ranges::unit_span(ru, cut.spans, cur.sp, cut.blocks);
        const int bytes = us.uhi - us.ulo;
        at = x + us.ulo + lane * 32;
        blocks = (bytes + kDirectBlockBytes - 1) / kDirectBlockBytes;
        if (blocks < 1) blocks = 1;
        rest = bytes - (blocks - 1) * kDirectBlockBytes - lane * 32;
        const int e = lane < 16 ? us.lo + lane * ES : us.uhi + (lane - 16) * ES;
        edge = -INFINITY;
        if (e < (lane < 16 ? us.ulo : us.hi)) edge = Elem<T>::load(x + e);
        if (kArg) {
            edge_idx = e / ES;
            unit_elem = us.ulo / ES + lane * (32 / ES);
        }
    };
    auto load_next = [&](Unit &d) { d = load_unit(at); at += kDirectBlockBytes; };
    auto load_last = [&](Unit &d) {
#pragma unroll
        for (int k = 0; k < 8; ++k) d.r[k] = Elem<T>::kNegInfBits;
        if (rest > 0) d = load_unit(at);
    };

    auto begin = [&](Unit &d) {
        open();
        if (blocks > 1) load_next(d); else load_last(d);
    };

    Unit u, v;
    begin(u);
    opened();
    for (;;) {
        Reference ref;
        const int row = cur.row, a = cur.a, sp = cur.sp;
        const float my_edge = edge;
        const int my_edge_idx = edge_idx, my_unit_elem = unit_elem;
        float vmax = -INFINITY, Sw = 0.f, total = 0.f;
        int vblk = 0;
        float2 Sa = make_float2(0.f, 0.f), Sb = Sa;
        ref.set<T>(warp_max(fmaxf(unit_max<T>(u), my_edge)));
        bool fast = fabsf(ref.m) < 4096.f;
        int left = fast ? blocks - 1 : 0;   // blocks that follow the one in u
        auto add = [&](const Unit &d, int blk) {
            if (kArg) {
                const float m = unit_max<T>(d);
                if (m > vmax) { vmax = m; vblk = blk; }
            }
            add_unit<T, kF>(d, ref, Sa, Sb);
        };
        while (left > 2) {
            const int stop = max(2, left - kGroupBlocks);
#pragma unroll 1
            for (; left > stop; left -= 2) {
                load_next(v);
                add(u, blocks - 1 - left);
                load_next(u);
                add(v, blocks - left);
            }
            total += (Sa.x + Sa.y) + (Sb.x + Sb.y);
            Sa = Sb = make_float2(0.f, 0.f);
        }
        if (left == 2) {
            load_next(v);
            add(u, blocks - 3);
            load_last(u);
            add(v, blocks - 2);
        } else if (left == 1) {
            load_last(v);
            add(u, blocks - 2);
            u = v;
        }
        const int last = blocks - 1;
        // the next span's first block is on its way before this span is finished
        step();
        settle();
        if (cur.valid) begin(v);
        if (fast) {
            add(u, last);
            Sw = warp_sum(total + ((Sa.x + Sa.y) + (Sb.x + Sb.y) + ex2(fmaf(my_edge, kLog2e, ref.nmh))));
            fast = Sw < kSpanSumLimit;
            Sw *= ex2(-fmaf(ref.m, kLog2e, ref.nmh));   // every exponent carried m*log2e + nmh
        }
        SpanResult out;
        if (fast) {
            out.m = ref.m;
            out.S = Sw;
            if (kArg) {
                // a lane's maximum is known to a unit: its first element stands for it, and
                // whoever closes the row looks the position up
                out.vmax = warp_max(fmaxf(vmax, my_edge));
                int idx = INT_MAX;
                if (my_edge == out.vmax && my_edge > -INFINITY) idx = my_edge_idx;
                if (vmax == out.vmax && vmax > -INFINITY)
                    idx = min(idx, my_unit_elem + vblk * (kDirectBlockBytes / ES));
                out.vidx = __reduce_min_sync(0xffffffffu, idx);
            }
        } else {
            out = span_running_max<T, kArg, kCaller>(p.logits + (int64_t)row * p.row_pitch, p.row_bytes, cut, sp, lane);
        }
        emit(row, a, sp, out);
        if (!cur.valid) return;
        u = v;
    }
}

template <typename T, int kF, bool kArg>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) verify_rows_direct(const DirectParams p) {
    extern __shared__ int32_t act[];
    __shared__ int32_t warp_tot[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool table = !kArg && p.table != 0;      // a greedy step reads all rows
    pdl_wait();
    pdl_launch_dependents();
    int rows = (int)p.M;
    Cut cut = p.cut[0];
    if (table) {
        rows = stream::count_rows(p.tok_off, p.skip, p.B, p.M, act, warp_tot, kWarps, nullptr);
#pragma unroll
        for (int q = 1; q < kCuts; ++q)
            if (rows <= (int)(p.M >> q)) cut = p.cut[q];
    }
    // counted so that neighbours go to different CTAs
    const Deal deal{blockIdx.x + gridDim.x * warp, gridDim.x * kWarps, rows, 0, 1, table, kArg || p.skip == nullptr};
    stream_spans<T, kF, kArg, 0>(p, cut, deal, act, [] {}, [&](int row, int, int sp, const SpanResult &out) {
        if (kArg) {
            if (lane == 0) reinterpret_cast<float4 *>(p.partials)[(int64_t)row * p.pairs + sp] =
                make_float4(out.m, out.S, out.vmax, __int_as_float(out.vidx));
        } else {
            // pairs that this cut has no span for add nothing
            const int at = sp + lane * cut.spans;
            if (at < p.pairs) reinterpret_cast<float2 *>(p.partials)[(int64_t)row * p.pairs + at] =
                lane == 0 ? make_float2(out.m, out.S) : make_float2(kNegInit, 0.f);
        }
    });
}

inline bool table_fits(int B, int64_t M) {
    // a malformed list of offsets may name a row more than once: B * M bounds the count
    return B + 1 <= stream::kOffCacheMax && (B + 1) * M < (1ll << 31);
}

// Column spans per row.  All warps of the grid get the same number of spans (plus or minus one),
// so the time goes with the number of rounds times the blocks of a span, and a span costs about
// three blocks' worth of instructions of its own (reference, merge, the next span's addresses).
// (A finer cut of the rows that do not fill a round, so that every warp gets the same bytes, was
// slower throughout: 22.4 against 21.1 us on 250 rows of 304 KB, 95 against 93.5 on 5,568 of 98.)
// Spans that all begin at one offset of 64 KB keep the warps, which go through them in step, on the same
// few memory channels: they count an eighth more (fp32 behind a gate, us, by spans of 64 KB, of 32 and by the
// ring: 1,500 rows of 192 KB 56.5, 48.2, 49.6; 750 of 384 KB 56.4, 48.3, 51.8; 1,500 of 195 KB do not
// mind: 49.6, 49.7, 50.6).
inline Cut plan_spans(int64_t M, int64_t row_bytes, int warps, int most) {
    const int64_t nb = row_blocks(row_bytes);
    int64_t best = 0;
    Cut cut{1, (int)nb};
    for (int rounds = 1; rounds <= 16; ++rounds) {
        int64_t ns = M > 0 ? (int64_t)rounds * warps / M : 1;
        ns = ns < 1 ? 1 : ns > most ? most : ns;
        const int64_t bps = (nb + ns - 1) / ns;
        ns = (nb + bps - 1) / bps;
        int64_t cost = (M * ns + warps - 1) / warps * (bps + 3);
        if (bps % 64 == 0 && row_bytes % 65536 == 0) cost += cost / 8;
        if (best == 0 || cost < best) { best = cost; cut = Cut{(int)ns, (int)bps}; }
        if (M > 0 && (int64_t)rounds * warps / M >= most) break;
    }
    return cut;
}

// With `skip` only the kernel knows how many rows are read, and the cut for all of a batch's rows leaves
// most warps without a span where few are.  So such a batch has a cut for every halving of its rows, and
// the kernel takes the one for what its table counted.  One cut, cuts, and the ring for comparison,
// us: bf16, 43,000 rows of 200 KB of which 330 are read 58.5, 21.1, 22.4; 46,000 of 304 KB, 990: 117, 66.7,
// 72.0; 30,000 of 98 KB, 2,800: 62.4, 50.4, 53.0; all 43,000: 1,276, 1,270, 1,361; fp32, 500 of 608 KB, 50:
// 24.9, 15.0, 20.0; 590 of 400 KB, 60: 19.0, 10.6, 14.5.  The finer cuts have up to eight spans, which the
// closing kernel takes in a lane or two; calls of few rows, whose cut for all of them has more, up to 32.
// (pairs > spans of a cut only here.)
inline void plan_cuts(int64_t M, int64_t row_bytes, int warps, int most, bool may_skip, Cut *cut, int *pairs) {
    cut[0] = plan_spans(M, row_bytes, warps, most);
    *pairs = cut[0].spans;
    const int finest = 8 * M < warps ? 32 : 8, fine = most < finest ? most : finest;
    for (int k = 1; k < kCuts; ++k) {
        cut[k] = may_skip ? plan_spans(M >> k, row_bytes, warps, fine) : cut[0];
        if (M < warps && cut[k].spans < cut[k - 1].spans) cut[k] = cut[k - 1];     // fewer by `fine` alone
        if (cut[k].spans > *pairs) *pairs = cut[k].spans;
    }
}

}  // namespace direct
}  // namespace ssd
