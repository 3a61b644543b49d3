// Stage 2 kernels: vocabulary-wide log-sum-exp of the LLM logits at the draft positions, the
// draft token's log-likelihood (Eq. 5), and the first rejected position (Section 2.3).
//
// The LLM logits [M, V] are read once by a streaming kernel that leaves, for every row, a few
// partial (max, sum-of-exponentials) pairs in the workspace; a small per-utterance kernel merges
// them, gathers x[i, draft_i], applies the acceptance rule and finds the first reject.
//
//   verify_rows_tma    persistent CTAs; warp 0 is the producer: it walks this CTA's work items
//                      (a row, or a column span of a row), and feeds a ring of shared-memory
//                      stages with 1-D bulk asynchronous copies (TMA) signalled through
//                      mbarriers.  The other warps consume: each thread keeps a sum of
//                      2^((x-m)*log2e) relative to a reference logit m of its own and checks
//                      once per stage that the sum stayed in range (see Online), so the common
//                      case is one exponential and no comparison per logit.
//   verify_rows_direct (ssd_direct.cuh) a warp per column span of a row, 32-byte loads into
//                      registers; what runs by default where it is faster (see use_direct).
//   verify_rows_plain  one CTA per item with scalar global loads; any alignment.  Fallback.
//
// The same streaming kernels with a running arg max serve the greedy decoding step (Eq. 6),
// and with a closing kernel that leaves (maximum, sum, draft logit) per row instead of the
// decision they serve an LLM head whose columns are split over several ranks (ssd_verify_shard,
// ssd_verify_combine).
#include <limits.h>
#include <math.h>

#include "ssd_common.cuh"
#include "ssd_direct.cuh"
#include "ssd_ranges.cuh"
#include "ssd_stream.cuh"
#include "ssd_whole.cuh"

namespace ssd {


namespace {

using namespace stream;

struct VerifyParams {
    const char *logits;
    int V;
    int64_t ld;
    int64_t M;
    int split;
    int64_t num_items;
    const int64_t *tok_off;
    int B;
    const uint8_t *skip;
    int table;            // count the rows to read per utterance in shared memory first
    float2 *partials;
    int partials_per_row;
    int warps;            // consumer warps
    int stages;
    int stage_bytes;
    unsigned long long *err_word;
    unsigned long long epoch;
};

// Up to so many utterances the ring's producing warp counts by itself, after a rehearsal while the kernel
// before still runs; beyond, all warps do (one warp's 128 at a time were a round trip each: 2,000 rows of 98
// KB, none skipped, of 500 utterances 44.3 us, of 2,000 67.5; 43.1 and 58.9 now; of 56 38.3 and 37.8).
// All warps through a rehearsal: 0.5 us less where rows are read, but 2 us more where all are skipped.
constexpr int kCountedByWarp = 128;

template <typename T, int kF, bool kArg>
__global__ void __launch_bounds__(544, 1) verify_rows_tma(const VerifyParams p) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int ES = Elem<T>::kBytes, EPC = Elem<T>::kPerChunk;
    // the greedy step's closing kernel reads nothing ahead of its own wait
    if (kArg) pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int S = p.stages, CW = p.warps;
    // layout: full[S] | empty[S] | desc[S] | rows to read before each utterance and what takes the
    // count of such rows to a row of the matrix | stages
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t full0 = sbase, empty0 = sbase + S * 8;
    StageDesc *desc = reinterpret_cast<StageDesc *>(smem + 2 * S * 8);
    const bool table = p.table != 0;
    int32_t *act = reinterpret_cast<int32_t *>(smem + 2 * S * 8 + S * sizeof(StageDesc));
    int32_t *shift = act + (table ? p.B + 1 : 0);
    const uint32_t hdr = (uint32_t)((2 * S * 8 + S * sizeof(StageDesc) +
                                     (table ? (size_t)(p.B + 1) * 8 : 0) + 127) & ~(size_t)127);
    const uint32_t stage0 = sbase + hdr;
    unsigned char *stage0_ptr = smem + hdr;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full0 + s * 8, 1); mbar_init(empty0 + s * 8, CW); }
        mbar_init_fence();
    }
    __syncthreads();             // the barriers are there
    int to_read = 0;
    if (table && p.B <= kCountedByWarp && warp == 0) {
#pragma unroll 1
        for (int real = 0; real < 2; ++real) {
            if (real) {
                pdl_wait();
                if (!kArg) pdl_launch_dependents();
            }
            to_read = count_rows_by_warp(p.tok_off, p.skip, p.B, p.M, act, shift, !real);
        }
    } else {
        pdl_wait();
        if (!kArg) pdl_launch_dependents();
        if (table && p.B > kCountedByWarp)     // (the stages are empty yet: the warps' counts pass through the first)
            to_read = count_rows(p.tok_off, p.skip, p.B, p.M, act, reinterpret_cast<int32_t *>(stage0_ptr),
                                 blockDim.x >> 5, shift);
    }

    const int64_t row_bytes = (int64_t)p.V * ES;
    if (warp == 0) {
        // =============================== producer ===============================
        // With skip flags only rows that are read are dealt out (with more utterances or rows than
        // the table takes, skipped ones are passed over instead): a batch of which nothing is read
        // costs a CTA its look at the flags.
        const int64_t num_items = table ? (int64_t)to_read * p.split : p.num_items;
        int s = 0;                  // stage to fill next, and the phase of its barriers
        uint32_t ph = 0;
        bool failed = false;
        const int max_chunks = p.stage_bytes >> 4;
        for (int64_t k0 = 0; !failed; k0 += 32) {
            const int64_t first = (int64_t)blockIdx.x + k0 * gridDim.x;
            if (first >= num_items) break;
            const int64_t mine = first + (int64_t)lane * gridDim.x;
            int64_t my_row = mine / p.split;
            const int my_span = (int)(mine - my_row * p.split);
            bool active = mine < num_items;
            if (active && table) {
                my_row += shift[utterance_of_count(act, p.B, (int)my_row)];
            } else if (active && p.skip) {
                const int b = utterance_of_row(p.tok_off, p.B, my_row);
                active = !(b >= 0 && p.skip[b]);
            }
            unsigned todo = __ballot_sync(0xffffffffu, active);
            while (todo && !failed) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1;
                const int64_t row = __shfl_sync(0xffffffffu, my_row, src);
                const int sp = __shfl_sync(0xffffffffu, my_span, src);
                const ranges::RowGeom geom = ranges::row_geom(
                    reinterpret_cast<uintptr_t>(p.logits), row, p.ld * ES, row_bytes);
                const uintptr_t g0 = geom.g0, g1 = geom.g1, f0 = geom.f0;
                const ranges::SpanCut cut = ranges::span_cut(geom.row_chunks, p.split, sp, max_chunks);
                const int sc1 = cut.sc1, parts = cut.parts, per_part = cut.per_part;
                const int64_t slot = row * p.partials_per_row + (int64_t)sp * CW;
                for (int part = 0; part < parts; ++part) {
                    if (!mbar_wait_bounded(empty0 + s * 8, ph ^ 1u)) { failed = true; break; }
                    const int pc0 = cut.sc0 + part * per_part;
                    const int pc1 = min(sc1, pc0 + per_part);
                    // chunks that are only partly inside the row (row start / end not on a
                    // 16-byte boundary) are filled here with plain loads and -inf padding; the
                    // bulk copy takes the fully valid chunks only, so it never leaves the row.
                    const ranges::PartReads pr = ranges::part_reads(geom, pc0, pc1);
                    const int b0 = pr.b0, b1 = pr.b1;
                    unsigned char *dst = stage0_ptr + (size_t)s * p.stage_bytes;
                    if (pr.head_plain) {
                        if (lane < EPC) {
                            const uintptr_t a = f0 + (uintptr_t)lane * ES;
                            const bool ok = a >= g0 && a < g1;
                            if (ES == 4) reinterpret_cast<uint32_t *>(dst)[lane] =
                                ok ? *reinterpret_cast<const uint32_t *>(a) : 0xff800000u;
                            else reinterpret_cast<uint16_t *>(dst)[lane] =
                                ok ? *reinterpret_cast<const uint16_t *>(a) : (uint16_t)0xff80u;
                        }
                    }
                    if (pr.tail_plain) {
                        if (lane < EPC) {
                            const uintptr_t a = f0 + (uintptr_t)(pc1 - 1) * 16 + (uintptr_t)lane * ES;
                            const bool ok = a >= g0 && a < g1;
                            unsigned char *d = dst + (size_t)(pc1 - 1 - pc0) * 16;
                            if (ES == 4) reinterpret_cast<uint32_t *>(d)[lane] =
                                ok ? *reinterpret_cast<const uint32_t *>(a) : 0xff800000u;
                            else reinterpret_cast<uint16_t *>(d)[lane] =
                                ok ? *reinterpret_cast<const uint16_t *>(a) : (uint16_t)0xff80u;
                        }
                    }
                    __syncwarp();
                    if (lane == 0) {
                        desc[s].nchunks = pc1 - pc0;
                        desc[s].flags = (part == parts - 1) ? kFlagLast : 0u;
                        desc[s].slot = slot;
                        desc[s].elem0 = (int32_t)(((int64_t)pc0 * 16 - (int64_t)(g0 - f0)) / ES);
                        const uint32_t bar = full0 + s * 8;
                        if (b1 > b0) {
                            const uint32_t bytes = (uint32_t)(b1 - b0) << 4;
                            fence_proxy_async();
                            mbar_arrive_expect_tx(bar, bytes);
                            bulk_g2s(stage0 + (uint32_t)s * p.stage_bytes + ((uint32_t)(b0 - pc0) << 4),
                                     reinterpret_cast<const void *>(f0 + ((uintptr_t)b0 << 4)),
                                     bytes, bar);
                        } else {
                            mbar_arrive(bar);
                        }
                    }
                    __syncwarp();
                    if (++s == S) { s = 0; ph ^= 1u; }
                }
            }
        }
        if (!failed) {
            if (mbar_wait_bounded(empty0 + s * 8, ph ^ 1u)) {
                if (lane == 0) {
                    desc[s].nchunks = 0; desc[s].flags = kFlagEnd; desc[s].slot = 0;
                    mbar_arrive(full0 + s * 8);
                }
            } else {
                failed = true;
            }
        }
        if (failed) {
            if (lane == 0) atomicExch(p.err_word, p.epoch);
            drain_after_error();
        }
    } else {
        // =============================== consumers ===============================
        const int cw = warp - 1;
        const int ct = cw * 32 + lane, NT = CW * 32;
        Online st;
        st.reset();
        ArgTrack at;
        at.reset();
        bool failed = false;
        int s = 0;
        uint32_t ph = 0;
        for (;;) {
            if (!mbar_wait_bounded(full0 + s * 8, ph)) { failed = true; break; }
            const int n = desc[s].nchunks;
            const uint32_t flags = desc[s].flags;
            if (flags & kFlagEnd) break;
            consume_stage<T, kF, kArg>(stage0 + (uint32_t)s * p.stage_bytes, n, ct, NT, st,
                                       kArg ? desc[s].elem0 : 0, at);
            int64_t slot = 0;
            if (flags & kFlagLast) slot = desc[s].slot;
            __syncwarp();
            if (lane == 0) mbar_arrive(empty0 + s * 8);
            if (flags & kFlagLast) {
                const float2 r = warp_merge<kArg>(st);
                if (kArg) {
                    // warp arg max: largest value, lowest index among the lanes that hold it
                    const float vm = warp_max(at.vmax);
                    const int vi = __reduce_min_sync(0xffffffffu, at.vmax == vm ? at.vidx : INT_MAX);
                    if (lane == 0)
                        reinterpret_cast<float4 *>(p.partials)[slot + cw] =
                            make_float4(r.x, r.y, vm, __int_as_float(vi));
                    at.reset();
                } else {
                    if (lane == 0) p.partials[slot + cw] = r;
                }
                st.reset();
            }
            if (++s == S) { s = 0; ph ^= 1u; }
        }
        if (failed) {
            if (lane == 0) atomicExch(p.err_word, p.epoch);
            drain_after_error();
        }
    }
}


// Merge of a row's P (reference, sum) pairs into (maximum, sum relative to it) by the G lanes of
// a group, lane `sub` of which takes pairs sub, sub + G, ..., L of them in one round trip.  All 32
// lanes of the warp call it.
template <int G, int L> __device__ __forceinline__ float2 merge_partials(const float2 *pp, int P, int sub) {
    float Mx = kNegInit, S = 0.f;
    if (P <= L * G) {
        float2 v[L];          // all of a lane's pairs are fetched together
#pragma unroll
        for (int j = 0; j < L; ++j) {
            v[j] = make_float2(kNegInit, 0.f);
            if (sub + j * G < P) v[j] = pp[sub + j * G];
        }
#pragma unroll
        for (int j = 0; j < L; ++j) Mx = fmaxf(Mx, v[j].x);
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) Mx = fmaxf(Mx, __shfl_xor_sync(0xffffffffu, Mx, o));
#pragma unroll
        for (int j = 0; j < L; ++j) S += v[j].y * ex2((v[j].x - Mx) * kLog2e);
    } else {
        for (int q = sub; q < P; q += G) Mx = fmaxf(Mx, pp[q].x);
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) Mx = fmaxf(Mx, __shfl_xor_sync(0xffffffffu, Mx, o));
        for (int q = sub; q < P; q += G) {
            const float2 v = pp[q];
            S += v.y * ex2((v.x - Mx) * kLog2e);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
    return make_float2(Mx, S);
}

// Eq. 5 for one row, given its maximum Mx, ln of its sum of exponentials relative to Mx and the
// draft token's logit x: the log-likelihood, whether the position is rejected (p <= tau; NaN
// rejects; tau <= 0 rejects nothing, tau >= 1 everything), and the status bits the row raises.
struct RowDecision {
    float logp, lse;
    bool reject;
    uint32_t flags;
};
__device__ __forceinline__ RowDecision decide_row(float x, float Mx, float lnS, bool id_ok,
                                                  float log_tau, int reject_none, int reject_all) {
    RowDecision d;
    d.lse = Mx + lnS;
    d.flags = fabsf(d.lse) < INFINITY ? 0u : (uint32_t)SSD_UTT_NONFINITE;
    if (!id_ok) {
        d.flags |= SSD_UTT_BAD_DRAFT_ID;
        d.logp = -INFINITY;
        d.reject = true;
    } else {
        d.logp = row_logp(x, Mx, lnS);
        d.reject = reject_none ? false : (reject_all || !(d.logp > log_tau));
    }
    return d;
}

// ---- verification finished inside the streaming kernel ----------------------------------------
// The same ring of stages as verify_rows_tma, for whole rows (no column spans).  The consumer
// warps leave a row's (reference, sum) pairs in shared memory instead of the workspace; the
// producer warp, when it next takes over the stage that held the row's last part and has the
// stage's next copy under way, merges them, adds the draft token's logit (which it fetched,
// with the draft id, one batch of rows ahead), writes the row's log-likelihood (Eq. 5) and, for
// a rejected position, lowers the utterance's first-reject word in the workspace.  The CTA that
// finishes last turns those words into accepted_len / all_accepted / utt_status (Section 2.3).
// The words are {epoch : 32 | value : 32}: nothing has to be cleared between calls.
struct FinParams {
    VerifyParams v;
    const int32_t *draft_ids;
    float log_tau;
    int reject_none, reject_all;
    float *token_logp, *row_lse;
    int32_t *accepted_len;
    uint8_t *all_accepted;
    uint32_t *utt_status;
    unsigned long long *utt_words;     // [2 * B]: first rejected position, status bits
    unsigned long long *done_ctas;
    uint32_t epoch32;
};

struct FinRow {
    int64_t row;
    int32_t b, pos, id_ok;
    float x;
};

__device__ __forceinline__ void utterance_outputs(int b, int64_t i0, int64_t i1, int64_t M,
                                                  bool skipped, int first, uint32_t flags,
                                                  uint32_t internal, int32_t *accepted_len,
                                                  uint8_t *all_accepted, uint32_t *utt_status) {
    if (i0 < 0 || i1 < i0 || i1 > M) {
        accepted_len[b] = 0; all_accepted[b] = 0;
        utt_status[b] = SSD_UTT_BAD_OFFSETS | internal;
        return;
    }
    const int64_t K64 = i1 - i0;
    const int K = K64 > 0x7fffffff ? 0x7fffffff : (int)K64;
    if (skipped) { accepted_len[b] = K; all_accepted[b] = 1; utt_status[b] = internal; return; }
    first = first < K ? first : K;
    accepted_len[b] = first;
    all_accepted[b] = first == K ? 1 : 0;
    utt_status[b] = flags | internal;
}

template <typename T, int kF>
__global__ void __launch_bounds__(544, 1) verify_rows_fin(const FinParams q) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int ES = Elem<T>::kBytes, EPC = Elem<T>::kPerChunk;
    __shared__ int s_last;
    const VerifyParams &p = q.v;
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int S = p.stages, CW = p.warps, NR = 2 * S;
    // layout: full[S] | empty[S] | desc[S] | rows[NR] | spart[NR*CW] | pending[S] | offsets | stages
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t full0 = sbase, empty0 = sbase + S * 8;
    size_t o = 2 * (size_t)S * 8;
    StageDesc *desc = reinterpret_cast<StageDesc *>(smem + o);     o += S * sizeof(StageDesc);
    FinRow *rows = reinterpret_cast<FinRow *>(smem + o);           o += NR * sizeof(FinRow);
    float2 *spart = reinterpret_cast<float2 *>(smem + o);          o += (size_t)NR * CW * 8;
    int32_t *pending = reinterpret_cast<int32_t *>(smem + o);      o += S * 4;
    o = (o + 7) & ~(size_t)7;
    int64_t *offs = reinterpret_cast<int64_t *>(smem + o);         o += (size_t)(p.B + 1) * 8;
    const uint32_t hdr = (uint32_t)((o + 127) & ~(size_t)127);
    const uint32_t stage0 = sbase + hdr;
    unsigned char *stage0_ptr = smem + hdr;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + s * 8, 1);
            mbar_init(empty0 + s * 8, CW);
            pending[s] = 0;
        }
        mbar_init_fence();
        s_last = 0;
    }
    pdl_wait();
    for (int i = threadIdx.x; i <= p.B; i += blockDim.x) offs[i] = p.tok_off[i];
    __syncthreads();

    const int64_t row_bytes = (int64_t)p.V * ES;
    bool failed = false;

    if (warp == 0) {
        // =============================== producer ===============================
        int s = 0;
        uint32_t ph = 0;
        int rowseq = 0;
        bool ok = true;
        const int max_chunks = p.stage_bytes >> 4;

        auto finalize = [&](int slot1) {
            if (slot1 == 0) return;
            const int slot = slot1 - 1;
            const float2 v = lane < CW ? spart[slot * CW + lane] : make_float2(kNegInit, 0.f);
            const float Mx = fmaxf(warp_max(v.x), kNegInit);
            const float Ssum = warp_sum(v.y * ex2((v.x - Mx) * kLog2e));
            if (lane == 0) {
                const FinRow rm = rows[slot];
                const RowDecision d = decide_row(rm.x, Mx, logf(Ssum), rm.id_ok != 0, q.log_tau,
                                                 q.reject_none, q.reject_all);
                const float logp = d.logp, lse = d.lse;
                const uint32_t fl = d.flags;
                const bool reject = d.reject;
                q.token_logp[rm.row] = logp;
                if (q.row_lse) q.row_lse[rm.row] = lse;
                if (fl) tagged_or(q.utt_words + 2 * rm.b + 1, q.epoch32, fl, ok);
                if (reject) tagged_min(q.utt_words + 2 * rm.b, q.epoch32, (uint32_t)rm.pos, ok);
            }
            __syncwarp();
        };

        // What a lane knows about its row of a batch of 32 rows (row first + lane * grid): the
        // utterance, the position, the draft id and the draft token's logit.  Loaded one batch
        // ahead, so that nothing here waits for memory.
        struct Mine { int64_t row; int b, pos, id; float x; bool active; };
        auto look_up = [&](int64_t k0) {
            Mine m{0, 0, 0, -1, 0.f, false};
            m.row = (int64_t)blockIdx.x + (k0 + lane) * gridDim.x;
            if (m.row < p.M) {
                m.b = utterance_of_row(offs, p.B, m.row);
                if (m.b >= 0) {
                    const int64_t i0 = offs[m.b], i1 = offs[m.b + 1];
                    m.active = i0 >= 0 && i1 <= p.M && m.row >= i0 && m.row < i1 &&
                               i1 - i0 <= 0x7fffffff && !(p.skip && p.skip[m.b]);
                    if (m.active) {
                        m.pos = (int)(m.row - i0);
                        m.id = q.draft_ids[m.row];
                        if (m.id >= 0 && m.id < p.V)
                            m.x = Elem<T>::load(p.logits + (m.row * p.ld + m.id) * ES);
                    }
                }
            }
            return m;
        };
        Mine next = look_up(0);
        for (int64_t k0 = 0; !failed; k0 += 32) {
            if ((int64_t)blockIdx.x + k0 * gridDim.x >= p.M) break;
            const Mine cur = next;
            next = look_up(k0 + 32);
            unsigned todo = __ballot_sync(0xffffffffu, cur.active);
            while (todo && !failed) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1;
                const int64_t row = __shfl_sync(0xffffffffu, cur.row, src);
                const int rslot = rowseq % NR;
                ++rowseq;
                const ranges::RowGeom geom = ranges::row_geom(
                    reinterpret_cast<uintptr_t>(p.logits), row, p.ld * ES, row_bytes);
                const uintptr_t g0 = geom.g0, g1 = geom.g1, f0 = geom.f0;
                const ranges::SpanCut cut = ranges::span_cut(geom.row_chunks, 1, 0, max_chunks);
                const int parts = cut.parts, per_part = cut.per_part;
                for (int part = 0; part < parts; ++part) {
                    if (!mbar_wait_bounded(empty0 + s * 8, ph ^ 1u)) { failed = true; break; }
                    const int done_slot1 = pending[s];     // the row this stage held last, if any
                    __syncwarp();
                    const int pc0 = part * per_part;
                    const int pc1 = min(geom.row_chunks, pc0 + per_part);
                    const ranges::PartReads pr = ranges::part_reads(geom, pc0, pc1);
                    const int b0 = pr.b0, b1 = pr.b1;
                    unsigned char *dst = stage0_ptr + (size_t)s * p.stage_bytes;
                    if (pr.head_plain) {
                        if (lane < EPC) {
                            const uintptr_t a = f0 + (uintptr_t)lane * ES;
                            const bool in = a >= g0 && a < g1;
                            if (ES == 4) reinterpret_cast<uint32_t *>(dst)[lane] =
                                in ? *reinterpret_cast<const uint32_t *>(a) : 0xff800000u;
                            else reinterpret_cast<uint16_t *>(dst)[lane] =
                                in ? *reinterpret_cast<const uint16_t *>(a) : (uint16_t)0xff80u;
                        }
                    }
                    if (pr.tail_plain) {
                        if (lane < EPC) {
                            const uintptr_t a = f0 + (uintptr_t)(pc1 - 1) * 16 + (uintptr_t)lane * ES;
                            const bool in = a >= g0 && a < g1;
                            unsigned char *d = dst + (size_t)(pc1 - 1 - pc0) * 16;
                            if (ES == 4) reinterpret_cast<uint32_t *>(d)[lane] =
                                in ? *reinterpret_cast<const uint32_t *>(a) : 0xff800000u;
                            else reinterpret_cast<uint16_t *>(d)[lane] =
                                in ? *reinterpret_cast<const uint16_t *>(a) : (uint16_t)0xff80u;
                        }
                    }
                    __syncwarp();
                    if (lane == 0) {
                        const bool last = part == parts - 1;
                        desc[s].nchunks = pc1 - pc0;
                        desc[s].flags = last ? kFlagLast : 0u;
                        desc[s].slot = rslot;
                        desc[s].elem0 = 0;
                        desc[s].gather = -1;
                        pending[s] = last ? rslot + 1 : 0;
                        const uint32_t bar = full0 + s * 8;
                        if (b1 > b0) {
                            const uint32_t bytes = (uint32_t)(b1 - b0) << 4;
                            fence_proxy_async();
                            mbar_arrive_expect_tx(bar, bytes);
                            bulk_g2s(stage0 + (uint32_t)s * p.stage_bytes + ((uint32_t)(b0 - pc0) << 4),
                                     reinterpret_cast<const void *>(f0 + ((uintptr_t)b0 << 4)),
                                     bytes, bar);
                        } else {
                            mbar_arrive(bar);
                        }
                    }
                    __syncwarp();
                    finalize(done_slot1);     // after the stage's next copy is under way
                    if (++s == S) { s = 0; ph ^= 1u; }
                }
                // what the row's finish needs; written after its copies are under way, since the
                // draft id and logit of a kernel's first rows may still be on their way
                if (lane == src) {
                    FinRow rm;
                    rm.row = cur.row; rm.b = cur.b; rm.pos = cur.pos;
                    rm.id_ok = (cur.id >= 0 && cur.id < p.V) ? 1 : 0; rm.x = cur.x;
                    rows[rslot] = rm;
                }
                __syncwarp();
            }
        }
        if (!failed) {
            // end marker into the next stage, then the rows still waiting in the other stages
            if (mbar_wait_bounded(empty0 + s * 8, ph ^ 1u)) {
                finalize(pending[s]);
                if (lane == 0) {
                    desc[s].nchunks = 0; desc[s].flags = kFlagEnd; desc[s].slot = 0; desc[s].gather = -1;
                    mbar_arrive(full0 + s * 8);
                }
                for (int t = 1; t < S && !failed; ++t) {
                    const int st = (s + t) % S;
                    const uint32_t par = st > s ? (ph ^ 1u) : ph;     // filled last round / this round
                    if (mbar_wait_bounded(empty0 + st * 8, par)) finalize(pending[st]);
                    else failed = true;
                }
            } else {
                failed = true;
            }
        }
        if (!__shfl_sync(0xffffffffu, (int)ok, 0)) failed = true;
        if (failed) {
            if (lane == 0) atomicExch(p.err_word, p.epoch);
            drain_after_error();
        }
    } else {
        // =============================== consumers ===============================
        const int cw = warp - 1;
        const int ct = cw * 32 + lane, NT = CW * 32;
        Online st;
        st.reset();
        ArgTrack unused;
        unused.reset();
        int s = 0;
        uint32_t ph = 0;
        for (;;) {
            if (!mbar_wait_bounded(full0 + s * 8, ph)) { failed = true; break; }
            const int n = desc[s].nchunks;
            const uint32_t flags = desc[s].flags;
            if (flags & kFlagEnd) break;
            consume_stage<T, kF, false>(stage0 + (uint32_t)s * p.stage_bytes, n, ct, NT, st, 0, unused);
            if (flags & kFlagLast) {
                const int slot = (int)desc[s].slot;
                const float2 r = warp_merge<false>(st);
                if (lane == 0) spart[slot * CW + cw] = r;
                st.reset();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty0 + s * 8);      // releases the write above as well
            if (++s == S) { s = 0; ph ^= 1u; }
        }
        if (failed) {
            if (lane == 0) atomicExch(p.err_word, p.epoch);
            drain_after_error();
        }
    }

    // ---- the CTA that finishes last writes the per-utterance outputs --------------------------
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        bool ok2 = true;
        const uint32_t before = tagged_add(q.done_ctas, q.epoch32, 1u, ok2);
        s_last = ok2 && before + 1 == gridDim.x;
        if (!ok2) atomicExch(p.err_word, p.epoch);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const uint32_t internal = (__ldcg(p.err_word) == p.epoch) ? (uint32_t)SSD_UTT_INTERNAL : 0u;
    for (int b = threadIdx.x; b < p.B; b += blockDim.x) {
        const unsigned long long w0 = __ldcg(q.utt_words + 2 * b), w1 = __ldcg(q.utt_words + 2 * b + 1);
        const int first = (uint32_t)(w0 >> 32) == q.epoch32 ? (int)min((uint32_t)w0, 0x7fffffffu)
                                                            : 0x7fffffff;
        const uint32_t fl = (uint32_t)(w1 >> 32) == q.epoch32 ? (uint32_t)w1 : 0u;
        utterance_outputs(b, offs[b], offs[b + 1], p.M, p.skip && p.skip[b], first, fl, internal,
                          q.accepted_len, q.all_accepted, q.utt_status);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) verify_rows_plain(const VerifyParams p) {
    constexpr int ES = Elem<T>::kBytes;
    pdl_wait();
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int64_t item = blockIdx.x; item < p.num_items; item += gridDim.x) {
        const int64_t row = item / p.split;
        const int sp = (int)(item - row * p.split);
        if (p.skip) {
            const int b = utterance_of_row(p.tok_off, p.B, row);
            if (b >= 0 && p.skip[b]) continue;
        }
        const int per = (p.V + p.split - 1) / p.split;
        const int v0 = min(p.V, sp * per), v1 = min(p.V, v0 + per);
        const char *rp = p.logits + row * p.ld * ES;
        float m = kNegInit, S = 0.f;
        for (int a = v0 + threadIdx.x; a < v1; a += blockDim.x) {
            const float x = Elem<T>::load(rp + (size_t)a * ES);
            if (x > m) { S = S * expf(m - x) + 1.f; m = x; }
            else S += expf(x - m);
        }
        const float Mw = warp_max(m);
        const float Sw = warp_sum(S * expf(m - Mw));
        if (lane == 0) p.partials[row * p.partials_per_row + (int64_t)sp * nw + warp] =
            make_float2(Mw, Sw);
    }
}

constexpr int kFinishThreads = 1024;   // one sweep for drafts of up to 1024 tokens

template <typename T, int G, int L>
__global__ void __launch_bounds__(kFinishThreads) verify_finish_kernel(
    const char *logits, int V, int64_t ld, int64_t M,
    const int64_t *tok_off, const int32_t *draft_ids, int B,
    float log_tau, int reject_none, int reject_all, const uint8_t *skip,
    const float2 *partials, int P, float *__restrict__ token_logp,
    float *__restrict__ row_lse, int32_t *__restrict__ accepted_len,
    uint8_t *__restrict__ all_accepted, uint32_t *__restrict__ utt_status,
    const unsigned long long *err_word, unsigned long long epoch) {
    constexpr int ES = Elem<T>::kBytes;
    __shared__ int first_reject;
    __shared__ unsigned flags;
    pdl_launch_dependents();
    // The kernel is a chain of dependent memory round trips.  What the caller passed in -- offsets,
    // skip flag, then the first sweep's draft ids, then their logits -- is fetched while the
    // streaming kernel still runs; after it a row waits for its pairs alone.
    const int b = blockIdx.x, tid = threadIdx.x, sub = tid % G;
    if (M == 0) pdl_wait();        // no streaming kernel of this call before this one
    const int64_t i0 = load_input(tok_off + b), i1 = load_input(tok_off + b + 1);
    const bool skipped = skip != nullptr && load_input(skip + b) != 0;
    auto draft_logit = [&](int64_t r, bool &id_ok) {
        const int id = load_input(draft_ids + r);
        id_ok = id >= 0 && id < V;
        return id_ok ? Elem<T>::load_l2(logits + (r * ld + id) * ES) : 0.f;
    };
    float x = 0.f;
    bool id_ok = false;
    const int64_t first = skipped || sub != 0 ? -1 : ranges::row_of_utterance(i0, i1, M, tid / G);
    if (first >= 0) x = draft_logit(first, id_ok);
    pdl_wait();
    const unsigned long long err = *err_word;
    const uint32_t internal = (err == epoch) ? (uint32_t)SSD_UTT_INTERNAL : 0u;
    if (!ranges::rows_sound(i0, i1, M)) {
        if (tid == 0) {
            accepted_len[b] = 0; all_accepted[b] = 0;
            utt_status[b] = SSD_UTT_BAD_OFFSETS | internal;
        }
        return;
    }
    const int64_t K64 = i1 - i0;
    const int K = K64 > 0x7fffffff ? 0x7fffffff : (int)K64;
    if (skipped) {
        if (tid == 0) { accepted_len[b] = K; all_accepted[b] = 1; utt_status[b] = internal; }
        return;
    }
    if (tid == 0) { first_reject = K; flags = 0; }
    __syncthreads();
    unsigned myflags = 0;
    int myfirst = K;
    for (int base = 0; base < K; base += kFinishThreads / G) {
        const int i = base + tid / G;
        const bool mine = i < K;
        const int64_t r = i0 + (mine ? i : 0);
        if (base > 0 && mine && sub == 0) x = draft_logit(r, id_ok);
        const float2 ms = merge_partials<G, L>(partials + r * P, P, sub);
        if (mine && sub == 0) {
            const RowDecision d = decide_row(x, ms.x, logf(ms.y), id_ok, log_tau, reject_none, reject_all);
            myflags |= d.flags;
            token_logp[r] = d.logp;
            if (row_lse) row_lse[r] = d.lse;
            const bool reject = d.reject;
            if (reject && i < myfirst) myfirst = i;
        }
    }
    if (myfirst < K) atomicMin(&first_reject, myfirst);
    if (myflags) atomicOr(&flags, myflags);
    __syncthreads();
    if (tid == 0) {
        accepted_len[b] = first_reject;
        all_accepted[b] = first_reject == K ? 1 : 0;
        utt_status[b] = flags | internal;
    }
}

constexpr uint32_t kStatsInternal = 0x7fc0dead;   // in place of a row's maximum: a wait ran out

// Vocabulary-parallel verification, per rank: for every row of a verified utterance the
// triple (maximum of the local columns, sum of exponentials relative to it, logit of the draft
// token if its column is local, else -inf).  Rows of skipped or malformed utterances are left
// untouched; the combining kernel does not read them.
template <typename T, int G, int L>
__global__ void __launch_bounds__(kFinishThreads) shard_finish_kernel(
    const char *logits, int V_local, int64_t ld, int64_t M, int64_t col0,
    const int64_t *tok_off, const int32_t *draft_ids, int B,
    const uint8_t *skip, const float2 *partials, int P,
    float *__restrict__ stats, const unsigned long long *err_word, unsigned long long epoch) {
    constexpr int ES = Elem<T>::kBytes;
    pdl_launch_dependents();
    // inputs before the wait, as in verify_finish_kernel
    const int b = blockIdx.x, tid = threadIdx.x, sub = tid % G;
    if (M == 0) pdl_wait();        // no streaming kernel of this call before this one
    const int64_t i0 = load_input(tok_off + b), i1 = load_input(tok_off + b + 1);
    const bool skipped = skip != nullptr && load_input(skip + b) != 0;
    const bool sound = ranges::rows_sound(i0, i1, M) && !skipped;
    auto draft_logit = [&](int64_t r) {
        const int64_t local = (int64_t)load_input(draft_ids + r) - col0;
        return local >= 0 && local < V_local ? Elem<T>::load_l2(logits + (r * ld + local) * ES) : -INFINITY;
    };
    float x = -INFINITY;
    const int64_t first = !sound || sub != 0 ? -1 : ranges::row_of_utterance(i0, i1, M, tid / G);
    if (first >= 0) x = draft_logit(first);
    pdl_wait();
    if (!sound) return;
    const bool internal = *err_word == epoch;
    for (int64_t base = i0; base < i1; base += kFinishThreads / G) {
        const bool mine = base + tid / G < i1;
        const int64_t r = mine ? base + tid / G : base;
        if (base > i0 && mine && sub == 0) x = draft_logit(r);
        const float2 ms = merge_partials<G, L>(partials + r * P, P, sub);
        if (mine && sub == 0) {
            stats[3 * r + 0] = internal ? __uint_as_float(kStatsInternal) : ms.x;
            stats[3 * r + 1] = ms.y;
            stats[3 * r + 2] = x;
        }
    }
}

// Vocabulary-parallel verification, after the exchange: stats_all holds R ranks' triples,
// [R, M, 3].  Per row the global maximum, the sum re-based to it, the draft token's logit (the
// one shard that owns the column has it), then Eq. 5 and the first reject exactly as in
// verify_finish_kernel.
__global__ void __launch_bounds__(kFinishThreads) combine_kernel(
    const float *stats_all, int R, int64_t V_total, int64_t M,
    const int64_t *tok_off, const int32_t *draft_ids, int B,
    float log_tau, int reject_none, int reject_all, const uint8_t *skip,
    float *__restrict__ token_logp, float *__restrict__ row_lse,
    int32_t *__restrict__ accepted_len, uint8_t *__restrict__ all_accepted,
    uint32_t *__restrict__ utt_status) {
    __shared__ int first_reject;
    __shared__ unsigned flags;
    pdl_enter();
    const int b = blockIdx.x, tid = threadIdx.x;
    const int64_t i0 = tok_off[b], i1 = tok_off[b + 1];
    const bool skipped = skip != nullptr && skip[b] != 0;
    if (i0 < 0 || i1 < i0 || i1 > M) {
        if (tid == 0) { accepted_len[b] = 0; all_accepted[b] = 0; utt_status[b] = SSD_UTT_BAD_OFFSETS; }
        return;
    }
    const int64_t K64 = i1 - i0;
    const int K = K64 > 0x7fffffff ? 0x7fffffff : (int)K64;
    if (skipped) {
        if (tid == 0) { accepted_len[b] = K; all_accepted[b] = 1; utt_status[b] = 0; }
        return;
    }
    if (tid == 0) { first_reject = K; flags = 0; }
    __syncthreads();
    unsigned myflags = 0;
    int myfirst = K;
    for (int i = tid; i < K; i += blockDim.x) {
        const int64_t r = i0 + i;
        const int id = draft_ids[r];
        const bool id_ok = id >= 0 && (int64_t)id < V_total;
        float Mx = kNegInit, x = -INFINITY;
        for (int q = 0; q < R; ++q) {
            const float *t = stats_all + ((int64_t)q * M + r) * 3;
            const float m = t[0];
            if (__float_as_uint(m) == kStatsInternal) myflags |= SSD_UTT_INTERNAL;
            Mx = fmaxf(Mx, m);
            x = fmaxf(x, t[2]);
        }
        float S = 0.f;
        for (int q = 0; q < R; ++q) {
            const float *t = stats_all + ((int64_t)q * M + r) * 3;
            S += t[1] * ex2((t[0] - Mx) * kLog2e);
        }
        const RowDecision d = decide_row(x, Mx, logf(S), id_ok, log_tau, reject_none, reject_all);
        myflags |= d.flags;
        token_logp[r] = d.logp;
        if (row_lse) row_lse[r] = d.lse;
        const bool reject = d.reject;
        if (reject && i < myfirst) myfirst = i;
    }
    if (myfirst < K) atomicMin(&first_reject, myfirst);
    if (myflags) atomicOr(&flags, myflags);
    __syncthreads();
    if (tid == 0) {
        accepted_len[b] = first_reject;
        all_accepted[b] = first_reject == K ? 1 : 0;
        utt_status[b] = flags;
    }
}

// Greedy step: closes the rows whose partials the streaming kernel left, one warp per row.
constexpr int kGreedyWarps = 8;
template <typename T, bool kUnit>
__global__ void __launch_bounds__(kGreedyWarps * 32) greedy_finish_kernel(
    const char *logits, int V, int64_t ld, int64_t R, const float4 *partials, int P,
    int32_t *__restrict__ next_token, float *__restrict__ next_logp, float *__restrict__ row_lse,
    uint32_t *__restrict__ row_status, const unsigned long long *err_word, unsigned long long epoch) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * kGreedyWarps + (threadIdx.x >> 5);
    if (r >= R) return;
    const float4 *pp = partials + r * P;
    const GreedyRow g = greedy_row<T, kUnit>([&](int q) { return pp[q]; }, P,
                                             logits + r * ld * Elem<T>::kBytes, V, lane);
    if (lane == 0) {
        const uint32_t internal = (*err_word == epoch) ? (uint32_t)SSD_UTT_INTERNAL : 0u;
        next_token[r] = g.token;
        if (next_logp) next_logp[r] = g.logp;
        if (row_lse) row_lse[r] = g.lse;
        if (row_status) row_status[r] = g.status | internal;
    }
}

}  // namespace

unsigned long long next_epoch();

// Whether rows are streamed by the direct-load kernel (it needs no more scratch than the pairs of
// the bulk-copy one).  Not where an option speaks about that one's ring.  Measured, ring against
// direct loads, us on one B200, passes back to back:
//   bf16, rows under 96 KB: direct (5,568 rows of 24 KB: 44.3 / 32.6; 20,000 of 48 KB: 197 / 160;
//     20,000 of 64 KB: 234 / 206).  The ring hands a stage of a whole row from warp to warp.
//   bf16, rows off a 16-byte boundary: direct (5,000 of 98 KB: 97.4 / 88.2; 20,000 of 64 KB:
//     272 / 211).  The ring's producer waits for the ragged ends of every row.
//   bf16, few rows (column spans in the ring): direct (300 of 98 KB: 15.0 / 12.0; 400 of 304 KB:
//     31.1 / 28.6)
//   bf16, aligned rows of 96 KB and more: the ring while the power cap does not bite (1,500 of
//     98 KB: 31.9 / 33.7; 8,000: 136 / 141), direct beyond (12,000: 200 / 200; 16,000: 265 / 245;
//     22,000 of 200 KB: 708 / 664): it spends a fifth fewer instructions on a logit.  With `skip`
//     half of the rows are taken to be read (a batch of 1.3 GB, partly gated: 199 / 206).
//   fp32 with skip flags, as behind a gate, up to 400 MB: direct, all rows read, half and a tenth of them (50
//     of 392 KB, all, 11.7 / 8.8; 300 of 192 KB 16.7 / 14.5, 13.4 / 12.0, 9.9 / 8.7; 590 of 608 KB 57.6 /
//     57.7, 39.8 / 37.6, 20.6 / 15.9; 2,000 of 128 KB 45.2 / 44.2, 29.1 / 28.1, 12.9 / 11.6): the ring cuts few
//     rows into spans of 32 KB and hands each over.  Of 64 sizes from 120 to 400 MB the ring is 4 % slower
//     in the mean, and the better one on some (all of 2,300 of 125 KB 50.3 / 51.6 to 53.5).
//   fp32 without skip flags: the ring (6,000 of 128 KB 117.0 / 118.3, 6,000 of 240 KB 208.8 / 213.0, 16,000 of
//     192 KB 437 / 455), which has more bytes in flight and half the logits per byte; the greedy step
//     on few rows: direct (200 of 196 KB: 14.0 / 12.3; 300 of 608 KB: 36.4 / 35.8; 500 of 196 KB: 21.9 / 23.3)
// The greedy step on bf16 rows: direct (1,024 of 304 KB: 59.5 / 55.1; 24 of 98 KB: 14.0 / 12.6).
static int use_direct(int64_t M, int64_t row_bytes, ssd_dtype dtype, int kernel, int sms,
                      const ssd_launch_opts *o, const RowsAt &at) {
    if (kernel != 2 || row_bytes >= (1ll << 30) || M >= (1ll << 30)) return 0;
    if (o && (o->kernel || o->warps || o->stages || o->stage_bytes || o->fma_exp || o->finish)) return 0;
    const bool few = M < 4ll * sms;
    if (dtype == SSD_F32) return at.greedy ? M <= 2ll * sms : at.skip && M * row_bytes < 400ll << 20;
    if (at.greedy || few || row_bytes < 96 * 1024 || M * row_bytes >= (at.skip ? 2400ll : 1200ll) << 20) return 1;
    return (reinterpret_cast<uintptr_t>(at.base) | (uintptr_t)(at.ld * 2)) % 16 != 0;
}

// How rows are dealt to clusters that close them (rows_whole): column spans, cluster size and number
// of clusters with the fewest block steps of a warp, counted as plan_spans counts them; that number,
// or 0 where a CTA's pairs do not fit.
// (Every call searches: in 32 bits, since rows and row_bytes are below 2^30, and no further than more rounds
// cut finer.  With 64-bit divisions throughout, 1.1 us of host time a call; now 0.2 to 0.6.)
static int64_t plan_whole(int64_t M, int64_t row_bytes, int sms, const RowsAt &at, int B, VerifyPlan *pl) {
    constexpr size_t kMostSmem = 12 * 1024;      // little enough for the L1-heavy split
    constexpr uint32_t kMostSpans = 128;
    const uint32_t nb = (uint32_t)direct::row_blocks(row_bytes), rows = (uint32_t)M;
    const size_t pair = at.greedy ? sizeof(float4) : sizeof(float2), draft = at.greedy ? 0 : sizeof(float2);
    uint64_t best = 0;
    for (int clog = 0; clog <= 3; ++clog) {
        const uint32_t C = 1u << clog, W = C * direct::kWarps;
        // clusters of four and eight CTAs do not fill the GPU's clusters of SMs: 71 of 74 and 33 of 37
        // run at a time, and one more waits for the longest of those (300 rows of 98 KB on 35 clusters
        // of eight: 13.9 us; on 32, 10.0)
        const uint32_t most = (uint32_t)direct::kCtasPerSm * sms / C * (clog == 3 ? 22 : clog == 2 ? 24 : 25) / 25;
        const uint32_t nc = rows < most ? rows : most > 0 ? most : 1;
        const uint32_t q = (rows + nc - 1) / nc;
        for (uint32_t rounds = 1; rounds <= 16; ++rounds) {
            const uint32_t share = rounds * W / q;
            uint32_t ns = share < 1 ? 1 : share > kMostSpans ? kMostSpans : share;
            const uint32_t bps = (nb + ns - 1) / ns;
            ns = (nb + bps - 1) / bps;
            const size_t smem = (size_t)((q + C - 1) / C) * (ns * pair + draft) + (at.skip ? (size_t)(B + 1) * 4 : 0);
            const uint64_t cost = ((uint64_t)q * ns + W - 1) / W * (bps + 3);
            if (smem <= kMostSmem && (best == 0 || cost < best)) {
                best = cost;
                pl->whole_cut = direct::Cut{(int)ns, (int)bps};
                pl->whole_cluster_log2 = clog;
                pl->whole_clusters = (int)nc;
                pl->whole_smem_bytes = smem;
            }
            if (share >= kMostSpans || bps == 1) break;
        }
    }
    return (int64_t)best;
}

// Whether the rows of a greedy step or a shard are closed by the clusters that read them.  Measured,
// us a call, passes back to back on one B200, before (pair kernel or, on fp32, ring, and a closing
// kernel) and after:
//   greedy step, bf16: 1 row of 98 KB 5.3 / 4.0, 24 rows 5.3 / 4.3, 148 7.6 / 6.4, 1,024 21.5 / 19.4;
//     of 304 KB: 24 rows 7.4 / 5.7, 200 14.5 / 14.0, 700 38.2 / 36.8, 1,024 51.3 / 49.6
//   greedy step, fp32, rows of 196 KB: 24 rows 5.9 / 5.4, 300 15.9 / 14.4, 600 25.3 / 21.9, 1,024
//     35.1 / 33.7, 2,000 62.1 / 61.1; 2,000 of 128 KB 43.7 / 45.2: eight rows an SM and more stay
//     with the ring
//   shard, bf16, rows of 24 KB: 250 rows 5.8 / 5.4, 1,500 10.5 / 9.6, 5,352 26.4 / 25.1
//   shard, fp32: 600 rows of 16 KB 9.1 / 5.1, 12,000 75 / 34; 5,352 of 32 KB 37.0 / 30.3, 1,500 of 76
//     KB 23.5 / 20.5; 12,000 of 152 KB 260 / 268: long rows of long batches stay with the ring, as
//     in use_direct, where rows start on 16-byte boundaries (12,000 of 64,004 bytes 138 / 113)
// Whole rows do not always come out even over the clusters.  Where that takes clusters of four and
// more in more than a few rows each, or a third more steps, the pair kernel's finer deal is better (600
// rows of 32 KB 7.7 / 8.7; the greedy step on 74 of 304 KB 9.3 / 9.9); for the greedy step also where the
// steps are more than the second launch is worth (1,500 rows of 98 KB 27.6 / 28.7 and of 304 KB 73.1 / 75.0, 1,800
// of 304 KB 86.1 / 87.7; but a shard's 3,000 rows of 24 KB 16.6 / 15.8).
// With skip flags on a row per warp and more only the kernel knows how many are read, and plan_cuts has
// cuts for that.
static int use_whole(int B, int64_t M, int64_t row_bytes, ssd_dtype dtype, int sms, const ssd_launch_opts *o,
                     const RowsAt &at, VerifyPlan *pl) {
    if (!(at.greedy || at.shard) || M == 0 || pl->kernel != 2 || row_bytes >= (1ll << 30) || M >= (1ll << 30)) return 0;
    if (o && (o->kernel || o->ctas || o->split || o->warps || o->stages || o->stage_bytes || o->fma_exp || o->finish))
        return 0;
    const int warps = direct::kCtasPerSm * sms * direct::kWarps;
    if (at.skip && (M >= warps || !direct::table_fits(B, M))) return 0;
    if (dtype == SSD_F32 && at.greedy && M >= 8ll * sms) return 0;
    if (dtype == SSD_F32 && at.shard && row_bytes >= 72 * 1024 && M * row_bytes >= 300ll << 20 &&
        (reinterpret_cast<uintptr_t>(at.base) | (uintptr_t)(at.ld * 4)) % 16 == 0)
        return 0;
    const int64_t cost = plan_whole(M, row_bytes, sms, at, B, pl);
    if (cost == 0) return 0;
    if (dtype == SSD_F32) return 1;
    const direct::Cut c = direct::plan_spans(M, row_bytes, warps, 64);
    const int64_t pairs = (M * c.spans + warps - 1) / warps * (c.blocks + 3);
    if (pl->whole_cluster_log2 >= 2) return cost <= pairs + 1 && M <= 8ll * pl->whole_clusters;
    return 3 * cost <= 4 * pairs + 3 && (at.shard || cost <= pairs + 6);
}

// Workspace: [0,256) header (error word, finished-CTA counter), two words per utterance, then
// M * partials float2.
int plan_verify(int B, int64_t M, int V, ssd_dtype dtype, const ssd_launch_opts *o,
                const RowsAt &at, VerifyPlan *plan) {
    const int es = dtype == SSD_F32 ? 4 : 2;
    VerifyPlan pl{};
    pl.kernel = (o && o->kernel) ? o->kernel : 2;
    if (pl.kernel != 1 && pl.kernel != 2) return SSD_ERR_ARG;
    const int sms = device_sm_count();
    if (sms <= 0 && !(o && o->ctas > 0)) return SSD_ERR_CUDA;
    pl.ctas = (o && o->ctas > 0) ? o->ctas : sms;
    const int64_t row_bytes = (int64_t)V * es;
    // column spans per row: enough items for a few balanced waves when there are few rows
    int split = 1;
    if (o && o->split > 0) {
        split = o->split;
    } else if (M > 0 && M < 4ll * pl.ctas) {
        // about four items per CTA, spans of 32 KB at least: every span is a stage hand-over
        // for the consumers, so more and smaller ones lose what the better balance gains
        // (250 rows of 98 KB: 13.9 us with 2 or 3 spans, 16.0 with 5, 16.9 with 6)
        const int64_t want = (4ll * pl.ctas + M - 1) / M;
        const int64_t most = row_bytes / 32768 > 1 ? row_bytes / 32768 : 1;
        split = (int)(want < most ? want : most);
    }
    if (split < 1) split = 1;
    if (split > 64) split = 64;
    pl.split = split;
    if (pl.kernel == 2) {
        pl.warps = (o && o->warps > 0) ? o->warps : (row_bytes >= 96 * 1024 ? 12 : 16);
        if (pl.warps > 16) return SSD_ERR_ARG;
        const int off_cache = (B + 1 <= kOffCacheMax) ? (B + 1) * 8 : 0;
        const int budget = 222 * 1024 - 512 - off_cache;
        const int max_stage = (budget / 2) & ~127;     // two stages must fit
        if (o && o->stage_bytes > 0) {
            pl.stage_bytes = o->stage_bytes;
        } else {
            // A span is cut into as few equal parts as a ring of two stages allows, one part per
            // stage.  Every stage costs each consumer warp about a hundred instructions of
            // hand-over whatever its size (measured: 0.33 us per stage and CTA), and two stages
            // of ~100 KB already keep enough bytes in flight, so few large stages beat a deeper
            // ring of small ones: a 98 KB row as one stage streams 6 % faster than as two.
            const int64_t span = (row_bytes + split - 1) / split + 32;
            const int64_t parts = (span + max_stage - 1) / max_stage;
            int64_t sb = ((span + parts - 1) / parts + 16 + 127) & ~127ll;
            if (sb < 4096) sb = 4096;
            if (sb > max_stage) sb = max_stage;
            pl.stage_bytes = (int)sb;
        }
        if (pl.stage_bytes < 1024 || pl.stage_bytes > max_stage || (pl.stage_bytes & 127))
            return SSD_ERR_ARG;
        pl.stages = (o && o->stages > 0) ? o->stages : budget / pl.stage_bytes;
        if (pl.stages > 16) pl.stages = 16;
        if (pl.stages < 2 || (int64_t)pl.stages * pl.stage_bytes > budget) return SSD_ERR_ARG;
        pl.smem_bytes = 128 + (size_t)((2 * pl.stages * 8 + pl.stages * sizeof(StageDesc) +
                                        off_cache + 127) & ~127) +
                        (size_t)pl.stages * pl.stage_bytes;
    } else {
        pl.warps = 8;
        pl.stages = 0; pl.stage_bytes = 0; pl.smem_bytes = 0;
    }
    // measured: one pair of four on the FMA pipe is the best split for bf16 (two lose to
    // instruction issue); fp32 logits are HBM-bound without it
    pl.fma_exp = (o && o->fma_exp) ? (o->fma_exp < 0 ? 0 : o->fma_exp) : (dtype == SSD_BF16 ? 1 : 0);
    if (pl.fma_exp > 3) return SSD_ERR_ARG;
    pl.partials = split * pl.warps;
    pl.direct = use_direct(M, row_bytes, dtype, pl.kernel, sms, o, at);
    if (pl.direct) {
        pl.direct_ctas = (o && o->ctas > 0) ? o->ctas : direct::kCtasPerSm * sms;
        if (o && o->split > 0) {
            pl.pairs = split;
            for (direct::Cut &c : pl.cut)
                c = direct::Cut{split, (direct::row_blocks(row_bytes) + split - 1) / split};
        } else {
            direct::plan_cuts(M, row_bytes, pl.direct_ctas * direct::kWarps,
                              pl.partials < 64 ? pl.partials : 64, at.skip && direct::table_fits(B, M),
                              pl.cut, &pl.pairs);
        }
    }
    pl.whole = use_whole(B, M, row_bytes, dtype, sms, o, at, &pl);
    // header | two words per utterance | partials
    pl.workspace_bytes = 256 + (((size_t)(B > 0 ? B : 0) * 16 + 255) & ~(size_t)255) +
                         (size_t)M * pl.partials * sizeof(float2);
    // Rows can be finished inside the streaming kernel where that kernel sees whole rows and can
    // keep the utterance offsets in shared memory.  It is not the default: in a chain of calls
    // the closing kernel's few microseconds are when the next streaming kernel's CTAs (which
    // need the SM's whole shared memory) get resident and past their set-up, and without it that
    // ramp-up is exposed instead (measured: 108 against 104 us per step on 32 utterances).
    const int finish = o ? o->finish : 0;
    if (finish < 0 || finish > 2) return SSD_ERR_ARG;
    pl.finish_inside = 0;
    if (finish == 2 && pl.kernel == 2 && split == 1 && B > 0 && B + 1 <= kOffCacheMax && M > 0) {
        const int NR = 2 * pl.stages;
        size_t hdr = 2 * (size_t)pl.stages * 8 + pl.stages * sizeof(StageDesc) + NR * sizeof(FinRow) +
                     (size_t)NR * pl.warps * 8 + pl.stages * 4 + 8 + (size_t)(B + 1) * 8;
        pl.fin_smem_bytes = 128 + ((hdr + 127) & ~(size_t)127) + (size_t)pl.stages * pl.stage_bytes;
        pl.finish_inside = pl.fin_smem_bytes <= 227 * 1024 ? 1 : 0;
    }
    if (finish == 2 && !pl.finish_inside) return SSD_ERR_ARG;
    *plan = pl;
    return SSD_OK;
}

static size_t partials_offset(int B) {
    return 256 + (((size_t)(B > 0 ? B : 0) * 16 + 255) & ~(size_t)255);
}

// Pairs per row that the streaming kernel of a plan leaves.
static int pairs_per_row(const VerifyPlan &plan) { return plan.direct ? plan.pairs : plan.partials; }

template <bool kArg>
static cudaError_t launch_direct(const void *logits, ssd_dtype dtype, int V, int64_t ld, int64_t M,
                                 const int64_t *tok_off, int B, const uint8_t *skip, void *partials,
                                 const VerifyPlan &plan, cudaStream_t stream) {
    const int es = dtype == SSD_F32 ? 4 : 2;
    direct::DirectParams p{};
    p.logits = static_cast<const char *>(logits);
    p.row_pitch = ld * es; p.row_bytes = V * es; p.M = M;
    for (int k = 0; k < direct::kCuts; ++k) p.cut[k] = plan.cut[k];
    p.pairs = plan.pairs;
    p.tok_off = tok_off; p.B = B; p.skip = skip; p.partials = partials;
    p.table = skip && direct::table_fits(B, M);
    const int64_t items = M * plan.pairs;
    const int64_t ctas = items < plan.direct_ctas ? items : plan.direct_ctas;
    const size_t smem = p.table ? (size_t)(B + 1) * sizeof(int32_t) : 0;
    // one pair in eight on the FMA pipe is the best split under the power cap (22,000 rows of
    // 200 KB: none 694 us, one 674, two 683); with the arg max none is (1,024 of 304 KB: 55.1
    // against 55.9)
    auto kern = direct::verify_rows_direct<bf16_t, kArg ? 0 : 1, kArg>;
    if (dtype == SSD_F32) kern = direct::verify_rows_direct<float, 0, kArg>;
    return launch_pdl(kern, (unsigned)ctas, (unsigned)direct::kThreads, smem, stream, p);
}

// The one launch of a call whose rows are closed where they are read.
template <int kEnd>
static int launch_whole(const void *logits, ssd_dtype dtype, int V, int64_t ld, int64_t M, const int64_t *tok_off,
                        int B, const uint8_t *skip, const whole::EndParams &end, const VerifyPlan &plan,
                        const Launch &L) {
    const ssd_launch_opts *o = L.opts;
    const int es = dtype == SSD_F32 ? 4 : 2;
    direct::DirectParams p{};
    p.logits = static_cast<const char *>(logits);
    p.row_pitch = ld * es; p.row_bytes = V * es; p.M = M;
    p.cut[0] = plan.whole_cut;
    p.tok_off = tok_off; p.B = B; p.skip = skip; p.table = skip != nullptr;
    whole::EndParams e = end;
    e.cluster_log2 = plan.whole_cluster_log2;
    e.V = V;
    constexpr int kF = kEnd == whole::kGreedy ? 0 : 1;       // as in launch_direct
    void (*kern)(const direct::DirectParams, const whole::EndParams) = whole::rows_whole<bf16_t, kF, kEnd, false>;
    if (dtype == SSD_F32) kern = whole::rows_whole<float, 0, kEnd, false>;
    if constexpr (kEnd == whole::kShard) {
        if (skip) kern = dtype == SSD_F32 ? whole::rows_whole<float, 0, kEnd, true> : whole::rows_whole<bf16_t, kF, kEnd, true>;
    }
    const unsigned cluster = 1u << plan.whole_cluster_log2;
    cudaError_t err = cudaSuccess;
    if (o && o->ev_begin) err = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_begin), L.stream);
    if (err == cudaSuccess)
        err = launch_clusters(kern, cluster, (unsigned)plan.whole_clusters * cluster, (unsigned)direct::kThreads,
                              plan.whole_smem_bytes, L.stream, p, e);
    if (err == cudaSuccess) err = cudaGetLastError();
    if (err == cudaSuccess && o && o->ev_end) err = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_end), L.stream);
    if (err != cudaSuccess) { record_cuda_error(err); return SSD_ERR_CUDA; }
    return SSD_OK;
}

// The closing kernel for P pairs per row and drafts of K tokens on average: four pairs a lane in
// one round trip, or eight and half the lanes per row where that makes a draft one sweep of the
// block instead of two (the call on 250 rows of 304 KB, 18 pairs each: 20.3 -> 19.1 us; 2 x 300
// rows, 9 pairs: 40.0 -> 37.5; with eight throughout, 5,568 rows of 3 pairs lose half a
// microsecond, 100 rows of 46 pairs a third).  A thread that walked 36 pairs by itself, twice,
// took 10 us for the closing kernel alone.
template <template <int, int> class Pick> static auto pick_lanes(int P, int64_t K) -> decltype(Pick<1, 4>::kernel()) {
    int G = 1;
    while (G < 32 && 4 * G < P) G *= 2;
    if (G > 1 && G < 32 && K >= 128 && K * G > kFinishThreads)
        return G == 2 ? Pick<1, 8>::kernel() : G == 4 ? Pick<2, 8>::kernel() : G == 8 ? Pick<4, 8>::kernel()
                                                                             : Pick<8, 8>::kernel();
    return G == 1 ? Pick<1, 4>::kernel() : G == 2 ? Pick<2, 4>::kernel() : G == 4 ? Pick<4, 4>::kernel()
         : G == 8 ? Pick<8, 4>::kernel() : G == 16 ? Pick<16, 4>::kernel() : Pick<32, 4>::kernel();
}
template <typename T> struct FinishKernels {
    template <int G, int L> struct Verify { static auto kernel() { return &verify_finish_kernel<T, G, L>; } };
    template <int G, int L> struct Shard { static auto kernel() { return &shard_finish_kernel<T, G, L>; } };
};

// Launches the streaming kernel that leaves pairs_per_row (reference, sum) pairs per row in the
// workspace (nothing for rows of skipped utterances).
static int launch_verify_rows(const void *logits, ssd_dtype dtype, int V, int64_t ld, int64_t M,
                              const int64_t *tok_off, int B, const uint8_t *skip, void *workspace,
                              unsigned long long epoch, const VerifyPlan &plan, const Launch &L) {
    if (M == 0) return SSD_OK;
    const ssd_launch_opts *o = L.opts;
    cudaError_t e;
    VerifyParams p{};
    p.logits = static_cast<const char *>(logits);
    p.V = V; p.ld = ld; p.M = M; p.split = plan.split; p.num_items = M * plan.split;
    p.tok_off = tok_off; p.B = B; p.skip = skip;
    p.table = skip && direct::table_fits(B, M);
    p.partials = reinterpret_cast<float2 *>(static_cast<char *>(workspace) + partials_offset(B));
    p.partials_per_row = plan.partials;
    p.warps = plan.warps; p.stages = plan.stages; p.stage_bytes = plan.stage_bytes;
    p.err_word = static_cast<unsigned long long *>(workspace); p.epoch = epoch;
    int64_t ctas = p.num_items < plan.ctas ? p.num_items : plan.ctas;
    if (o && o->ev_begin) {
        e = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_begin), L.stream);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    }
    if (plan.direct) {
        e = launch_direct<false>(logits, dtype, V, ld, M, tok_off, B, skip, p.partials, plan, L.stream);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    } else if (plan.kernel == 2) {
        void (*kern)(const VerifyParams) = verify_rows_tma<float, 0, false>;
        if (dtype == SSD_BF16)
            kern = plan.fma_exp == 1 ? verify_rows_tma<bf16_t, 1, false>
                 : plan.fma_exp == 2 ? verify_rows_tma<bf16_t, 2, false>
                 : plan.fma_exp == 3 ? verify_rows_tma<bf16_t, 3, false>
                                     : verify_rows_tma<bf16_t, 0, false>;
        e = ensure_dynamic_smem(reinterpret_cast<const void *>(kern), plan.smem_bytes);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
        e = launch_pdl(kern, (unsigned)ctas, (unsigned)((plan.warps + 1) * 32), plan.smem_bytes,
                       L.stream, p);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    } else {
        ctas = p.num_items < 8ll * plan.ctas ? p.num_items : 8ll * plan.ctas;
        e = launch_pdl(dtype == SSD_F32 ? verify_rows_plain<float> : verify_rows_plain<bf16_t>,
                       (unsigned)ctas, 256u, 0, L.stream, p);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    if (o && o->ev_end) {
        e = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_end), L.stream);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    }
    return SSD_OK;
}

// Eq. 5's threshold on the host: log(tau) in fp64, rounded to fp32.  tau <= 0 rejects nothing
// (p > 0 always), tau >= 1 everything (p <= 1 always), whatever rounding does to log p.
struct Threshold {
    float log_tau;
    int reject_none, reject_all;
};
static Threshold threshold_of(float tau_slm) {
    const double tau = (double)tau_slm;
    Threshold t;
    t.reject_none = !(tau > 0.0);
    t.reject_all = tau >= 1.0;
    t.log_tau = t.reject_none ? -INFINITY : (float)log(tau);
    return t;
}

int launch_verify(const void *logits, ssd_dtype dtype, int V, int64_t ld, int64_t M,
                  const int64_t *tok_off, const int32_t *draft_ids, int B, float tau_slm,
                  const uint8_t *skip, void *workspace, float *token_logp, float *row_lse,
                  int32_t *accepted_len, uint8_t *all_accepted, uint32_t *utt_status,
                  const VerifyPlan &plan, const Launch &L) {
    if (B == 0) return SSD_OK;
    const ssd_launch_opts *o = L.opts;
    unsigned long long *err_word = static_cast<unsigned long long *>(workspace);
    float2 *partials = reinterpret_cast<float2 *>(static_cast<char *>(workspace) + partials_offset(B));
    const unsigned long long epoch = next_epoch();
    const Threshold th = threshold_of(tau_slm);
    cudaError_t e;
    if (plan.finish_inside) {
        // The per-utterance words of this variant are told apart from leftovers by the host's
        // call number, which a captured launch would repeat at every replay: not while capturing.
        cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
        e = cudaStreamIsCapturing(L.stream, &capturing);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
        if (capturing != cudaStreamCaptureStatusNone) return SSD_ERR_ARG;
        FinParams q{};
        VerifyParams &p = q.v;
        p.logits = static_cast<const char *>(logits);
        p.V = V; p.ld = ld; p.M = M; p.split = 1; p.num_items = M;
        p.tok_off = tok_off; p.B = B; p.skip = skip;
        p.warps = plan.warps; p.stages = plan.stages; p.stage_bytes = plan.stage_bytes;
        p.err_word = err_word; p.epoch = epoch;
        q.draft_ids = draft_ids;
        q.log_tau = th.log_tau; q.reject_none = th.reject_none; q.reject_all = th.reject_all;
        q.token_logp = token_logp; q.row_lse = row_lse;
        q.accepted_len = accepted_len; q.all_accepted = all_accepted; q.utt_status = utt_status;
        q.utt_words = reinterpret_cast<unsigned long long *>(static_cast<char *>(workspace) + 256);
        q.done_ctas = err_word + 1;
        q.epoch32 = scratch_tag((uint32_t)epoch);
        const int64_t ctas = M < plan.ctas ? M : plan.ctas;
        if (o && o->ev_begin) {
            e = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_begin), L.stream);
            if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
        }
        void (*kern)(const FinParams) = verify_rows_fin<float, 0>;
        if (dtype == SSD_BF16)
            kern = plan.fma_exp == 1 ? verify_rows_fin<bf16_t, 1>
                 : plan.fma_exp == 2 ? verify_rows_fin<bf16_t, 2>
                 : plan.fma_exp == 3 ? verify_rows_fin<bf16_t, 3>
                                     : verify_rows_fin<bf16_t, 0>;
        e = ensure_dynamic_smem(reinterpret_cast<const void *>(kern), plan.fin_smem_bytes);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
        e = launch_pdl(kern, (unsigned)ctas, (unsigned)((plan.warps + 1) * 32), plan.fin_smem_bytes,
                       L.stream, q);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
        if (o && o->ev_end) {
            e = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_end), L.stream);
            if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
        }
        return SSD_OK;
    }
    const int rc = launch_verify_rows(logits, dtype, V, ld, M, tok_off, B, skip, workspace, epoch,
                                      plan, L);
    if (rc != SSD_OK) return rc;
    const int P = pairs_per_row(plan);
    e = launch_pdl(
        dtype == SSD_F32 ? pick_lanes<FinishKernels<float>::Verify>(P, M / B)
                         : pick_lanes<FinishKernels<bf16_t>::Verify>(P, M / B),
        (unsigned)B, (unsigned)kFinishThreads, 0, L.stream,
        static_cast<const char *>(logits), V, ld, M, tok_off, draft_ids, B, th.log_tau,
        th.reject_none, th.reject_all, skip, static_cast<const float2 *>(partials), P,
        token_logp, row_lse, accepted_len, all_accepted, utt_status,
        static_cast<const unsigned long long *>(err_word), epoch);
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    e = cudaGetLastError();
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    return SSD_OK;
}

// Vocabulary-parallel verification, this rank's part: the same streaming kernel over the local
// columns, then one (maximum, sum, draft logit) triple per row.
int launch_verify_shard(const void *logits, ssd_dtype dtype, int V_local, int64_t ld, int64_t M,
                        int64_t col0, const int64_t *tok_off, const int32_t *draft_ids, int B,
                        const uint8_t *skip, void *workspace, float *shard_stats,
                        const VerifyPlan &plan, const Launch &L) {
    if (B == 0) return SSD_OK;
    unsigned long long *err_word = static_cast<unsigned long long *>(workspace);
    float2 *partials = reinterpret_cast<float2 *>(static_cast<char *>(workspace) + partials_offset(B));
    if (plan.whole) {
        whole::EndParams end{};
        end.col0 = col0; end.draft_ids = draft_ids; end.stats = shard_stats;
        return launch_whole<whole::kShard>(logits, dtype, V_local, ld, M, tok_off, B, skip, end, plan, L);
    }
    const unsigned long long epoch = next_epoch();
    const int rc = launch_verify_rows(logits, dtype, V_local, ld, M, tok_off, B, skip, workspace,
                                      epoch, plan, L);
    if (rc != SSD_OK) return rc;
    const int P = pairs_per_row(plan);
    cudaError_t e = launch_pdl(
        dtype == SSD_F32 ? pick_lanes<FinishKernels<float>::Shard>(P, M / B)
                         : pick_lanes<FinishKernels<bf16_t>::Shard>(P, M / B),
        (unsigned)B, (unsigned)kFinishThreads, 0, L.stream,
        static_cast<const char *>(logits), V_local, ld, M, col0, tok_off, draft_ids, B, skip,
        static_cast<const float2 *>(partials), P, shard_stats,
        static_cast<const unsigned long long *>(err_word), epoch);
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    e = cudaGetLastError();
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    return SSD_OK;
}

int launch_verify_combine(const float *stats_all, int R, int64_t V_total, const int64_t *tok_off,
                          const int32_t *draft_ids, int B, int64_t M, float tau_slm,
                          const uint8_t *skip, float *token_logp, float *row_lse,
                          int32_t *accepted_len, uint8_t *all_accepted, uint32_t *utt_status,
                          cudaStream_t stream) {
    if (B == 0) return SSD_OK;
    const Threshold th = threshold_of(tau_slm);
    cudaError_t e = launch_pdl(combine_kernel, (unsigned)B, (unsigned)kFinishThreads, 0, stream,
                               stats_all, R, V_total, M, tok_off, draft_ids, B, th.log_tau,
                               th.reject_none, th.reject_all, skip, token_logp, row_lse,
                               accepted_len, all_accepted, utt_status);
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    e = cudaGetLastError();
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    return SSD_OK;
}

size_t greedy_workspace_bytes(int64_t R, const VerifyPlan &plan) {
    return 256 + (size_t)R * plan.partials * sizeof(float4);
}

int launch_greedy(const void *logits, ssd_dtype dtype, int V, int64_t ld, int64_t R,
                  void *workspace, int32_t *next_token, float *next_logp, float *row_lse,
                  uint32_t *row_status, const VerifyPlan &plan, const Launch &L) {
    if (R == 0) return SSD_OK;
    if (plan.kernel != 2) return SSD_ERR_ARG;      // only the bulk-copy kernel tracks the arg max
    const ssd_launch_opts *o = L.opts;
    unsigned long long *err_word = static_cast<unsigned long long *>(workspace);
    float4 *partials = reinterpret_cast<float4 *>(static_cast<char *>(workspace) + 256);
    if (plan.whole) {
        whole::EndParams end{};
        end.token = next_token; end.logp = next_logp; end.lse = row_lse; end.status = row_status;
        return launch_whole<whole::kGreedy>(logits, dtype, V, ld, R, nullptr, 0, nullptr, end, plan, L);
    }
    const unsigned long long epoch = next_epoch();
    VerifyParams p{};
    p.logits = static_cast<const char *>(logits);
    p.V = V; p.ld = ld; p.M = R; p.split = plan.split; p.num_items = R * plan.split;
    p.tok_off = nullptr; p.B = 0; p.skip = nullptr;
    p.partials = reinterpret_cast<float2 *>(partials); p.partials_per_row = plan.partials;
    p.warps = plan.warps; p.stages = plan.stages; p.stage_bytes = plan.stage_bytes;
    p.err_word = err_word; p.epoch = epoch;
    const int64_t ctas = p.num_items < plan.ctas ? p.num_items : plan.ctas;
    cudaError_t e;
    if (o && o->ev_begin) {
        e = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_begin), L.stream);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    }
    if (plan.direct) {
        e = launch_direct<true>(logits, dtype, V, ld, R, nullptr, 0, nullptr, partials, plan, L.stream);
    } else {
        void (*kern)(const VerifyParams) = verify_rows_tma<float, 0, true>;
        if (dtype == SSD_BF16)
            kern = plan.fma_exp >= 1 ? verify_rows_tma<bf16_t, 1, true> : verify_rows_tma<bf16_t, 0, true>;
        e = ensure_dynamic_smem(reinterpret_cast<const void *>(kern), plan.smem_bytes);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
        e = launch_pdl(kern, (unsigned)ctas, (unsigned)((plan.warps + 1) * 32), plan.smem_bytes,
                       L.stream, p);
    }
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    if (o && o->ev_end) {
        e = cudaEventRecord(static_cast<cudaEvent_t>(o->ev_end), L.stream);
        if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    }
    auto finish = dtype == SSD_F32 ? greedy_finish_kernel<float, false> : greedy_finish_kernel<bf16_t, false>;
    if (plan.direct)
        finish = dtype == SSD_F32 ? greedy_finish_kernel<float, true> : greedy_finish_kernel<bf16_t, true>;
    e = launch_pdl(finish,
                   (unsigned)((R + kGreedyWarps - 1) / kGreedyWarps),
                   (unsigned)(kGreedyWarps * 32), 0, L.stream, p.logits, V, ld, R,
                   static_cast<const float4 *>(partials), pairs_per_row(plan), next_token, next_logp,
                   row_lse, row_status, static_cast<const unsigned long long *>(err_word), epoch);
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    e = cudaGetLastError();
    if (e != cudaSuccess) { record_cuda_error(e); return SSD_ERR_CUDA; }
    return SSD_OK;
}

}  // namespace ssd
