// rows_whole: the direct-load kernel for calls that need a row's sums and nothing across rows (the
// greedy step, a rank's statistics): a thread-block cluster sees its rows from end to end and closes
// them in the same launch (use_whole in ssd_verify.cu says where it runs).
//
// A launch costs the host 2 us and the GPU about one, whatever it does, and a closing kernel begins
// with a round trip for its inputs; on calls of a few microseconds that is most of the time.  Rows
// are dealt to clusters whole, their column spans to the cluster's warps exactly as
// verify_rows_direct does it over the grid.  A span's pair goes straight into the shared memory of
// the CTA that closes the row (st.shared::cluster); one cluster barrier later that CTA merges.
// Nothing passes through the workspace.  (The decision of Eq. 5 needs all rows of an utterance.
// With the last CTA to arrive taking it -- a fence, an atomic and a read of what the others left,
// one after another -- ssd_verify took 7.6 us instead of 5.7 on 20 rows of 128 KB, 11.8 instead of
// 11.0 on 250 of 98: it keeps its closing kernel.)
#pragma once

#include <type_traits>

#include "ssd_common.cuh"
#include "ssd_direct.cuh"
#include "ssd_ranges.cuh"
#include "ssd_stream.cuh"

namespace ssd {
namespace whole {

using direct::Cut;
using direct::Deal;
using direct::DirectParams;
using direct::kThreads;
using direct::kWarps;
using direct::SpanResult;

enum End { kGreedy, kShard };

struct EndParams {
    int cluster_log2;
    int V;
    int32_t *token;                // greedy step
    float *logp, *lse;
    uint32_t *status;
    int64_t col0;                  // shard
    const int32_t *draft_ids;
    float *stats;
};

__device__ __forceinline__ bool owns(const int64_t *tok_off, const uint8_t *skip, int64_t M, int b, int row) {
    const int64_t i0 = tok_off[b], i1 = tok_off[b + 1];
    return ranges::rows_sound(i0, i1, M) && i0 <= row && row < i1 && !(skip && skip[b]);
}
// Whether an utterance that the search does not find has the row.  Asking every utterance for each row that
// none has -- behind the last one's rows, or in front of the first one's -- took 174 us for 4,000 rows of 8 KB
// of which 2,000 utterances have half (15 now; 20 with a closing kernel): only where the offsets fall
// somewhere.  Called by all lanes of a warp; out of line, away from what every row needs.
template <typename T, bool kSkip>
__device__ __noinline__ bool owned_elsewhere(const int64_t *tok_off, const uint8_t *skip, int B, int64_t M, int row) {
    bool owned = false;
    if (!stream::offsets_ordered(tok_off, B))
        for (int b = 0; !owned && b < B; ++b) owned = owns(tok_off, skip, M, b, row);
    return owned;
}

// Shared memory: the pairs of the rows this CTA closes, their drafts, and (with skip flags) the rows
// to read before each utterance.
// (kSkip: a call with skip flags.  Without, the code for them in the same kernel cost a shard 1 % and more.)
template <typename T, int kF, int kEnd, bool kSkip>
__global__ void __launch_bounds__(kThreads, direct::kCtasPerSm) rows_whole(const DirectParams p, const EndParams e) {
    constexpr bool kArg = kEnd == kGreedy;
    constexpr int ES = Elem<T>::kBytes;
    using Pair = typename std::conditional<kArg, float4, float2>::type;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int32_t warp_tot[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int clog = e.cluster_log2, C = 1 << clog;
    const int rank = blockIdx.x & (C - 1), cl = blockIdx.x >> clog, nc = gridDim.x >> clog;
    const Cut cut = p.cut[0];
    Pair *pairs = reinterpret_cast<Pair *>(smem);
    const int rows_per_cta = (((int)p.M + nc - 1) / nc + C - 1) >> clog;
    float2 *drafts = reinterpret_cast<float2 *>(pairs + rows_per_cta * cut.spans);
    int32_t *act = reinterpret_cast<int32_t *>(drafts + (kArg ? 0 : rows_per_cta));
    cluster_arrive();
    pdl_wait();
    pdl_launch_dependents();
    // A malformed list of offsets may name rows more than once, more of them than this CTA's shared
    // memory is laid out for: then every row is read once and asked for its owner (look_up).
    int rows = (int)p.M;
    if (kSkip && p.table) rows = stream::count_rows(p.tok_off, p.skip, p.B, p.M, act, warp_tot, kWarps, nullptr);
    const bool table = kSkip && p.table && rows <= (int)p.M;
    if (!table) rows = (int)p.M;
    const int here = cl < rows ? (rows - cl + nc - 1) / nc : 0;
    cluster_wait();          // all CTAs of the cluster run: their shared memory may be written

    // row index a (closed by CTA a mod C, warp a / C mod kWarps) stands for this row of the matrix
    auto row_of = [&](int a) {
        const int at = cl + a * nc;
        if (!table) return at;
        const int b = stream::utterance_of_count(act, p.B, at);
        return at + (int)p.tok_off[b] - act[b];
    };
    // What the caller passed in for the rows this CTA closes, a row a lane: the draft token's logit
    // and whether anyone wants the row.  The last warp fetches it while its own first block is on its
    // way: where spans do not fill the last round it has the fewest.
    auto look_up = [&]() {
        if (warp != kWarps - 1) return;
        for (int k0 = 0; (k0 << clog) + rank < here; k0 += 32) {
            const bool mine = ((k0 + lane) << clog) + rank < here;
            const int k = mine ? k0 + lane : k0;
            const int row = row_of((k << clog) + rank);
            const int64_t id = (int64_t)e.draft_ids[row] - e.col0;
            float x = -INFINITY;
            if (id >= 0 && id < e.V) x = Elem<T>::load(p.logits + (int64_t)row * p.row_pitch + id * ES);
            // rows of no sound utterance that is read are left alone; those of the table all have one
            bool wanted = table || owns(p.tok_off, p.skip, p.M, utterance_of_row(p.tok_off, p.B, row), row);
            if (__any_sync(0xffffffffu, !wanted)) wanted |= owned_elsewhere<T, kSkip>(p.tok_off, p.skip, p.B, p.M, row);
            if (mine) drafts[k] = make_float2(x, wanted ? 1.f : 0.f);
        }
    };
    const int first = (warp << clog) + rank;
    direct::stream_spans<T, kF, kArg, 1 + kEnd + 2 * kSkip>(
        p, cut, Deal{(unsigned)first, (unsigned)(kWarps << clog), here, cl, nc, table, true}, act,
        [&] { if (!kArg) look_up(); },
        [&](int, int a, int sp, const SpanResult &out) {
            const uint32_t to = cluster_address(smem_u32(pairs + (a >> clog) * cut.spans + sp), a & (C - 1));
            if (lane != 0) return;
            if (kArg)
                asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(to), "f"(out.m), "f"(out.S),
                             "f"(out.vmax), "f"(__int_as_float(out.vidx)) : "memory");
            else
                asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(to), "f"(out.m), "f"(out.S) : "memory");
        });
    __syncwarp();
    cluster_arrive();
    cluster_wait();

    for (int a = first; a < here; a += kWarps << clog) {
        const Pair *pp = pairs + (a >> clog) * cut.spans;
        const int64_t row = row_of(a);
        if constexpr (kEnd == kGreedy) {
            const stream::GreedyRow g = stream::greedy_row<T, true>([&](int q) { return pp[q]; }, cut.spans,
                                                                    p.logits + row * p.row_pitch, e.V, lane);
            if (lane == 0) {
                e.token[row] = g.token;
                if (e.logp) e.logp[row] = g.logp;
                if (e.lse) e.lse[row] = g.lse;
                if (e.status) e.status[row] = g.status;
            }
        } else {
            const float2 d = drafts[a >> clog];
            float Mx = kNegInit, S = 0.f;
            for (int q = lane; q < cut.spans; q += 32) Mx = fmaxf(Mx, pp[q].x);
            Mx = warp_max(Mx);
            for (int q = lane; q < cut.spans; q += 32) S += pp[q].y * ex2((pp[q].x - Mx) * kLog2e);
            S = warp_sum(S);
            if (d.y != 0.f && lane == 0) {
                e.stats[3 * row + 0] = Mx;
                e.stats[3 * row + 1] = S;
                e.stats[3 * row + 2] = d.x;
            }
        }
    }
}

}  // namespace whole
}  // namespace ssd
