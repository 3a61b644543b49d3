"""Performance cases of the decision path: what a program that decodes speech with CTC drafts has
the library do, at the sizes it does it.

Four kinds of pass, each through the public binding and into buffers that the program keeps from
batch to batch (plain calls, since a batch's row counts change from one call to the next):

  step     ssd_ctc_draft -> ssd_entropy_gate_from_maxima -> ssd_verify(skip = gate) -> ssd_assemble:
           the whole decision for one ragged batch, from logits to final hypotheses and the list
           of utterances left to the auto-regressive pass; with `early_exit`
           ssd_verify_early_exit stands in the place of ssd_verify
  greedy   ssd_greedy_step: one step of the auto-regressive fallback over the utterances left
  shard    ssd_verify_shard -> ssd_verify_combine: one rank of an LLM head whose columns are split
           over several ranks, the other ranks' statistics already gathered

The shape of a batch (utterance lengths, which utterances are confident, where a reject is) comes
from the case alone, the values from the seed.
"""
import math
import random

import torch

from paper_2603_11243_b200 import binding as ssd

BYTES = {"f32": 4, "bf16": 2}
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}
MOST_BYTES = 40e9                 # of one drawn pass's logits; the largest listed case has more


def step(name, **kw):
    """A step case: 50 CTC frames a second, ragged lengths, bf16, high-accuracy thresholds unless said."""
    c = dict(name=name, kind="step", B=1, t_dist="uniform", t_lo=1000, t_hi=1000, V_ctc=1025,
             V_llm=49152, pad=0, dtype="bf16", cap=250, tau_ctc=0.7, tau_slm=0.1, flat=0.1,
             confident=0.0, accept=0.3, early_exit=False, shape=4)
    c.update(kw)
    return c


def listed():
    return [
        # one short utterance, a small symbol set and fp32 logits: the interactive call, all latency
        step("utterance_200x129_f32", t_lo=200, t_hi=200, V_ctc=129, V_llm=32000, dtype="f32",
             cap=50, tau_ctc=0.5, accept=0.0, shape=0),
        # one 20 s utterance against the widest LLM vocabulary: a server that does not batch
        step("utterance_1000_v152064", V_llm=152064),
        # a dozen short utterances; both vocabularies odd, so no row starts on a 16-byte boundary,
        # and the LLM's logits are a slice of a padded matrix
        step("batch12_odd_v32003", B=12, t_lo=60, t_hi=700, V_ctc=349, V_llm=32003, pad=2, cap=200,
             confident=0.25, shape=11),
        # a small serving batch, every utterance verified
        step("batch32_v49152", B=32, t_lo=250, t_hi=750, cap=200, shape=1),
        # an ordinary batch; half of the utterances pass the gate and are never verified
        step("batch128_v100352", B=128, t_lo=500, t_hi=1500, V_llm=100352, cap=400, flat=0.05,
             confident=0.5, shape=2),
        # the largest batch that one card is given: heavy-tailed lengths, the widest vocabularies
        step("batch512_v152064", B=512, t_dist="lognormal", t_lo=100, t_hi=3000, V_ctc=4097,
             V_llm=152064, cap=600, accept=0.0, shape=3),
        # fp32 logits in an ordinary batch
        step("batch64_v49152_f32", B=64, dtype="f32"),
        # the high-throughput operating point: 50,000 frames of a character head in one batch, the
        # gate accepts all of it and verification has nothing to read
        step("batch56_chars_gated", B=56, t_lo=750, t_hi=1030, V_ctc=348, cap=1500, tau_ctc=3.0,
             flat=0.0, confident=1.0, shape=6),
        # the high-accuracy operating point on such a batch, verification stopping at first rejects
        step("batch56_chars_early_exit", B=56, t_lo=750, t_hi=1030, V_ctc=348, cap=1500,
             tau_slm=0.2, flat=0.05, confident=0.14, accept=0.547, early_exit=True, shape=5),
        # the fallback's decoding step: two dozen utterances left over from a batch ...
        dict(name="greedy_24_v49152", kind="greedy", R=24, V_llm=49152, pad=0, dtype="bf16"),
        # ... and the leftovers of many batches pooled
        dict(name="greedy_1024_v152064", kind="greedy", R=1024, V_llm=152064, pad=0, dtype="bf16"),
        # the small serving batch with the LLM head's columns split over four ranks
        dict(name="shard_batch32_v12288of49152", kind="shard", B=32, t_dist="uniform", t_lo=250,
             t_hi=750, V_llm=12288, ranks=4, pad=0, dtype="bf16", cap=200, tau_slm=0.1, accept=0.3,
             shape=1),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "early_exit", "greedy", "shard"])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    V_llm = _log_uniform(rng, 32000, 152064)
    V_llm -= rng.choice([0, 1, V_llm % 64])
    pad = rng.choice([0, 0, rng.randrange(1, 65)])
    if kind == "greedy":
        return dict(kind="greedy", R=_log_uniform(rng, 1, 1024), V_llm=V_llm, pad=pad, dtype=dtype)
    # most utterances, for batches of verification rows up to the byte limit
    t_lo = _log_uniform(rng, 100, 1000)
    t_hi = min(3000, int(t_lo * rng.uniform(1.0, 4.0)))
    cap = rng.choice([50, 200, 250, 400, 600])
    rows = min(cap, 0.4 * 0.5 * (t_lo + t_hi)) + 1
    B = min(_log_uniform(rng, 1, 512), max(1, int(MOST_BYTES / (rows * V_llm * BYTES[dtype]))))
    shape = rng.randrange(1 << 16)
    if kind == "shard":
        ranks = rng.choice([2, 4, 8])
        return dict(kind="shard", B=B, t_dist="uniform", t_lo=t_lo, t_hi=t_hi, V_llm=V_llm // ranks,
                    ranks=ranks, pad=pad, dtype=dtype, cap=cap, tau_slm=0.1, accept=0.3, shape=shape)
    c = step("", B=B, t_dist=rng.choice(["uniform", "lognormal"]), t_lo=t_lo, t_hi=t_hi,
             V_ctc=_log_uniform(rng, 129, 4097), V_llm=V_llm, pad=pad, dtype=dtype, cap=cap,
             tau_slm=rng.choice([0.1, 0.2]), flat=rng.choice([0.05, 0.1]),
             confident=rng.choice([0.0, 0.14, 0.5, 0.9]), accept=rng.choice([0.0, 0.3, 0.55]),
             early_exit=kind == "early_exit", shape=shape)
    del c["name"]
    return c


def _shape(case):
    """Lengths, draft lengths, which utterances are confident and where each has its reject
    (its draft length: nowhere)."""
    rng = random.Random(case["shape"])
    T, K, sure, reject = [], [], [], []
    for _ in range(case["B"]):
        if case["t_dist"] == "lognormal":
            t = math.exp(rng.gauss(0.5 * (math.log(case["t_lo"]) + math.log(case["t_hi"])), 0.75))
            t = max(case["t_lo"], min(case["t_hi"], int(round(t))))
        else:
            t = rng.randint(case["t_lo"], case["t_hi"])
        k = min(case["cap"], int(round(0.4 * t)))      # two frames in five are not blank
        T.append(t)
        K.append(k)
        sure.append(rng.random() < case.get("confident", 0.0))
        reject.append(k if rng.random() < case["accept"] else min(k, int(rng.random() * k)))
    return T, K, sure, reject


def _offsets(lengths):
    off = torch.zeros(len(lengths) + 1, dtype=torch.int64)
    off[1:] = torch.cumsum(torch.tensor(lengths, dtype=torch.int64), 0)
    return off


def _rows(n, V, pad, dtype, cols, vals, gen):
    """n rows of unit-normal logits in a matrix `pad` columns wider, entry cols[r] set to vals[r]."""
    x = torch.empty((n, V + pad), dtype=TORCH[dtype], device="cuda")
    x.normal_(generator=gen)
    x[torch.arange(n, device="cuda"), cols] = vals.to(x.dtype)
    return x[:, :V]


def _uniform(n, lo, hi, gen):
    return lo + (hi - lo) * torch.rand((n,), device="cuda", generator=gen)


def _verify_inputs(case, K, reject, V_total, gen):
    """Draft ids, the boosted token of every row (the draft's, but for the rejected position) and
    its logit: 3 to 10 above the level at which its likelihood is tau_SLM."""
    M = sum(K)
    ids = torch.randint(0, V_total, (M,), device="cuda", generator=gen)
    planted = [sum(K[:b]) + reject[b] for b in range(len(K)) if reject[b] < K[b]]
    boosted = ids.clone()
    at = torch.tensor(planted, dtype=torch.int64, device="cuda")
    boosted[at] = (ids[at] + 1 + torch.randint(0, V_total - 1, (len(planted),), device="cuda",
                                               generator=gen)) % V_total
    tau = case["tau_slm"]
    level = math.log(V_total) + 0.5 + math.log(tau / (1.0 - tau))
    return ids.to(torch.int32), boosted, level + _uniform(M, 3.0, 10.0, gen)


def _zeroed(out):
    """Entries that a call leaves alone (rows of gated utterances, tokens past a draft's end) are
    zeros from the start."""
    for t in out.values():
        t.zero_()
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1_000_003 * (seed + 1))
    code = ssd.F32 if case["dtype"] == "f32" else ssd.BF16
    if case["kind"] == "greedy":
        R, V = case["R"], case["V_llm"]
        top = torch.randint(0, V, (R,), device="cuda", generator=gen)
        logits = _rows(R, V, case["pad"], case["dtype"], top,
                       math.log(V) + 0.5 + _uniform(R, -1.0, 8.0, gen), gen)
        i32, f32 = torch.int32, torch.float32
        out = {k: torch.zeros((R,), dtype=d, device="cuda") for k, d in
               (("next_token", i32), ("next_logp", f32), ("row_lse", f32), ("row_status", i32))}
        out["workspace"] = torch.zeros((max(256, ssd.ssd_greedy_step_workspace_bytes(R, V, code)),),
                                       dtype=torch.uint8, device="cuda")
        return dict(case=case, logits=logits, out=out)
    T, K, sure, reject = _shape(case)
    B, M, V = case["B"], sum(K), case["V_llm"]
    ranks = case.get("ranks", 1)
    s = dict(case=case, tok_off=_offsets(K).cuda())
    s["ids"], boosted, vals = _verify_inputs(case, K, reject, V * ranks, gen)
    if ranks > 1:
        # rank 0 has columns [0, V): rows whose boosted token lies elsewhere are plain noise here
        here = boosted < V
        s["logits"] = _rows(M, V, case["pad"], case["dtype"], torch.where(here, boosted, 0),
                            torch.where(here, vals, 0.0), gen)
        # what the all-gather brings from the others: maximum, sum relative to it, draft logit
        stats = torch.zeros((ranks, M, 3), dtype=torch.float32, device="cuda")
        stats[1:, :, 0] = _uniform((ranks - 1) * M, 3.8, 4.8, gen).view(ranks - 1, M)
        stats[1:, :, 1] = V * math.exp(0.5) * torch.exp(-stats[1:, :, 0])
        stats[1:, :, 2] = -math.inf
        rows = torch.arange(M, device="cuda")
        for ids, logit in ((boosted, vals), (s["ids"].long(), torch.where(boosted == s["ids"], vals, 0.5))):
            r, i = (ids // V).long(), rows
            far = r > 0
            r, i, x = r[far], i[far], logit[far].float()
            old = stats[r, i, 0]
            new = torch.maximum(old, x)
            stats[r, i, 1] = stats[r, i, 1] * torch.exp(old - new) + torch.exp(x - new)
            stats[r, i, 0] = new
        far = s["ids"] >= V
        stats[(s["ids"][far] // V).long(), rows[far], 2] = torch.where(boosted == s["ids"], vals, 0.5)[far].float()
        s["stats"] = stats
        s["workspace"] = torch.zeros((max(256, ssd.ssd_verify_workspace_bytes(B, M, V, code)),),
                                     dtype=torch.uint8, device="cuda")
        s["out"] = _zeroed(ssd.alloc_verify_outputs(M, B, "cuda", 0))
        return s
    s["logits"] = _rows(M, V, case["pad"], case["dtype"], boosted, vals, gen)
    N, V_ctc = sum(T), case["V_ctc"]
    s["frame_off"] = _offsets(T).cuda()
    winner = torch.randint(1, V_ctc, (N,), device="cuda", generator=gen)
    winner[torch.rand((N,), device="cuda", generator=gen) < 0.6] = 0
    boost = _uniform(N, 2.0, 12.0, gen)
    flat = torch.rand((N,), device="cuda", generator=gen) < case["flat"]
    flat[s["frame_off"][:-1]] = True                 # no doubtful utterance is gated by luck
    boost = torch.where(flat, _uniform(N, 0.0, 1.0, gen), boost)
    sure_frame = torch.repeat_interleave(torch.tensor(sure), torch.tensor(T)).cuda()
    boost = torch.where(sure_frame, _uniform(N, 8.0, 12.0, gen), boost)
    s["ctc"] = _rows(N, V_ctc, 0, case["dtype"], winner, math.log(V_ctc) + 0.5 + boost, gen)
    s["draft"] = _zeroed(ssd.alloc_ctc_outputs(N, B, "cuda"))
    s["gate"] = dict(gate_accept=torch.zeros((B,), dtype=torch.uint8, device="cuda"),
                     max_entropy=torch.zeros((B,), dtype=torch.float32, device="cuda"))
    if case["early_exit"]:
        s["out"] = _zeroed(ssd.alloc_early_exit_outputs(M, B, V, code, "cuda"))
    else:
        s["out"] = _zeroed(ssd.alloc_verify_outputs(
            M, B, "cuda", ssd.ssd_verify_workspace_bytes(B, M, V, code)))
    i32 = torch.int32
    s["final"] = {k: torch.zeros((n,), dtype=d, device="cuda") for k, n, d in
                  (("final_tokens", M, i32), ("final_len", B, i32), ("is_final", B, torch.uint8),
                   ("ar_count", 1, i32), ("ar_utt", B, i32), ("ar_resume", B, i32))}
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "greedy":
        out = ssd.ssd_greedy_step(s["logits"], out=s["out"])
        return {k: out[k] for k in ("next_token", "next_logp", "row_lse", "row_status")}
    results = ("token_logp", "row_lse", "accepted_len", "all_accepted", "utt_status")
    if c["kind"] == "shard":
        ssd.ssd_verify_shard(s["logits"], 0, s["tok_off"], s["ids"], stats=s["stats"][0],
                             workspace=s["workspace"])
        out = ssd.ssd_verify_combine(s["stats"], c["V_llm"] * c["ranks"], s["tok_off"], s["ids"],
                                     c["tau_slm"], out=s["out"])
        # a rank's (maximum, sum) pair stands for one log-sum-exp and is as good relative to any
        # other logit of the row: what it is for comes back in row_lse and token_logp
        return {k: out[k] for k in results}
    d = ssd.ssd_ctc_draft(s["ctc"], s["frame_off"], 0, c["cap"], out=s["draft"])
    g = ssd.ssd_entropy_gate_from_maxima(d["utt_max_entropy"], d["utt_status"], c["tau_ctc"],
                                         out=s["gate"])
    if c["early_exit"]:
        # which rows after an utterance's first reject still get read depends on timing, and with
        # them token_logp, row_lse and rows_read: the decisions are what this call is for
        results = ("accepted_len", "all_accepted", "utt_status")
        v = ssd.ssd_verify_early_exit(s["logits"], s["tok_off"], s["ids"], c["tau_slm"],
                                      skip=g["gate_accept"], out=s["out"])
    else:
        v = ssd.ssd_verify(s["logits"], s["tok_off"], s["ids"], c["tau_slm"],
                           skip=g["gate_accept"], out=s["out"])
    f = ssd.ssd_assemble(s["ids"], s["tok_off"], g["gate_accept"], v["accepted_len"],
                         v["all_accepted"], out=s["final"])
    return dict(draft={k: t for k, t in d.items() if k != "workspace"}, gate=g,
                verify={k: v[k] for k in results}, final=f)


def _log_sum_exp(x, entropy=False):
    """Per row of x, in 64 bits and a gigabyte at a time: log-sum-exp and, if asked for, entropy."""
    lse = torch.empty((x.shape[0],), dtype=torch.float64, device=x.device)
    ent = torch.empty_like(lse) if entropy else None
    step = max(1, (1 << 27) // x.shape[1])
    for r in range(0, x.shape[0], step):
        c = x[r:r + step].double()
        top = c.amax(1)
        c -= top[:, None]
        e = c.exp()
        total = e.sum(1)
        lse[r:r + step] = top + total.log()
        if entropy:
            ent[r:r + step] = total.log() - (c * e).sum(1) / total
    return lse, ent


def exact(case, seed):
    """What run() returns, in 64 bits, and None in the place of whole numbers."""
    s = prepare(case, seed)
    x = s["logits"]
    lse, _ = _log_sum_exp(x)
    if case["kind"] == "greedy":
        return dict(next_token=None, next_logp=x.amax(1).double() - lse, row_lse=lse, row_status=None)
    ids = s["ids"].long()
    whole = dict.fromkeys(("accepted_len", "all_accepted", "utt_status"))
    if case["kind"] == "shard":
        here = ids < case["V_llm"]
        mine = x.gather(1, torch.where(here, ids, 0)[:, None])[:, 0].double()
        mine = torch.where(here, mine, -math.inf)
        others = s["stats"][1:].double()
        lse = torch.logsumexp(torch.cat([lse[None], others[..., 0] + others[..., 1].log()]), 0)
        logit = torch.maximum(mine, others[..., 2].amax(0))
        return dict(whole, token_logp=logit - lse, row_lse=lse)
    lengths = s["frame_off"].diff()
    frame_lse, entropy = _log_sum_exp(s["ctc"], entropy=True)
    utterance = torch.repeat_interleave(torch.arange(len(lengths), device=x.device), lengths)
    most = torch.zeros((len(lengths),), dtype=torch.float64, device=x.device)
    most.scatter_reduce_(0, utterance, entropy, "amax")
    draft = dict(dict.fromkeys(k for k in s["draft"] if k != "workspace"),
                 frame_entropy=entropy, frame_lse=frame_lse, utt_max_entropy=most)
    verify = dict(whole)
    if not case["early_exit"]:
        read = torch.repeat_interleave(most >= case["tau_ctc"], s["tok_off"].diff())
        logp = x.gather(1, ids[:, None])[:, 0].double() - lse
        verify.update(token_logp=torch.where(read, logp, 0.0), row_lse=torch.where(read, lse, 0.0))
    return dict(draft=draft, gate=dict(gate_accept=None, max_entropy=most), verify=verify,
                final=dict.fromkeys(s["final"]))


def work(case):
    """Each logit that the decisions need read once, each output written once; an exponential, a
    multiply-add and an addition a logit."""
    es = BYTES[case["dtype"]]
    if case["kind"] == "greedy":
        n = case["R"] * case["V_llm"]
        return {"bytes": n * es + 16 * case["R"], "flops": 4.0 * n}
    T, K, sure, reject = _shape(case)
    if case["kind"] == "shard":
        n = sum(K) * case["V_llm"]
        return {"bytes": n * es + (12 * case["ranks"] + 24) * sum(K), "flops": 4.0 * n}
    if case["early_exit"]:
        rows = sum(min(k, r + 1) for k, r, ok in zip(K, reject, sure) if not ok)
    else:
        rows = sum(k for k, ok in zip(K, sure) if not ok)
    n_llm, n_ctc = rows * case["V_llm"], sum(T) * case["V_ctc"]
    return {"bytes": (n_llm + n_ctc) * es + 12 * sum(T) + 8 * sum(K) + 12 * rows + 8 * sum(K),
            "flops": 4.0 * n_llm + 6.0 * n_ctc}


def tolerance(case):
    """Four times what was measured against the same path in 64 bits.  Log-sum-exps and
    log-likelihoods are off by 1e-7 to 3e-6 of their norm.  An entropy is off by about 1e-6 nats
    whatever its size, so the less doubt there is in a batch the larger that is beside the norm of
    its entropies: 4e-6 of it with half of the utterances confident, 1e-3 where every frame is
    confident and entropies are around 1e-3 nats."""
    if case["kind"] == "step":
        if all(_shape(case)[2]):
            return {"rel": 4e-3, "max": 3e-2}
        if case["confident"] > 0.5:
            return {"rel": 4e-5, "max": 4e-4}
    return {"rel": 1.6e-5, "max": 1.6e-4}
