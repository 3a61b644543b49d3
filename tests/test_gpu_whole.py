"""Rows closed by the clusters that read them (the greedy step and a rank's statistics on most sizes)
against the oracle and the plain-load kernel: one to eight CTAs a cluster, rows that do not come out
even over the clusters, rows of less than a unit and of several spans, offsets that name no row, some
twice or leave some out."""
import numpy as np
import pytest
import torch

import helpers as H
from oracle import ref
from paper_2603_11243_b200 import binding as ssd

pytestmark = pytest.mark.gpu


def _matrix(R, V, dtype, seed, pad=7):
    g = torch.Generator()
    g.manual_seed(seed)
    return (torch.randn((R, V + pad), generator=g) * 3.0).to(dtype)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("R,V", [(1, 1), (1, 70001), (2, 33), (31, 9000), (33, 513), (73, 4097), (147, 1039),
                                 (149, 15), (285, 2048), (297, 3001), (593, 600), (1025, 514)])
def test_greedy_step(cuda_device, R, V, dtype):
    wide = _matrix(R, V, dtype, 3 * R + V)
    for r in range(0, R, 5):                       # the largest value twice: the first counts
        wide[r, 2 + V // 3] = wide[r, 1 + V] = 40.0
    want = ref.greedy_step(H.storage_numpy(wide[:, 2:2 + V].contiguous()), V)
    before = ssd.lib().ssd_launch_count()
    got = ssd.ssd_greedy_step(wide.to(cuda_device)[:, 2:2 + V])
    torch.cuda.synchronize()
    assert ssd.lib().ssd_launch_count() - before == 1
    np.testing.assert_array_equal(got["next_token"].cpu().numpy(), want["next_token"])
    assert np.abs(got["row_lse"].cpu().numpy() - want["row_lse"]).max() <= H.FLOAT_TOL
    assert np.abs(got["next_logp"].cpu().numpy() - want["next_logp"]).max() <= H.FLOAT_TOL


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [600, 9000])
@pytest.mark.parametrize("split", [0, 1])
def test_greedy_step_of_large_finite_logits(cuda_device, split, V, dtype):
    """A token forced with a large logit, and rows with nothing above a large negative one, by the clusters
    and by the pair kernel: finite rows, whatever the rounding of a logit times log2e."""
    largest = torch.finfo(dtype).max
    values = (5000.0, 1e6, 1e9, 2e9, 1e10, 1e12, 1e20, 1e30, 1e38, largest, -5000.0, -1e9, -1e10, -1e20, -9e29)
    wide = _matrix(2 * len(values), V, dtype, V)
    x = wide[:, 3:3 + V]
    for k, v in enumerate(values):
        x[2 * k + 1] = -largest                    # alone, and behind a masked first half
        if v > 0:
            x[2 * k, 11 * k] = x[2 * k + 1, V - 1 - k] = v
        else:
            x[2 * k, :] = v
            x[2 * k + 1, V // 2:] = v
    want = ref.greedy_step(H.storage_numpy(x.contiguous()), V)
    got = ssd.ssd_greedy_step(wide.to(cuda_device)[:, 3:3 + V], opts=H.opts(split=split) if split else None)
    torch.cuda.synchronize()
    got = {k: got[k].cpu().numpy() for k in ("next_token", "next_logp", "row_lse", "row_status")}
    assert not got["row_status"].any()
    np.testing.assert_array_equal(got["next_token"], want["next_token"])
    # nothing beside a forced token; V or V - V // 2 equal logits (a difference of log-sum-exps of 1e20 does
    # not show either in 64 bits)
    likely = [0.0 if v > 0 else -np.log(n) for v in values for n in (V, V - V // 2)]
    assert np.abs(got["next_logp"] - likely).max() <= H.FLOAT_TOL
    # the sum and the result are rounded once each
    assert (np.abs(got["row_lse"] - want["row_lse"]) <= H.FLOAT_TOL + 2.0 ** -23 * np.abs(want["row_lse"])).all()
    forced = [r for r in range(len(x)) if values[r // 2] > 0]
    assert (got["next_logp"][forced] == 0).all()


# [0, M] as it should be; a gap before, between and after; one utterance's end before its start; one
# past the matrix; two that overlap
OFFSETS = {"sound": lambda M: [0, M // 3, M // 3, M], "gaps": lambda M: [M // 5, M // 2, M - 1],
           "reversed": lambda M: [0, M // 2, M // 4, M], "past": lambda M: [0, M // 2, M + 3],
           "twice": lambda M: [0, M // 2, M // 4, M // 2, M // 3, M],
           # more utterances than a warp looks at in one go, most of them empty: rows in front of the first and
           # behind the last one's, and one that ends past the matrix
           "many": lambda M: [M // 4 + min(b // 8, M // 2) for b in range(700)],
           "many, past": lambda M: [M // 4 + min(b // 8, M // 2) for b in range(700)] + [M + 1],
           "many, falling": lambda M: [M // 4 + min(b // 8, M // 2) for b in range(700)] + [M // 8, M // 4]}


@pytest.mark.parametrize("offsets", sorted(OFFSETS))
@pytest.mark.parametrize("skipping", [False, True])
@pytest.mark.parametrize("M,V,dtype", [(8, 513, torch.bfloat16), (61, 5001, torch.float32), (299, 1100, torch.bfloat16),
                                       (640, 257, torch.float32), (1500, 1024, torch.bfloat16)])
def test_shard_statistics(cuda_device, M, V, dtype, skipping, offsets):
    x = _matrix(M, V, dtype, M)[:, 3:3 + V].to(cuda_device)
    off = torch.tensor(OFFSETS[offsets](M), dtype=torch.int64, device=cuda_device)
    B, col0 = off.numel() - 1, 1000
    g = torch.Generator()
    g.manual_seed(M + 1)
    ids = torch.randint(0, col0 + 2 * V, (M,), generator=g, dtype=torch.int32).to(cuda_device)
    skip = torch.tensor([b % 2 for b in range(B)], dtype=torch.uint8, device=cuda_device) if skipping else None
    size = max(256, ssd.ssd_verify_workspace_bytes(B, M, V, ssd.F32 if dtype == torch.float32 else ssd.BF16))
    got, want = (torch.full((M, 3), 7.5, device=cuda_device) for _ in range(2))
    before = ssd.lib().ssd_launch_count()
    ssd.ssd_verify_shard(x, col0, off, ids, skip=skip, stats=got,
                         workspace=torch.zeros((size,), dtype=torch.uint8, device=cuda_device))
    assert ssd.lib().ssd_launch_count() - before == 1
    ssd.ssd_verify_shard(x, col0, off, ids, skip=skip, stats=want, opts=H.opts(kernel=1))
    torch.cuda.synchronize()
    # the same rows written, the draft logits as they are, the pairs for one log-sum-exp
    assert torch.equal(got == 7.5, want == 7.5)
    assert torch.equal(got[:, 2], want[:, 2])
    lse = [s[:, 0].double() + s[:, 1].double().log() for s in (got, want)]
    assert float((lse[0] - lse[1]).abs().max()) <= H.FLOAT_TOL
