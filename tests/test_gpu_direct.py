"""The direct-load streaming kernel (what ssd_verify, ssd_verify_shard and ssd_greedy_step run by
default on most bf16 calls) against the fp64 oracle and the plain-load kernel, at the sizes where
its units, blocks, spans and tables have their edges."""
import numpy as np
import pytest
import torch

import helpers as H
from oracle import ref
from paper_2603_11243_b200 import binding as ssd

pytestmark = pytest.mark.gpu

# a unit is 16 bf16 logits, a block 512; sizes around both, and one of several spans
SIZES = (1, 2, 15, 16, 17, 31, 33, 47, 511, 512, 513, 1024, 1039, 4097, 20011)


def _rows(M, V, col0, seed, dtype=torch.bfloat16, scale=2.0):
    g = torch.Generator()
    g.manual_seed(seed)
    wide = (torch.randn((M, V + 19), generator=g) * scale).to(dtype)
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32)
    return wide, wide[:, col0:col0 + V], ids


def _offsets(lens):
    return torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int64)


def _verify(view, off, ids, dev, wide, col0, skip=None, opts=None):
    x = wide.to(dev)[:, col0:col0 + view.shape[1]]
    sk = None if skip is None else torch.as_tensor(skip, dtype=torch.uint8).to(dev)
    out = ssd.ssd_verify(x, off.to(dev), ids.to(dev), 0.1, skip=sk, opts=opts)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("col0", [0, 1, 7, 13])
@pytest.mark.parametrize("V", SIZES)
def test_verify_sizes_and_alignments(cuda_device, V, col0):
    lens = [5, 0, 17, 1, 9]
    wide, view, ids = _rows(sum(lens), V, col0, 7 * V + col0)
    off = _offsets(lens)
    skip = [0, 0, 1, 0, 0]
    out = _verify(view, off, ids, cuda_device, wide, col0, skip)
    orc = ref.verify(H.storage_numpy(view.contiguous()), V, off.numpy(), ids.numpy(),
                     float(np.float32(0.1)), skip=np.array(skip, np.uint8))
    H.compare_stage2(out, orc, off.numpy(), 0.1, skip=np.array(skip, np.uint8), require_all_margins=False)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", SIZES)
def test_greedy_first_of_equals(cuda_device, V, dtype):
    """The largest logit planted several times, next to unit and block edges: the first counts."""
    wide, view, _ = _rows(23, V, 3, V, dtype)
    rng = np.random.default_rng(V)
    for r in range(23):
        for c in {int(rng.integers(0, V)), V - 1, min(V - 1, 16 * int(rng.integers(0, 1 + V // 16)))}:
            view[r, c] = 30.0
    want = ref.greedy_step(H.storage_numpy(view.contiguous()), V)
    got = ssd.ssd_greedy_step(wide.to(cuda_device)[:, 3:3 + V])
    torch.cuda.synchronize()
    np.testing.assert_array_equal(got["next_token"].cpu().numpy(), want["next_token"])
    assert np.abs(got["row_lse"].cpu().numpy() - want["row_lse"]).max() <= H.FLOAT_TOL


@pytest.mark.parametrize("V", [700, 5000])
def test_rows_outside_the_fast_pass(cuda_device, V):
    """Masked vocabularies, logits far from the reference in both directions, large magnitudes:
    the same answers as the plain-load kernel; NaN and +inf are flagged by both."""
    lens = [4] * 12
    wide, view, ids = _rows(48, V, 5, V)
    lowest = torch.finfo(torch.bfloat16).min
    view[0:4, :600] = float("-inf")              # nothing finite in a span's first block
    view[4:8, :] = float("-inf")
    view[4:8, V // 2] = 1.5                      # one finite logit
    view[8:12, :] = lowest
    view[8:12, 3] = 0.0
    view[12:16, V - 1] = 300.0                   # far above everything before it
    view[16:20, 0] = 300.0                       # a first logit far above the rest
    view[20:24] += 6000.0
    view[24:28] -= 6000.0
    view[28:32, V - 2] = float("nan")
    view[32:36, 1] = float("inf")
    view[36:40, :] = float("-inf")               # a row of nothing
    for r in list(range(0, 28)) + list(range(40, 48)):
        ids[r] = int(view[r].float().argmax())
    off = _offsets(lens)
    a = _verify(view, off, ids, cuda_device, wide, 5)
    b = _verify(view, off, ids, cuda_device, wide, 5, opts=H.opts(kernel=1))
    for k in ("accepted_len", "all_accepted", "utt_status"):
        assert torch.equal(a[k], b[k]), k
    assert (a["utt_status"].cpu().numpy()[[7, 8, 9]] == ssd.UTT_NONFINITE).all()
    fine = [r for r in range(48) if not 28 <= r < 40]
    for k in ("token_logp", "row_lse"):
        x, y = a[k].cpu()[fine].double(), b[k].cpu()[fine].double()
        # the two sum in different orders: a few units in the last place of values up to 6,000
        assert bool(((x - y).abs() <= H.FLOAT_TOL + 4 * 2.0 ** -23 * y.abs()).all()), k
    ga = ssd.ssd_greedy_step(wide.to(cuda_device)[:, 5:5 + V])
    want = view.float().argmax(1).numpy()
    rows = [r for r in range(48) if not 28 <= r < 40]
    np.testing.assert_array_equal(ga["next_token"].cpu().numpy()[rows], want[rows])


@pytest.mark.parametrize("B,split", [(1, 0), (2046, 0), (2047, 0), (2500, 0), (700, 3)])
def test_skipped_utterances(cuda_device, B, split):
    """The count of rows to read in shared memory, its largest size, and the way without it."""
    rng = np.random.default_rng(B)
    lens = rng.integers(0, 4, size=B)
    skip = (rng.random(B) < 0.6).astype(np.uint8)
    V = 1100
    wide, view, ids = _rows(int(lens.sum()) or 1, V, 2, B)
    off = _offsets(lens)
    M = int(off[-1])
    if M == 0:
        wide, view, ids = wide[:0], view[:0], ids[:0]
    o = H.opts(split=split) if split else None
    a = _verify(view, off, ids, cuda_device, wide, 2, skip, o)
    b = _verify(view, off, ids, cuda_device, wide, 2, skip, H.opts(kernel=1))
    for k in ("accepted_len", "all_accepted", "utt_status"):
        assert torch.equal(a[k], b[k]), k
    rows = torch.from_numpy(np.repeat(skip == 0, lens))
    diff = (a["token_logp"].cpu()[rows] - b["token_logp"].cpu()[rows]).abs()
    assert diff.numel() == 0 or float(diff.max()) <= H.FLOAT_TOL


@pytest.mark.parametrize("kernel", [0, 2])
@pytest.mark.parametrize("B", [31, 32, 33, 64, 65, 97, 128, 129, 511, 512, 513, 1024, 1025, 1537, 2047])
def test_count_of_rows_to_read(cuda_device, B, kernel):
    """As many utterances as a warp, a turn and the block count, one fewer and one more, by the direct loads
    and by the ring: each utterance's own rows are read, and no others."""
    rng = np.random.default_rng(B)
    lens = rng.integers(0, 4, size=B)
    lens[[0, -1]] = 3
    skip = (rng.random(B) < 0.4).astype(np.uint8)
    skip[[0, -1]] = 0
    V, M = 40, int(lens.sum())
    wide, view, ids = _rows(M, V, 0, B)
    off = _offsets(lens).to(cuda_device)
    args = (wide.to(cuda_device)[:, :V], off, ids.to(cuda_device), 0.1)
    plain = ssd.ssd_verify(*args, opts=H.opts(kernel=1))
    out = ssd.alloc_verify_outputs(M, B, cuda_device, ssd.ssd_verify_workspace_bytes(B, M, V, ssd.BF16))
    for k in ("token_logp", "row_lse"):
        out[k].fill_(7.0)
    ssd.ssd_verify(*args, skip=torch.from_numpy(skip).to(cuda_device), out=out, opts=H.opts(kernel=kernel))
    torch.cuda.synchronize()
    read = torch.from_numpy(np.repeat(skip == 0, lens)).to(cuda_device)
    for k in ("token_logp", "row_lse"):
        assert float((out[k][read] - plain[k][read]).abs().max()) <= H.FLOAT_TOL, k
        assert bool((out[k][~read] == 7.0).all()), k
    was_read = torch.from_numpy(skip == 0).to(cuda_device)
    assert torch.equal(out["accepted_len"][was_read], plain["accepted_len"][was_read])
    assert not out["utt_status"].any()


def test_malformed_offsets(cuda_device):
    """Offsets that run backwards: flagged, the sound utterances around them unharmed."""
    wide, view, ids = _rows(30, 900, 0, 3)
    off = torch.tensor([0, 10, 4, 20, 31, 30], dtype=torch.int64)
    skip = [0, 0, 0, 0, 0]
    a = _verify(view, off, ids, cuda_device, wide, 0, skip)
    b = _verify(view, off, ids, cuda_device, wide, 0, skip, H.opts(kernel=1))
    for k in ("accepted_len", "all_accepted", "utt_status"):
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("V", [n * 512 + d for n in (16, 17, 18, 19, 34, 35) for d in (-1, 0, 1)])
def test_groups_of_blocks(cuda_device, V):
    """One span a row, whose blocks end just before, on and after the groups that a lane sums apart."""
    wide, view, ids = _rows(9, V, 0, V)
    off = _offsets([4, 5])
    out = _verify(view, off, ids, cuda_device, wide, 0, opts=H.opts(split=1))
    orc = ref.verify(H.storage_numpy(view.contiguous()), V, off.numpy(), ids.numpy(), float(np.float32(0.1)))
    H.compare_stage2(out, orc, off.numpy(), 0.1, require_all_margins=False)
    got = ssd.ssd_greedy_step(wide.to(cuda_device)[:, :V], opts=H.opts(split=1))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(got["next_token"].cpu().numpy(), ref.greedy_step(H.storage_numpy(view.contiguous()), V)["next_token"])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [49152, 152064])
def test_small_terms_behind_a_peak(cuda_device, V, dtype):
    """A row's first block (1 KB) holds equal peaks, the rest of the row lies 17 below them: what a
    unit of it adds to a lane's sum of the peaks is under half an ulp, all of it together is 1.2e-5
    of the row."""
    x = torch.full((4, V), -23.0, dtype=dtype)
    peaks = 1024 // x.element_size()
    x[:, :peaks] = -6.0
    want = -6.0 + np.log(peaks + (V - peaks) * np.exp(-17.0))
    # the terms added one by one: 16 blocks of a group, the groups, four sums, a tree of 32 lanes; each
    # loses at most 2^-25 of the sum.  An exponential is good to 2^-22, the result to an ulp of it.
    terms = 16 + -(-V // (16 * peaks)) + 4 + 5
    bound = terms * 2.0 ** -25 + 2.0 ** -22 + 2.0 ** -23 * abs(want)
    off = torch.tensor([0, 4]).to(cuda_device)
    ids = torch.zeros(4, dtype=torch.int32, device=cuda_device)
    got = [ssd.ssd_greedy_step(x.to(cuda_device), opts=H.opts(split=1))]
    if dtype == torch.bfloat16:
        got.append(ssd.ssd_verify(x.to(cuda_device), off, ids, 0.1, opts=H.opts(split=1)))
    torch.cuda.synchronize()
    for o in got:
        assert np.abs(o["row_lse"].cpu().numpy().astype(np.float64) - want).max() <= bound


@pytest.mark.parametrize("V,col0", [(700, 0), (8003, 1)])
@pytest.mark.parametrize("B", [64, 2046, 2500])
def test_shares_of_a_large_batch(cuda_device, B, V, col0):
    """More rows than warps, all, half, and ever fewer of them read: the row counts around those at
    which the kernel changes its cut; with 2,500 utterances it cannot count and keeps one."""
    M, dev = 5000, cuda_device
    g = torch.Generator(device=dev).manual_seed(V + B)
    wide = torch.randn((M, V + 3), generator=g, device=dev).bfloat16()
    x = wide[:, col0:col0 + V]
    ids = torch.randint(0, V, (M,), generator=g, device=dev, dtype=torch.int32)
    # utterance lengths of 1 and more, so that the rows read can be set to one
    rng = np.random.default_rng(B)
    cuts = np.sort(rng.choice(np.arange(1, M), size=B - 1, replace=False))
    off = torch.tensor(np.concatenate([[0], cuts, [M]]), dtype=torch.int64)
    lens = np.diff(off.numpy())
    plain = ssd.ssd_verify(x, off.to(dev), ids, 0.1, opts=H.opts(kernel=1))
    for target in (M, M // 2 + 40, M // 2, M // 4, M // 8 + 1, M // 16, M // 32, M // 32 + 1, 60, 1):
        skip, left = np.ones(B, np.uint8), target
        for b in rng.permutation(B):
            if lens[b] <= left:
                skip[b], left = 0, left - lens[b]
        out = ssd.alloc_verify_outputs(M, B, dev, ssd.ssd_verify_workspace_bytes(B, M, V, ssd.BF16))
        for t in (out["token_logp"], out["row_lse"]):
            t.fill_(7.0)
        out["workspace"].fill_(0xff)                     # pairs that nobody writes would be NaN
        ssd.ssd_verify(x, off.to(dev), ids, 0.1, skip=torch.from_numpy(skip).to(dev), out=out)
        torch.cuda.synchronize()
        read = torch.from_numpy(np.repeat(skip == 0, lens)).to(dev)
        for k in ("token_logp", "row_lse"):
            d = (out[k][read] - plain[k][read]).abs()
            assert d.numel() == 0 or float(d.max()) <= H.FLOAT_TOL, (k, target)
            assert bool((out[k][~read] == 7.0).all()), (k, target)
        was_read = torch.from_numpy(skip == 0).to(dev)
        assert torch.equal(out["accepted_len"][was_read], plain["accepted_len"][was_read]), target
        assert not out["utt_status"].any()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("M,V", [(33, 40003), (300, 40003), (591, 20011), (593, 20011), (1500, 16384), (5000, 700)])
def test_shares_of_a_small_batch(cuda_device, M, V, dtype):
    """Fewer rows than warps (and, at the end, a few more) of both types, all to none of them read, at the counts
    where the kernel changes its cut: more spans a row than the cut for all rows has."""
    dev, B = cuda_device, min(M, 120)
    code = ssd.F32 if dtype == torch.float32 else ssd.BF16
    g = torch.Generator(device=dev).manual_seed(M)
    wide = torch.randn((M, V + 3), generator=g, device=dev).to(dtype)
    x = wide[:, 1:1 + V]
    ids = torch.randint(0, V, (M,), generator=g, device=dev, dtype=torch.int32)
    rng = np.random.default_rng(M)
    cuts = np.sort(rng.choice(np.arange(1, M), size=B - 1, replace=False)) if B < M else np.arange(1, M)
    off = torch.tensor(np.concatenate([[0], cuts, [M]]), dtype=torch.int64)
    lens = np.diff(off.numpy())
    plain = ssd.ssd_verify(x, off.to(dev), ids, 0.1, opts=H.opts(kernel=1))
    for target in sorted({M} | {(M >> k) + d for k in range(1, 7) for d in (0, 1)}):
        skip, left = np.ones(B, np.uint8), target
        for b in rng.permutation(B):
            if lens[b] <= left:
                skip[b], left = 0, left - lens[b]
        out = ssd.alloc_verify_outputs(M, B, dev, ssd.ssd_verify_workspace_bytes(B, M, V, code))
        for t in (out["token_logp"], out["row_lse"]):
            t.fill_(7.0)
        out["workspace"].fill_(0xff)                     # pairs that nobody writes would be NaN
        ssd.ssd_verify(x, off.to(dev), ids, 0.1, skip=torch.from_numpy(skip).to(dev), out=out)
        torch.cuda.synchronize()
        read = torch.from_numpy(np.repeat(skip == 0, lens)).to(dev)
        for k in ("token_logp", "row_lse"):
            d = (out[k][read] - plain[k][read]).abs()
            assert d.numel() == 0 or float(d.max()) <= H.FLOAT_TOL, (k, target)
            assert bool((out[k][~read] == 7.0).all()), (k, target)
        was_read = torch.from_numpy(skip == 0).to(dev)
        assert torch.equal(out["accepted_len"][was_read], plain["accepted_len"][was_read]), target
        assert not out["utt_status"].any()
