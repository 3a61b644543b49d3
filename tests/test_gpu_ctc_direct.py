"""Frame statistics of rows that are read into registers (ssd_ctc_draft by default on rows of up to 4 KB)
against the oracle and the plain-load kernel: every number of units a lane may have, ragged ends of every
length, ties, and rows that take the second pass or the one element by element."""
import numpy as np
import pytest
import torch

import helpers as H
from oracle import ref
from paper_2603_11243_b200 import binding as ssd

pytestmark = pytest.mark.gpu

# a unit is 16 bf16 or 8 fp32 logits, a row at most 128 units and two ragged ends
SIZES = {torch.bfloat16: (1, 2, 15, 16, 17, 31, 33, 129, 255, 257, 348, 384, 400, 513, 770, 1025, 1536, 1540, 2047, 2063),
         torch.float32: (1, 2, 7, 8, 9, 65, 129, 193, 200, 257, 385, 513, 770, 1025, 1031)}


def _statistics(x, dev, **kw):
    """Of every row, without utterances."""
    out = ssd.ssd_ctc_draft(x, torch.zeros((1,), dtype=torch.int64, device=dev), 0, 0, **kw)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("dtype,V", [(d, V) for d in SIZES for V in SIZES[d]])
@pytest.mark.parametrize("N,col0", [(1, 0), (13, 1), (70, 3), (300, 16)])
def test_against_the_oracle(cuda_device, N, col0, dtype, V):
    g = torch.Generator()
    g.manual_seed(V + N)
    wide = (torch.randn((N, V + 21), generator=g) * 4.0).to(dtype)
    view = wide[:, col0:col0 + V]
    for r in range(0, N, 3):                       # the largest value three times: the first counts
        for c in torch.randint(0, V, (3,), generator=g).tolist():
            view[r, c] = 25.0
    orc = ref.ctc_draft(H.storage_numpy(view.contiguous()), V, np.array([0, N], np.int64), 0, 0)
    out = _statistics(wide.to(cuda_device)[:, col0:col0 + V], cuda_device, want_logprob=True)
    np.testing.assert_array_equal(out["frame_argmax"].cpu().numpy(), orc["frame_argmax"])
    for k in ("frame_entropy", "frame_lse"):
        assert np.abs(out[k].cpu().numpy() - orc[k]).max() <= H.FLOAT_TOL, k
    lp = out["frame_logprob"].cpu()[:, :V].double() - (view.double() - torch.from_numpy(orc["frame_lse"])[:, None])
    assert float(lp.abs().max()) <= H.FLOAT_TOL


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [24, 348, 1000])
def test_rows_that_are_not_plain(cuda_device, V, dtype):
    g = torch.Generator()
    g.manual_seed(V)
    wide = torch.randn((64, V + 9), generator=g).to(dtype)
    x = wide[:, 2:2 + V]
    lowest = torch.finfo(dtype).min
    x[0:4, : V // 2] = float("-inf")               # masked, in front, behind and all but one
    x[4:8, V // 2:] = float("-inf")
    x[8:12, :] = float("-inf")
    x[8:12, V // 3] = -2.0
    x[12:16, 1:] = lowest
    x[16:20] += 5000.0
    x[20:24] -= 30000.0
    x[24:28, 5] = 300.0
    x[28:32, V - 1] = float("-inf")
    x[40:44, V - 2] = float("nan")
    x[44:48, 0] = float("inf")
    x[48:52, :] = float("-inf")
    dev = wide.to(cuda_device)[:, 2:2 + V]
    a, b = _statistics(dev, cuda_device), _statistics(dev, cuda_device, opts=H.opts(kernel=1))
    odd = torch.zeros((64,), dtype=torch.bool, device=cuda_device)
    odd[40:52] = True
    for out in (a, b):
        assert torch.equal(torch.isnan(out["frame_entropy"]), odd)
    assert torch.equal(a["frame_argmax"][~odd], b["frame_argmax"][~odd])
    assert float((a["frame_entropy"] - b["frame_entropy"])[~odd].abs().max()) <= H.FLOAT_TOL
    d = (a["frame_lse"] - b["frame_lse"])[~odd].abs()
    # a few units in the last place of values up to 30,000
    assert bool((d <= H.FLOAT_TOL + 4 * 2.0 ** -23 * b["frame_lse"][~odd].abs()).all())


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [9, 300, 1000])
@pytest.mark.parametrize("times", [1, 4])
def test_rows_of_large_finite_logits(cuda_device, times, V, dtype):
    """One large logit, alone and among others; rows with nothing above a large negative one; also columns
    of a matrix so wide that the bulk-copy tiles do not take it."""
    largest = torch.finfo(dtype).max
    values = (1e6, 1.3e7, 2e7, 1e8, 1e10, 1e20, 1e38, largest, -1e6, -2e7, -1e10, -1e20, -1e30, -largest)
    g = torch.Generator()
    g.manual_seed(V)
    x = torch.randn((2 * len(values), V * times), generator=g).to(dtype)[:, :V]
    for k, v in enumerate(values):
        x[2 * k + 1] = float("-inf")
        if v > 0:
            x[2 * k, k % V] = x[2 * k + 1, V - 1 - k % V] = v
        else:
            x[2 * k, :] = v
            x[2 * k + 1, V // 2:] = v
    orc = ref.ctc_draft(H.storage_numpy(x.contiguous()), V, np.array([0, len(x)], np.int64), 0, 0)
    wide = torch.zeros((len(x), V * times), dtype=dtype, device=cuda_device)
    wide[:, :V] = x.to(cuda_device)
    out = _statistics(wide[:, :V], cuda_device)
    np.testing.assert_array_equal(out["frame_argmax"].cpu().numpy(), orc["frame_argmax"])
    # equal logits or one by itself, whatever they are: 64 bits do not hold this beside 1e20 either
    entropy = [0.0 if v > 0 else np.log(n) for v in values for n in (V, V - V // 2)]
    assert np.abs(out["frame_entropy"].cpu().numpy() - entropy).max() <= H.FLOAT_TOL
    d = np.abs(out["frame_lse"].cpu().numpy().astype(np.float64) - orc["frame_lse"])
    assert (d <= H.FLOAT_TOL + 2.0 ** -23 * np.abs(orc["frame_lse"])).all()


@pytest.mark.parametrize("N,V,direct", [(4736, 2047, 1), (5500, 2047, 0), (24000, 200, 0), (44000, 128, 1),
                                        (11500, 700, 1), (13000, 600, 0), (15000, 1025, 1)])
def test_rounds_of_either_kernel(cuda_device, N, V, direct):
    """bf16 rows that registers would need a second round for and tiles would not, and sizes beside them: the
    kernel that is meant runs, and agrees with the plain loads."""
    direct = direct if torch.cuda.get_device_properties(0).multi_processor_count == 148 else None
    x = torch.randn((N, V), generator=torch.Generator(device=cuda_device).manual_seed(N), device=cuda_device).bfloat16()
    off = torch.tensor([0, N // 3, N], device=cuda_device)
    span = ssd.ssd_ctc_draft_read_span(x.data_ptr(), ssd.BF16, V, V, N)
    assert span.faults == 0 and direct in (None, span.direct)
    a, b = ssd.ssd_ctc_draft(x, off, 0, 50), ssd.ssd_ctc_draft(x, off, 0, 50, opts=H.opts(kernel=1))
    torch.cuda.synchronize()
    assert torch.equal(a["frame_argmax"], b["frame_argmax"]) and torch.equal(a["draft_len"], b["draft_len"])
    for k in ("frame_entropy", "frame_lse"):
        assert float((a[k] - b[k]).abs().max()) <= H.FLOAT_TOL, k
