"""fp32 rows of a gated batch through the direct-load kernel (what ssd_verify does with skip flags on up to
400 MB) against the oracle: ragged ends, spans, rows outside the fast pass, and the ring for comparison."""
import numpy as np
import pytest
import torch

import helpers as H
from oracle import ref
from paper_2603_11243_b200 import binding as ssd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("col0", [0, 1, 3])
@pytest.mark.parametrize("V", [1, 7, 9, 255, 257, 2049, 20011, 150000])
def test_gated_rows(cuda_device, V, col0):
    lens = [5, 0, 17, 1, 9]
    g = torch.Generator()
    g.manual_seed(V + col0)
    wide = torch.randn((32, V + 7), generator=g) * 2.0
    view = wide[:, col0:col0 + V]
    if V > 300:
        view[0, :280] = float("-inf")              # nothing finite in a span's first block
        view[1, V - 1] = 300.0
        view[2] -= 6000.0
        view[24, : V // 2] = float(torch.finfo(torch.float32).min)
    ids = view.argmax(1).to(torch.int32)
    ids[::3] = torch.randint(0, V, (11,), generator=g, dtype=torch.int32)
    ids[0] = view[0].argmax()
    off = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int64)
    skip = np.array([0, 0, 1, 0, 0], np.uint8)
    args = (wide.to(cuda_device)[:, col0:col0 + V], off.to(cuda_device), ids.to(cuda_device), 0.1)
    out = ssd.ssd_verify(*args, skip=torch.from_numpy(skip).to(cuda_device))
    ring = ssd.ssd_verify(*args, skip=torch.from_numpy(skip).to(cuda_device), opts=H.opts(kernel=2))
    torch.cuda.synchronize()
    orc = ref.verify(H.storage_numpy(view.contiguous()), V, off.numpy(), ids.numpy(), float(np.float32(0.1)), skip=skip)
    for k in ("accepted_len", "all_accepted", "utt_status"):
        assert torch.equal(out[k], ring[k]), k
    read = [r for r in range(32) if not 5 <= r < 22]
    for k in ("token_logp", "row_lse"):
        got, want = out[k].cpu().numpy()[read].astype(np.float64), orc[k][read]
        # two units in the last place of values up to 6,000 beside the tolerance
        assert (np.abs(got - want) <= H.FLOAT_TOL + 2 * 2.0 ** -23 * np.abs(want)).all(), k
