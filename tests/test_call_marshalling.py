"""The native marshalling of the hot calls: what it does not take goes the general way and raises
what that raises; what it takes computes what the general way computes."""
import sys
import warnings

import pytest
import torch

import helpers as H
import paper_2603_11243_b200
from paper_2603_11243_b200 import binding as ssd
from paper_2603_11243_b200 import build as ssd_build


@pytest.fixture(scope="module", autouse=True)
def built():
    ssd_build.build()


def _verify_inputs(device, M=6, V=40):
    x = torch.zeros((M, V), dtype=torch.bfloat16, device=device)
    off = torch.tensor([0, M], dtype=torch.int64, device=device)
    ids = torch.zeros((M,), dtype=torch.int32, device=device)
    out = ssd.alloc_verify_outputs(M, 1, device, 4096)
    return x, off, ids, out


def test_what_is_not_plainly_fine_is_declined():
    call = ssd._native()
    x, off, ids, out = _verify_inputs("cpu")
    assert call.verify(x, off, ids, 0.1, None, None, out) is None               # host tensors
    assert call.verify("logits", off, ids, 0.1, None, None, out) is None
    assert call.verify(x, off, ids, 0.1, None, None) is None                    # an argument short
    assert call.greedy_step(x.half(), None, out) is None
    assert call.ctc_draft(x, off, 0, 1 << 40, None, out) is None
    assert call.assemble(ids, off, ids, ids, ids, None) is None
    assert call.verify_combine(x, 4, off, ids, "0.1", None, out) is None


def test_errors_are_those_of_the_general_way():
    x, off, ids, out = _verify_inputs("cpu")
    with pytest.raises(ValueError):
        ssd.ssd_verify(x, off, ids, 0.1, out=out)                               # no host path
    with pytest.raises(TypeError):
        ssd.ssd_verify(x, off.int(), ids, 0.1, out=out)
    with pytest.raises(ValueError):
        ssd.ssd_greedy_step(x.t(), out=out)
    with pytest.raises(ValueError):
        ssd.ssd_verify_combine(x, 4, off, ids, 0.1, out=out)
    with pytest.raises(KeyError):
        ssd.ssd_verify(x, off, ids, 0.1, out={})


@pytest.mark.parametrize("broken", ["absent", "of another torch"])
def test_without_a_usable_extension_calls_go_the_general_way(monkeypatch, broken):
    monkeypatch.setattr(ssd, "_call", None)
    if broken == "absent":
        monkeypatch.setitem(sys.modules, "paper_2603_11243_b200._ssd_call", None)      # import raises
        monkeypatch.delattr(paper_2603_11243_b200, "_ssd_call", raising=False)
    else:
        monkeypatch.setattr(ssd_build, "built_for", lambda: "torch 1.0, cp30")
    x, off, ids, out = _verify_inputs("cpu")
    with pytest.warns(RuntimeWarning, match="ctypes"):
        with pytest.raises(ValueError, match="must be a CUDA tensor"):
            ssd.ssd_verify(x, off, ids, 0.1, out=out)
    with warnings.catch_warnings():
        warnings.simplefilter("error")                                           # said once
        with pytest.raises(ValueError, match="must be a CUDA tensor"):
            ssd.ssd_greedy_step(x, out=dict(out, next_token=ids))


def test_the_extension_is_rebuilt_for_another_torch(monkeypatch):
    assert not ssd_build._other_torch()
    assert ssd._native().built_for == "_ssd_call for " + ssd_build.built_for()
    monkeypatch.setattr(ssd_build, "built_for", lambda: "torch 1.0, cp30")
    assert ssd_build._other_torch()


@pytest.mark.gpu
def test_same_results_both_ways(cuda_device):
    """opts given (all automatic) is the general way.  Padded rows, V below the row's width,
    absent optional buffers, a stream of the caller's."""
    dev = cuda_device
    g = torch.Generator().manual_seed(5)
    wide = torch.randn((37, 1203), generator=g).bfloat16().to(dev)
    x = wide[:, 3:1200]
    off = torch.tensor([0, 9, 9, 37], dtype=torch.int64, device=dev)
    ids = torch.randint(0, 1000, (37,), generator=g, dtype=torch.int32).to(dev)
    skip = torch.tensor([0, 0, 1], dtype=torch.uint8, device=dev)
    side = torch.cuda.Stream(dev)
    auto = H.opts()

    def both(run):
        with torch.cuda.stream(side):
            a, b = run(None), run(auto)
        side.synchronize()
        for k in a:
            if k != "workspace":
                assert torch.equal(a[k].cpu(), b[k].cpu()), k

    side.wait_stream(torch.cuda.current_stream())
    for V in (None, 1000):
        need = ssd.ssd_verify_workspace_bytes(3, 37, V or x.shape[1], ssd.BF16)

        def zeroed(o, *drop):
            for k in drop:
                del o[k]
            for t in o.values():
                t.zero_()
            return o

        both(lambda o: ssd.ssd_verify(x, off, ids, 0.1, skip=skip, V=V, opts=o,
                                      out=zeroed(ssd.alloc_verify_outputs(37, 3, dev, need), "row_lse")))
        both(lambda o: ssd.ssd_verify_early_exit(
            x, off, ids, 0.1, V=V, opts=o,
            out=zeroed(ssd.alloc_early_exit_outputs(37, 3, V or x.shape[1], ssd.BF16, dev))))
        both(lambda o: ssd.ssd_ctc_draft(x, off, 0, 20, V=V, opts=o,
                                         out=zeroed(ssd.alloc_ctc_outputs(37, 3, dev), "draft_frames")))
        both(lambda o: {"stats": ssd.ssd_verify_shard(
            x, 5, off, ids, skip=skip, V_local=V, opts=o, stats=torch.zeros((37, 3), device=dev),
            workspace=torch.zeros((max(need, 256),), dtype=torch.uint8, device=dev))})
        ws = ssd.ssd_greedy_step_workspace_bytes(37, V or x.shape[1], ssd.BF16)
        both(lambda o: ssd.ssd_greedy_step(x, V=V, opts=o, out=dict(
            next_token=torch.zeros((37,), dtype=torch.int32, device=dev),
            workspace=torch.zeros((ws,), dtype=torch.uint8, device=dev))))
    out = ssd.alloc_verify_outputs(37, 3, dev, 16)
    with pytest.raises(ssd.SsdError) as e:
        ssd.ssd_verify(x, off, ids, 0.1, out=dict(out, workspace=out["workspace"][:16]))
    assert e.value.code == ssd.ERR_WORKSPACE


@pytest.mark.gpu
def test_every_hot_call_is_taken_and_computes_the_same(cuda_device, monkeypatch):
    """The eight functions asked directly: each answers a status, not None.  Then all eight through the
    binding, natively and with an extension that declines everything."""
    dev, B, N, M, V = cuda_device, 3, 40, 25, 700
    g = torch.Generator().manual_seed(8)
    ctc = torch.randn((N, 60), generator=g).to(dev)
    logits = torch.randn((M, V), generator=g).bfloat16().to(dev)
    f_off = torch.tensor([0, 13, 13, N], dtype=torch.int64, device=dev)
    t_off = torch.tensor([0, 9, 9, M], dtype=torch.int64, device=dev)
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32).to(dev)
    i32, f32, u8 = torch.int32, torch.float32, torch.uint8
    zeros = lambda n, t: torch.zeros((n,), dtype=t, device=dev)

    def outputs():
        o = dict(
            draft=ssd.alloc_ctc_outputs(N, B, dev), gate=dict(gate_accept=zeros(B, u8), max_entropy=zeros(B, f32)),
            verify=ssd.alloc_verify_outputs(M, B, dev, ssd.ssd_verify_workspace_bytes(B, M, V, ssd.BF16)),
            early=ssd.alloc_early_exit_outputs(M, B, V, ssd.BF16, dev),
            stats=torch.zeros((2, M, 3), dtype=f32, device=dev), combine=ssd.alloc_verify_outputs(M, B, dev, 0),
            final=dict(final_tokens=zeros(M, i32), final_len=zeros(B, i32), is_final=zeros(B, u8),
                       ar_count=zeros(1, i32), ar_utt=zeros(B, i32), ar_resume=zeros(B, i32)),
            greedy=dict(next_token=zeros(M, i32), next_logp=zeros(M, f32), row_lse=zeros(M, f32),
                        row_status=zeros(M, i32),
                        workspace=zeros(ssd.ssd_greedy_step_workspace_bytes(M, V, ssd.BF16), u8)))
        for d in o.values():
            for t in d.values() if isinstance(d, dict) else ():
                t.zero_()
        return o

    def native(o):
        call, d, a, v = ssd._native(), o["draft"], o["gate"], o["verify"]
        half, ws = V // 2, o["verify"]["workspace"]
        yield "ctc_draft", call.ctc_draft(ctc, f_off, 0, 10, None, d)
        yield "gate_from_maxima", call.gate_from_maxima(d["utt_max_entropy"], d["utt_status"], 3.6, a)
        yield "verify", call.verify(logits, t_off, ids, 0.001, a["gate_accept"], None, v)
        yield "verify_early_exit", call.verify_early_exit(logits, t_off, ids, 0.001, None, None, o["early"])
        for r in (0, 1):
            yield "verify_shard", call.verify_shard(logits[:, r * half:(r + 1) * half], r * half, t_off, ids, None,
                                                    None, o["stats"][r], ws)
        yield "verify_combine", call.verify_combine(o["stats"], V, t_off, ids, 0.001, None, o["combine"])
        yield "assemble", call.assemble(ids, t_off, a["gate_accept"], v["accepted_len"], v["all_accepted"], o["final"])
        yield "greedy_step", call.greedy_step(logits, None, o["greedy"])

    def bound(o):
        d, a, v = o["draft"], o["gate"], o["verify"]
        half, ws = V // 2, o["verify"]["workspace"]
        ssd.ssd_ctc_draft(ctc, f_off, 0, 10, out=d)
        ssd.ssd_entropy_gate_from_maxima(d["utt_max_entropy"], d["utt_status"], 3.6, out=a)
        ssd.ssd_verify(logits, t_off, ids, 0.001, skip=a["gate_accept"], out=v)
        ssd.ssd_verify_early_exit(logits, t_off, ids, 0.001, out=o["early"])
        for r in (0, 1):
            ssd.ssd_verify_shard(logits[:, r * half:(r + 1) * half], r * half, t_off, ids, stats=o["stats"][r],
                                 workspace=ws)
        ssd.ssd_verify_combine(o["stats"], V, t_off, ids, 0.001, out=o["combine"])
        ssd.ssd_assemble(ids, t_off, a["gate_accept"], v["accepted_len"], v["all_accepted"], out=o["final"])
        ssd.ssd_greedy_step(logits, out=o["greedy"])

    ways = [outputs() for _ in range(3)]
    for name, rc in native(ways[0]):
        assert rc == ssd.OK, (name, rc)
    bound(ways[1])
    monkeypatch.setattr(ssd, "_call", ssd._Declines())
    bound(ways[2])
    torch.cuda.synchronize()
    assert int(ways[0]["draft"]["draft_len"].sum()) > 0 and int(ways[0]["final"]["ar_count"]) > 0
    for way in ways[1:]:
        for part, d in ways[0].items():
            for k, t in d.items() if isinstance(d, dict) else [("", d)]:
                if k != "workspace":
                    assert torch.equal(t, way[part][k] if k else way[part]), (part, k)


@pytest.mark.gpu
def test_a_dict_that_answers_for_itself(cuda_device):
    """Result buffers in a dict subclass are whatever its item access says, not what it stores."""
    class Elsewhere(dict):
        def __getitem__(self, key):
            return other[key]

        def get(self, key, default=None):
            return other.get(key, default)

    x, off, ids, out = _verify_inputs(cuda_device)
    other = {k: torch.zeros_like(t) for k, t in out.items()}
    out["accepted_len"].fill_(-5)
    ssd.ssd_verify(x, off, ids, 0.001, out=Elsewhere(out))
    torch.cuda.synchronize()
    assert other["accepted_len"].tolist() == [6] and out["accepted_len"].tolist() == [-5]
