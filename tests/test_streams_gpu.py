"""What calls leave on the library's side streams: replay diagnostics under capture and beside a
caller's own capture of a tail, and a call that fails between its fork and its join."""
import pytest
import torch

from paper_2609_33390_gb300 import synth

pytestmark = pytest.mark.gpu

BF16 = torch.bfloat16


@pytest.fixture(scope="module")
def brisk():
    from paper_2609_33390_gb300 import build
    build.build()
    from paper_2609_33390_gb300 import brisk as B
    return B


def _workload(brisk, **kw):
    wl = synth.Workload("streams", agree0=0.9, agree_decay=0.97, weight_std=0.2, **kw)
    tail = brisk.DecodeTail.for_workload(wl, synth.make_weights(wl, "cuda"))
    tail.prepare()
    return tail, synth.make_block(wl, "cuda")


@pytest.mark.parametrize("kw", [dict(B=2, L=8, V=4099), dict(B=16, L=32, V=64003),
                                dict(B=80, L=32, V=32000)])
def test_captured_replay_matches_direct_calls(brisk, kw):
    """A captured call stays on its stream, so this also compares the direct call's concurrent
    sweeps, of up to 160 MB each, with the same work in order."""
    tail, blk = _workload(brisk, d=256, K=8, r=64, **kw)
    direct = [tail.replay(blk) for _ in range(3)]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = tail.replay(blk)
    for _ in range(2):
        for v in out.values():
            v.zero_()
        g.replay()
        torch.cuda.synchronize()
        for d in direct:
            for k in out:
                assert torch.equal(out[k], d[k]), k
    assert tail.device_status() == brisk.OK


def test_replay_while_a_caller_captures_a_tail(brisk):
    """The capture owns the side streams until it ends; a replay on another stream goes on without
    them and leaves it whole."""
    tail, blk = _workload(brisk, B=4, L=16, V=20011, d=128, K=8, r=32)
    other, blk2 = _workload(brisk, B=3, L=8, V=9001, d=128, K=8, r=32)
    want, want2 = tail.tail(blk), other.replay(blk2)
    out = tail.alloc_outputs()
    torch.cuda.synchronize()
    stream, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        tail.tail(blk, out=out)
        with torch.cuda.stream(stream):
            got2 = other.replay(blk2)
    torch.cuda.synchronize()
    assert all(torch.equal(got2[k], want2[k]) for k in want2)
    g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(out[k], want[k]) for k in want)
    again = other.replay(blk2)
    torch.cuda.synchronize()
    assert all(torch.equal(again[k], want2[k]) for k in want2)


def test_a_failed_tail_is_joined(brisk):
    """The verification of 2^24 ids needs more shared memory than a block may have, which the host
    finds after the other stages have been enqueued: what follows on the caller's stream still comes
    after them (a hidden product of k = 2^20 among them, which takes the longest)."""
    L, V, d, K, r = 2, 1 << 24, 1 << 20, 4, 16
    t = torch.zeros(8, dtype=BF16, device="cuda")
    names = ("E_in", "E_out", "P_e", "P_phi", "pos", "W0", "Wz", "Wh", "W_s", "W_c", "w_g")
    w = dict({n: t for n in names}, P_h=torch.full((r, d), 0.01, dtype=BF16, device="cuda"),
             b_g=0.0, alpha=0.0)
    tail = brisk.DecodeTail(1, L, V, d, K, r, BF16, BF16, w)
    tail.tables.zero_()
    blk = {"hidden": torch.ones((1, L, d), dtype=BF16, device="cuda"),
           "h_c": torch.ones((1, d), dtype=BF16, device="cuda"),
           "x0": torch.zeros(1, dtype=torch.int32, device="cuda"),
           "logits_q": torch.randn((1, L, V), device="cuda").to(BF16),
           "logits_p": torch.randn((1, L, V), device="cuda").to(BF16)}
    for _ in range(3):   # (the first call loads the kernels, which takes longer than they run)
        tail.workspace.zero_()
        torch.cuda.synchronize()
        with pytest.raises(brisk.BriskError):
            tail.tail(blk)
        after = tail.workspace.clone()
        torch.cuda.synchronize()
        assert torch.equal(after, tail.workspace)
