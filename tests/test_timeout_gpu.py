"""A bounded device-side wait that runs out (failure detection without a GPU fault).

The tensor-core products wait on mbarriers for their TMA loads and tensor-core operations; each
wait gives up after a limit of SM cycles; so do the corrector's waits for its candidates' table
rows. A limit of one cycle makes the first wait whose data is
still arriving give up (a TMA load from memory takes far longer): the call must report
BRISK_ERR_TIMEOUT through the device status, drain what it started, leave the context usable,
and the next call with the default limit must return the same results as before."""
import pytest
import torch

from paper_2609_33390_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def brisk():
    from paper_2609_33390_gb300 import build
    build.build()
    from paper_2609_33390_gb300 import brisk as B
    return B


def test_expired_wait_reports_timeout_and_the_next_call_is_correct(brisk):
    wl = synth.Workload("timeout", B=2, L=16, V=2048, d=4096, K=8, r=64, agree0=0.9,
                        agree_decay=0.97)
    w = synth.make_weights(wl, "cuda")
    blk = synth.make_block(wl, "cuda")
    tail = brisk.DecodeTail.for_workload(wl, w)
    tail.prepare()
    c = tail.topk(blk["logits_q"])
    args = (blk["hidden"], blk["h_c"], blk["x0"], blk["logits_q"], c["cand_ids"],
            c["cand_logprob"])
    ref = tail.select(*args)
    torch.cuda.synchronize()
    assert tail.device_status() == brisk.OK
    prev = brisk.set_wait_limit(1)
    try:
        tail.select(*args)
        torch.cuda.synchronize()
        assert tail.device_status() == brisk.ERR_TIMEOUT
    finally:
        brisk.set_wait_limit(prev)
    again = tail.select(*args)
    torch.cuda.synchronize()
    assert tail.device_status() == brisk.OK
    assert torch.equal(again["sel_tokens"], ref["sel_tokens"])
    assert torch.equal(again["refined"], ref["refined"])


@pytest.mark.parametrize("kw", [dict(V=4096), dict(V=4096, L=5), dict(V=20011)])
def test_expired_wait_of_the_corrector(brisk, kw):
    """fp32 weights: the products have no bounded wait, so the status is the corrector's. Its ring
    of two stages of 80 KB fills more slowly than a position is computed, so that a stage is asked
    for again while its earlier rows are still arriving. V = 20011: verifying in the same CTA."""
    size = dict(B=4, L=24, d=64, K=16, r=512, agree0=0.9, agree_decay=0.97)
    size.update(kw)
    wl = synth.Workload("timeout_corrector", logits_dtype=torch.float32,
                        hidden_dtype=torch.float32, **size)
    w = synth.make_weights(wl, "cuda")
    blk = synth.make_block(wl, "cuda")
    tail = brisk.DecodeTail.for_workload(wl, w)
    tail.prepare()
    ref, rep = tail.tail(blk), tail.replay(blk)
    torch.cuda.synchronize()
    assert tail.device_status() == brisk.OK
    for call in (lambda: tail.tail(blk), lambda: tail.replay(blk)):
        prev = brisk.set_wait_limit(1)
        try:
            call()
            torch.cuda.synchronize()
            assert tail.device_status() == brisk.ERR_TIMEOUT
        finally:
            brisk.set_wait_limit(prev)
        again, rep2 = tail.tail(blk), tail.replay(blk)
        torch.cuda.synchronize()
        assert tail.device_status() == brisk.OK
        assert all(torch.equal(again[k], ref[k]) for k in ref)
        assert all(torch.equal(rep2[k], rep[k]) for k in rep)
