"""Calls of several host threads, each on a stream and buffers of its own."""
import threading

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


def test_select_beside_tails_and_replays(brisk):
    """One corrector kernel with the shared memory that a lone call takes (132 KB) and with what a
    call beside a sweep takes (76 KB at most), and product tiles of two widths: every call succeeds
    and gives the results of a call alone, whichever thread prepared the kernel last."""
    jobs, expect, errors = [], [], []
    for r, kind in ((256, "select"), (256, "replay"), (256, "tail"), (64, "select")):
        wl = synth.Workload("threads", B=3, L=6, V=8200, d=256, K=8, r=r, agree0=0.9,
                            agree_decay=0.97)
        tail = brisk.DecodeTail.for_workload(wl, synth.make_weights(wl, "cuda"))
        tail.prepare()
        blk = synth.make_block(wl, "cuda")
        c = tail.topk(blk["logits_q"])
        call = {"select": lambda t=tail, b=blk, c=c: t.select(
                    b["hidden"], b["h_c"], b["x0"], b["logits_q"], c["cand_ids"],
                    c["cand_logprob"]),
                "replay": lambda t=tail, b=blk: t.replay(b),
                "tail": lambda t=tail, b=blk: t.tail(b)}[kind]
        jobs.append(call)
        expect.append({k: v.clone() for k, v in call().items()})
    torch.cuda.synchronize()

    def work(call, want):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for n in range(1500):
                    out = call()
                    if n % 100 == 99:
                        torch.cuda.current_stream().synchronize()
                        for k in want:
                            assert torch.equal(out[k], want[k]), k
        except Exception as e:   # noqa: BLE001 (reported by the test's own thread)
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in zip(jobs, expect)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
