"""What calls leave on the library's side streams: a call that fails between its fork and its join."""
import pytest
import torch

pytestmark = pytest.mark.gpu

BF16 = torch.bfloat16


@pytest.fixture(scope="module")
def brisk():
    from paper_2609_33390_gb300 import build
    build.build()
    from paper_2609_33390_gb300 import brisk as B
    return B


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
