"""GPU tests of the branches that the sizes of a call choose: the dense products' split of K and
narrow tiles."""
import numpy as np
import pytest
import torch

from paper_2609_33390_gb300 import synth

from test_parity_gpu import _run_and_check, _to, brisk  # noqa: F401  (brisk: a fixture)

pytestmark = pytest.mark.gpu

BF16, F32 = torch.bfloat16, torch.float32


@pytest.mark.parametrize("dtype", [BF16, F32])
@pytest.mark.parametrize("B,L,d,r", [(1, 3, 512, 16), (2, 5, 2048, 48), (3, 43, 1024, 80),
                                     (9, 15, 1000, 272), (2, 2, 8, 112)])
def test_split_products_parity(brisk, dtype, B, L, d, r):  # noqa: F811
    """Hidden products whose K is split over a cluster: tiles of fewer than 64 columns, a last tile
    that reaches past the product, 1 to 135 rows, one K step and K that no step divides. Against
    the oracle; twice the same bits."""
    wl = synth.Workload("split", B=B, L=L, V=400, d=d, K=8, r=r, hidden_dtype=dtype, agree0=0.9,
                        weight_std=0.02)
    weights = _to(synth.make_weights(wl, "cpu"), "cuda")
    block = _to(synth.make_block(wl, "cpu"), "cuda")
    rep, g = _run_and_check(brisk, wl, weights, block, seqs=[0, B - 1])
    _, g2 = _run_and_check(brisk, wl, weights, block, seqs=[])
    assert rep.max_ref_err <= 1e-3
    for k in g:
        np.testing.assert_array_equal(g[k], g2[k], err_msg=k)
