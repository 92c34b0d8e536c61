"""GPU tests of the branches that the sizes of a call choose: the sweep's buffers, threshold and
segments on rows that stress them, the dense products' split of K and narrow tiles."""
import numpy as np
import pytest
import torch

from paper_2609_33390_gb300 import synth

from test_parity_gpu import _run_and_check, _to, brisk  # noqa: F401  (brisk: a fixture)

pytestmark = pytest.mark.gpu

BF16, F32 = torch.bfloat16, torch.float32


def _rows(V, kind, dtype):
    """[n, V] logits of one kind."""
    g = torch.Generator().manual_seed(V)
    x = torch.randn((5, V), generator=g)
    if kind == "sorted":          # every logit raises the threshold / none after the first does
        x = torch.sort(x, dim=1, descending=False).values
        x[1::2] = x[1::2].flip(1)
    elif kind == "masked":        # a few allowed ids, the rest at the type's lowest value
        m = torch.full_like(x, torch.finfo(dtype).min)
        for r in range(5):
            at = torch.randperm(V, generator=g)[:6 + 9 * r]
            m[r, at] = x[r, at]
        x = m
    elif kind == "infinite":      # fewer finite logits than candidates
        m = torch.full_like(x, float("-inf"))
        m[:, V // 2:V // 2 + 3] = x[:, :3]
        x = m
    elif kind == "ties":          # a handful of values
        x = torch.round(x)
    elif kind == "constant":
        x = torch.full_like(x, 1.5)
    return x.to(dtype).cuda()


@pytest.mark.parametrize("K", [4, 8, 17, 32])
@pytest.mark.parametrize("kind", ["normal", "sorted", "masked", "infinite", "ties", "constant"])
@pytest.mark.parametrize("V,dtype", [(33, BF16), (2047, BF16), (16384 + 7, BF16), (70001, BF16),
                                     (1000, F32), (8192, F32), (66000, F32)])
def test_topk_against_a_stable_sort(brisk, V, dtype, kind, K):  # noqa: F811
    """Rows shorter than one batch of one warp, of one batch a warp, and split into segments."""
    x = _rows(V, kind, dtype)
    B, L = 5, 1
    tail = brisk.DecodeTail(B, L, V, 16, K, 16, dtype, BF16, _params(V))
    got = tail.topk(x.view(B, L, V))
    torch.cuda.synchronize()
    want = torch.sort(x.float(), dim=1, descending=True, stable=True).indices[:, :K]
    assert torch.equal(got["cand_ids"].view(B, K).long(), want)
    lse = torch.logsumexp(x.double(), 1)
    # sums of V positive fp32 terms, pairwise over lanes and warps: below 20 roundings of 2^-24
    # each on the path of a term, and the logarithm's
    assert torch.allclose(got["lse_q"].view(B).double(), lse, rtol=2e-6, atol=4e-6)
    again = tail.topk(x.view(B, L, V))
    assert all(torch.equal(got[k], again[k]) for k in got)


@pytest.mark.parametrize("dtype", [BF16, F32])
@pytest.mark.parametrize("V", [1000, 16384 + 7, 70001])
@pytest.mark.parametrize("mask", [-1e4, -1e9, -1e10, -1e20, -1e30, 1e10])
def test_masked_ranges(brisk, mask, V, dtype):  # noqa: F811
    """A whole range of the vocabulary at one far value (every lane of some batches holds nothing
    else; last, every logit of a row), so that no exponential of the others is lost or spoilt."""
    g = torch.Generator().manual_seed(V)
    x = torch.randn((4, V), generator=g)
    x[0, V // 8:] = mask
    x[1, :V - 100] = mask
    x[2] = mask
    x[3, ::2] = mask
    x = x.to(dtype).cuda()
    tail = brisk.DecodeTail(4, 1, V, 16, 8, 16, dtype, BF16, _params(V))
    got = tail.topk(x.view(4, 1, V))
    torch.cuda.synchronize()
    assert tail.device_status() == brisk.OK
    want = torch.sort(x.float(), dim=1, descending=True, stable=True).indices[:, :8]
    assert torch.equal(got["cand_ids"].view(4, 8).long(), want)
    lse = torch.logsumexp(x.double(), 1)
    # as above, and the rounding of the far value's product with log2 e: an ulp of it
    assert torch.allclose(got["lse_q"].view(4).double(), lse, rtol=2e-6, atol=4e-6)


@pytest.mark.parametrize("K", [8, 32])
@pytest.mark.parametrize("rows,V,dtype", [(5, 6407, BF16), (5, 6415, BF16), (1823, 9001, BF16),
                                          (1824, 9001, BF16), (1824, 65601, BF16),
                                          (2431, 70001, BF16), (2432, 70001, BF16),
                                          (2433, 58381, BF16), (2433, 58401, BF16),
                                          (3, 3203, F32), (3, 3207, F32), (2433, 4999, F32)])
def test_layout_borders(brisk, rows, V, dtype, K):  # noqa: F811
    """Both sides of the rows and lengths at which a warp, not a CTA, takes a row."""
    g = torch.Generator("cuda").manual_seed(V + rows)
    x = torch.randn((rows, V), generator=g, device="cuda").to(dtype)
    tail = brisk.DecodeTail(rows, 1, V, 16, K, 16, dtype, BF16, _params(V))
    got = tail.topk(x.view(rows, 1, V))
    step = 512
    for s in range(0, rows, step):
        part = x[s:s + step]
        want = torch.sort(part.float(), dim=1, descending=True, stable=True).indices[:, :K]
        assert torch.equal(got["cand_ids"].view(rows, K)[s:s + step].long(), want)
        lse = torch.logsumexp(part.double(), 1)
        # sums as above
        assert torch.allclose(got["lse_q"].view(rows)[s:s + step].double(), lse, rtol=2e-6,
                              atol=4e-6)


def _params(V):
    t = torch.zeros(8, dtype=BF16, device="cuda")
    names = ("E_in", "E_out", "P_h", "P_e", "P_phi", "pos", "W0", "Wz", "Wh", "W_s", "W_c", "w_g")
    return dict({n: t for n in names}, b_g=0.0, alpha=0.0)


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


@pytest.mark.parametrize("B,L,d,r", [(1, 1, 8, 16), (1, 4, 1000, 512), (4, 1, 2000, 80), (1, 5, 96, 128),
                                     (8, 1, 128, 16), (1, 8, 136, 144), (9, 1, 40, 32)])
def test_few_row_products_parity(brisk, B, L, d, r):  # noqa: F811
    """fp32 products of 1 to 4 rows, of 5 to 8 rows up to a k of 128, and just past either. Against
    the oracle."""
    wl = synth.Workload("few", B=B, L=L, V=400, d=d, K=8, r=r, hidden_dtype=F32, agree0=0.9,
                        weight_std=0.05)
    weights = _to(synth.make_weights(wl, "cpu"), "cuda")
    block = _to(synth.make_block(wl, "cpu"), "cuda")
    rep, _ = _run_and_check(brisk, wl, weights, block)
    assert rep.max_ref_err <= 1e-3


@pytest.mark.parametrize("B,K,r", [(153, 8, 256), (305, 32, 128), (457, 16, 16), (609, 8, 64)])
def test_more_sequences_than_sms_parity(brisk, B, K, r):  # noqa: F811
    """A lone corrector of two, three and four sequences an SM, and of a wave more: the same bits as
    beside a sweep, and the oracle's results."""
    wl = synth.Workload("sequences", B=B, L=5, V=900, d=64, K=K, r=r, agree0=0.9, weight_std=0.1)
    weights = _to(synth.make_weights(wl, "cpu"), "cuda")
    block = _to(synth.make_block(wl, "cpu"), "cuda")
    rep, _ = _run_and_check(brisk, wl, weights, block, seqs=[0, B - 1])
    assert rep.max_ref_err <= 1e-3
