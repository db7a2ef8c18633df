"""Selection from Q and K: the one-pass routes (up to 128 and up to 512 key blocks per row), the two-pass route beyond
them, and the route with the caller's LSE, at the sizes where one ends and the next begins and on ragged query and key tiles."""
import numpy as np
import pytest
import torch

from oracle import sparsed_oracle as orc
from paper_2509_24014_b200 import synthetic as syn
from tests.parity_util import gpu_full, gpu_select, to_f64
from tests.test_gpu_parity_configs import SCORE_ATOL, SCORE_RTOL

pytestmark = pytest.mark.gpu
DEV = "cuda"


def check(q, k, bs, rho, p, lse=None):
    pat, row_ptr, col_idx, scores = gpu_select(q, k, bs, rho, p, lse=lse)
    a = scores.cpu().numpy()
    np.testing.assert_allclose(a, orc.pooled_scores(to_f64(q), to_f64(k), bs), rtol=SCORE_RTOL, atol=SCORE_ATOL)
    rp, ci = orc.select_blocks(a, bs, p, rho)          # bit-exact on its own scores
    np.testing.assert_array_equal(row_ptr.cpu().numpy(), rp)
    np.testing.assert_array_equal(col_idx.cpu().numpy(), ci)
    # the lists are the same whether the scores are written out or not
    _, _, col_idx2, _ = gpu_select(q, k, bs, rho, p, lse=lse, want_scores=False)
    assert torch.equal(col_idx, col_idx2)
    return a


@pytest.mark.parametrize("bs,nb,Hq,Hkv,batch,p_blocks", [
    (32, 1, 1, 1, 1, 0), (32, 3, 2, 1, 2, 1), (32, 127, 1, 1, 1, 60), (32, 128, 2, 2, 1, 0), (32, 129, 1, 1, 1, 7),
    (64, 1, 2, 2, 1, 0), (64, 5, 4, 2, 1, 2), (64, 128, 1, 1, 1, 31), (64, 129, 1, 1, 1, 0),
    (128, 1, 1, 1, 1, 0), (128, 3, 3, 1, 2, 1), (32, 383, 1, 1, 1, 100), (32, 385, 1, 1, 1, 9), (32, 511, 1, 1, 1, 0), (32, 512, 1, 1, 1, 77),
    (64, 200, 2, 1, 1, 64), (32, 513, 1, 1, 1, 200)])
def test_every_route_at_its_ends(bs, nb, Hq, Hkv, batch, p_blocks):
    cfg = syn.AttnConfig("routes", batch, Hq, Hkv, nb * bs, 128, bs, 0.3, p_blocks * bs, seed=71, plant_norm=6.0)
    q, k, v = syn.make_qkv(cfg, DEV)
    _, lse = gpu_full(q, k, v)
    own = check(q, k, bs, 0.3, p_blocks * bs)
    given = check(q, k, bs, 0.3, p_blocks * bs, lse=lse)
    np.testing.assert_allclose(own, given, rtol=2 * SCORE_RTOL, atol=2 * SCORE_ATOL)


def test_more_than_128_blocks_of_128_keys_sampled():
    bs, nb = 128, 130
    cfg = syn.AttnConfig("routes130", 1, 1, 1, nb * bs, 128, bs, 0.1, 0, seed=72)
    q, k, _ = syn.make_qkv(cfg, DEV)
    _, row_ptr, col_idx, scores = gpu_select(q, k, bs, 0.1, 0)
    a = scores.cpu().numpy()
    for ib in (0, 64, nb - 1):
        np.testing.assert_allclose(a[0, 0, ib], orc.head_pooled_row(to_f64(q[0, 0]), to_f64(k[0, 0]), ib, bs),
                                   rtol=SCORE_RTOL, atol=SCORE_ATOL)
    rp, ci = orc.select_blocks(a, bs, 0, 0.1)
    np.testing.assert_array_equal(col_idx.cpu().numpy(), ci)


@pytest.mark.parametrize("bs,L", [(32, 1024), (128, 1024), (32, 6016), (32, 16384)])
def test_logits_that_outgrow_the_rows_reference(bs, L):
    """The reference of a row is its first tile's maximum until a sum passes 2^60: here the logits of half the rows
    rise by about 2^100 between the first and later keys (more than once for some), those of the others fall."""
    g = torch.Generator(device=DEV).manual_seed(73)
    q = torch.randn(1, 1, L, 128, generator=g, device=DEV) * 0.05
    k = torch.randn(1, 1, L, 128, generator=g, device=DEV) * 0.05
    u = torch.randn(128, generator=g, device=DEV)
    u = u / u.norm()
    level = torch.zeros(L, device=DEV)
    level[200:], level[L // 2:], level[-500:] = 28.0, 42.0, 56.0
    q += 28.0 * u * torch.where(torch.arange(L, device=DEV) % 2 == 0, 1.0, -1.0)[None, None, :, None]
    k += u * level[None, None, :, None]      # scaled logits 28 * level / sqrt(128): 0, 69, 104, 139 (base e)
    q, k = q.bfloat16(), k.bfloat16()
    # fp32 logits of up to 139 are known to 2^-17 here (six more binades than those SCORE_RTOL is stated for)
    _, _, _, scores = gpu_select(q, k, bs, 0.3, 0)
    ref = orc.pooled_scores(to_f64(q), to_f64(k), bs)
    np.testing.assert_allclose(scores.cpu().numpy(), ref, rtol=16 * SCORE_RTOL, atol=1e-7)
