"""Selection from Q and K: the one-pass routes (up to 128, 384 and 512 key blocks per row), the two-pass route beyond them
and the route with the caller's LSE, each with rows ranked in the scoring kernel and by the kernel of its own, at the sizes
where one ends and the next begins and on ragged query and key tiles."""
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
    (128, 1, 1, 1, 1, 0), (128, 3, 3, 1, 2, 1), (32, 383, 1, 1, 1, 100), (32, 385, 1, 1, 1, 9), (32, 511, 1, 1, 1, 0),
    (32, 512, 1, 1, 1, 77), (64, 200, 2, 1, 1, 64), (32, 513, 1, 1, 1, 200),
    # with the LSE one group folds its sums inside its loop and the other after it: 64 n - 1 key tiles, the last ones of
    # group 0 alone
    (32, 125, 1, 1, 1, 0), (32, 126, 2, 1, 1, 31), (64, 127, 1, 1, 1, 0), (32, 254, 1, 1, 1, 0), (64, 255, 1, 1, 1, 128)])
def test_every_route_at_its_ends(bs, nb, Hq, Hkv, batch, p_blocks):
    cfg = syn.AttnConfig("routes", batch, Hq, Hkv, nb * bs, 128, bs, 0.3, p_blocks * bs, seed=71, plant_norm=6.0)
    q, k, v = syn.make_qkv(cfg, DEV)
    _, lse = gpu_full(q, k, v)
    own = check(q, k, bs, 0.3, p_blocks * bs)
    given = check(q, k, bs, 0.3, p_blocks * bs, lse=lse)
    np.testing.assert_allclose(own, given, rtol=2 * SCORE_RTOL, atol=2 * SCORE_ATOL)


@pytest.mark.parametrize("bs,nb,p_blocks", [(64, 513, 100), (64, 1024, 0), (128, 1025, 1000)])
def test_long_rows_ranked_in_the_scoring_kernel_sampled(bs, nb, p_blocks):
    """More than 512 key blocks per row: a log-sum-exp pass and a pooling pass that ranks its rows itself, or the latter
    alone with the caller's LSE."""
    cfg = syn.AttnConfig("long rows", 1, 1, 1, nb * bs, 128, bs, 0.05, p_blocks * bs, seed=75, plant_norm=6.0)
    q, k, v = syn.make_qkv(cfg, DEV)
    _, lse = gpu_full(q, k, v)
    qd, kd = to_f64(q[0, 0]), to_f64(k[0, 0])
    for given in (None, lse):
        _, row_ptr, col_idx, scores = gpu_select(q, k, bs, 0.05, p_blocks * bs, lse=given)
        a = scores.cpu().numpy()
        for ib in (0, p_blocks, nb // 2, nb - 1):
            np.testing.assert_allclose(a[0, 0, ib], orc.head_pooled_row(qd, kd, ib, bs), rtol=SCORE_RTOL, atol=SCORE_ATOL)
        rp, ci = orc.select_blocks(a, bs, p_blocks * bs, 0.05)
        np.testing.assert_array_equal(row_ptr.cpu().numpy(), rp)
        np.testing.assert_array_equal(col_idx.cpu().numpy(), ci)


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


@pytest.mark.parametrize("bs,spans,levels", [
    # one group's reference lies far below the other's, its sums above its reference
    (128, 16, {0: -140, 1: 0, 2: -100, 3: -80, 14: -90}), (32, 16, {0: -140, 1: 0, 2: -100, 3: -80, 14: -90}),
    (64, 190, {0: -140, 1: 0, 2: -100, 3: -80, 188: -90}), (128, 400, {0: -140, 1: 0, 2: -100, 3: -80, 398: -90}),
    (128, 16, {0: -140, 1: -140, 2: -100, 3: 0, 5: -80, 14: -90}), (32, 16, {0: -140, 1: -140, 2: 0, 5: -80, 7: -90}),
    (64, 190, {0: -140, 1: -140, 3: 0, 188: -90}), (128, 400, {0: -140, 1: -140, 2: -100, 3: -80, 397: 0, 398: -90}),
    # a group's reference moves by more than fp32's exponents reach below one
    (128, 16, {0: -140, 2: -100, 4: 0, 6: -110}), (32, 16, {0: -140, 2: -100, 4: 0, 6: -110}),
    (64, 190, {1: -140, 3: -100, 181: 0, 189: -110}), (128, 400, {0: -140, 386: -100, 396: 0, 398: -110})])
def test_probabilities_down_to_the_end_of_fp32(bs, spans, levels):
    """Rows whose logits (base 2) lie at a few levels, one per 128 keys: block scores down to 2^-120 keep their value and
    their rank (everything below the levels is 2^-200, which fp32 does not hold)."""
    L, per = spans * 128, 128 // bs
    x = torch.full((spans,), -200.0)
    for span, level in levels.items():
        x[span] = level
    q, k = torch.zeros(1, 1, L, 128, device=DEV), torch.zeros(1, 1, L, 128, device=DEV)
    q[..., 0], k[..., 0] = 8.0, x.repeat_interleave(128).to(DEV)   # scaled logits: 1.02 times the levels
    spans_kept = sorted(s for s in levels if levels[s] != -140)
    kept = len(spans_kept) * per
    _, _, col_idx, scores = gpu_select(q.bfloat16(), k.bfloat16(), bs, kept / (spans * per), 0)
    want = torch.tensor(spans_kept).repeat_interleave(per) * per + torch.arange(per).repeat(len(spans_kept))
    assert torch.equal(col_idx.cpu().view(-1, kept), want.to(torch.int32).expand(spans * per, kept))
    p = torch.softmax(x.double().repeat_interleave(per) * 8.0 / 128 ** 0.5, -1).numpy() / bs
    p[p < 2.0 ** -120] = 0.0
    # fp32 logits of up to 143 are known to 2^-17 (as above)
    np.testing.assert_allclose(scores[0, 0].cpu().numpy(), np.broadcast_to(p, (spans * per,) * 2),
                               rtol=16 * SCORE_RTOL, atol=2.0 ** -120)


@pytest.mark.parametrize("bs,nb,period", [(128, 32, 3), (64, 63, 3), (32, 64, 5), (128, 160, 3), (64, 400, 7),
                                          (32, 500, 9)])
def test_equal_key_blocks_rank_by_index(bs, nb, period):
    """Key blocks that hold the same keys have bitwise equal scores, wherever they lie."""
    g = torch.Generator(device=DEV).manual_seed(74)
    q = (torch.randn(1, 2, nb * bs, 128, generator=g, device=DEV) * 2).bfloat16()
    k = torch.randn(1, 2, period * bs, 128, generator=g, device=DEV).bfloat16().repeat(1, 1, -(-nb // period), 1)
    _, _, col_idx, scores = gpu_select(q, k[:, :, :nb * bs].contiguous(), bs, 0.2, 0)
    assert torch.equal(scores, scores[..., torch.arange(nb, device=DEV) % period])
    _, ci = orc.select_blocks(scores.cpu().numpy(), bs, 0, 0.2)
    np.testing.assert_array_equal(col_idx.cpu().numpy(), ci)


@pytest.mark.parametrize("bs,tiles", [(128, 24), (64, 24), (32, 24), (128, 300), (64, 300), (64, 500), (32, 250)])
@pytest.mark.parametrize("rises", [(1, 5, -4), (2, 7, -1), (3, -8, -5), (4, -6, -3)])
def test_references_that_move_at_any_tile_of_a_block(bs, tiles, rises):
    """Probabilities of 2^-200 but for three tiles of 64 keys, each 2^62 above the one before it: whatever half of a
    block or of a pair of tiles that happens in, what was summed before is kept and what is not summed yet not touched."""
    L, nb = tiles * 64, tiles * 64 // bs
    x = torch.full((tiles,), -200.0)
    for level, tile in zip((-122, -61, 0), rises):
        x[tile] = level
    q, k = torch.zeros(1, 1, L, 128, device=DEV), torch.zeros(1, 1, L, 128, device=DEV)
    q[..., 0], k[..., 0] = 8.0, x.repeat_interleave(64).to(DEV)
    _, _, _, scores = gpu_select(q.bfloat16(), k.bfloat16(), bs, 0.3, 0)
    p = torch.softmax(x.double().repeat_interleave(64) * 8.0 / 128 ** 0.5, -1).view(nb, bs).mean(-1)
    p[p < 2.0 ** -120] = 0.0
    np.testing.assert_allclose(scores[0, 0].cpu().numpy(), np.broadcast_to(p.numpy(), (nb, nb)), rtol=16 * SCORE_RTOL,
                               atol=2.0 ** -120)


@pytest.mark.parametrize("bs,nb", [(32, 64), (32, 200), (32, 500)])
@pytest.mark.parametrize("key", [0, 6, 18, 26, 31])
def test_a_key_of_nan_makes_every_score_nan(bs, nb, key):
    """Whichever way a column's exponentials are taken (with 129 to 512 key blocks per row, columns 6, 18 and 26 of 32 are
    among those that do without the exponential unit)."""
    g = torch.Generator(device=DEV).manual_seed(76)
    q, k = (torch.randn(1, 1, nb * bs, 128, generator=g, device=DEV).bfloat16() for _ in range(2))
    k[0, 0, 7 * 32 + key] = float("nan")
    _, _, col_idx, scores = gpu_select(q, k, bs, 0.2, 0)
    assert torch.isnan(scores).all()
    assert int(col_idx.min()) >= 0 and int(col_idx.max()) < nb
