"""Selection from the row statistics at the edges of its reading: a warp takes eight key blocks at a time and four warps 32,
so one block, one short of and one beyond both, and query tiles that are not full."""
import numpy as np
import pytest

from oracle import sparsed_oracle as orc
from paper_2509_24014_b200 import synthetic as syn
from tests.parity_util import to_f64
from tests.test_gpu_parity_configs import SCORE_ATOL, SCORE_RTOL
from tests.test_gpu_switch_step_stats import gpu_switch_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bs", [32, 64, 128])
@pytest.mark.parametrize("nb", [1, 7, 8, 9, 31, 32, 33, 65])
def test_block_counts_around_a_batch(bs, nb):
    q, k, v = syn.make_qkv(syn.AttnConfig("edges", 1, 2, 1, nb * bs, 128, bs, 0.3, 0, seed=61, plant_norm=6.0), "cuda")
    _, _, _, row_ptr, col_idx, scores = gpu_switch_step(q, k, v, bs, 0.3, 0)
    a = scores.cpu().numpy()
    np.testing.assert_allclose(a, orc.pooled_scores(to_f64(q), to_f64(k), bs), rtol=SCORE_RTOL, atol=SCORE_ATOL)
    rp, ci = orc.select_blocks(a, bs, 0, 0.3)          # bit-exact on its own scores
    np.testing.assert_array_equal(row_ptr.cpu().numpy(), rp)
    np.testing.assert_array_equal(col_idx.cpu().numpy(), ci)
