"""The CTA-pair dense kernel on grids whose last clusters (or all of them) own one stream of 256 query rows: the same
bits as the single-CTA kernel gives, for query tiles that fill clusters wholly, half and by one tile. (Grids of up to one
query tile per SM come here with fewer than 256 keys only.)"""
import pytest
import torch

import paper_2509_24014_b200 as sd
from paper_2509_24014_b200 import synthetic as syn
from tests.parity_util import gpu_full
from tests.test_gpu_switch_step_stats import gpu_switch_step

pytestmark = pytest.mark.gpu


def _splits(Hq, L):
    """Whether the pass that records statistics runs on the pair kernel and its last clusters are split."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles, pairs = (L + 127) // 128, sms // 2
    clusters = Hq * ((tiles + 3) // 4)
    last = clusters % pairs
    return (Hq * tiles > sms or L < 256) and 0 < 2 * last <= pairs and clusters < 2 * pairs


@pytest.mark.parametrize("Hq,Hkv,L,bs", [
    (1, 1, 128, 64), (37, 37, 192, 64), (5, 1, 224, 32), (37, 37, 128, 128),   # all clusters split (37: the most on 74 SM pairs)
    (2, 1, 640, 128), (37, 37, 512, 64),                      # up to one query tile per SM: neither of the two kernels
    (38, 38, 512, 64),                                        # none split
    (16, 4, 2944, 128), (19, 19, 2080, 32), (37, 37, 1536, 64)])   # a wave of whole clusters, then split ones
def test_same_bits_as_the_single_cta_kernel(Hq, Hkv, L, bs):
    q, k, v = syn.make_qkv(syn.AttnConfig("split", 1, Hq, Hkv, L, 128, bs, 0.3, 0, seed=95, plant_norm=6.0), "cuda")
    o, lse, _, _, _, scores = gpu_switch_step(q, k, v, bs, 0.3, 0)
    assert _splits(Hq, L) == ((Hq, L) not in ((2, 640), (37, 512), (38, 512)))
    o_plain, lse_plain = gpu_full(q, k, v)
    assert torch.equal(o, o_plain) and torch.equal(lse, lse_plain)
    assert torch.allclose(scores.double().sum(-1), torch.full_like(scores[..., 0], 1.0 / bs).double(), rtol=2e-5)


@pytest.mark.parametrize("Hq,L,bs", [(2, 640, 128), (38, 512, 64), (1, 4096, 32),   # none split
                                     (19, 2080, 32), (37, 192, 64)])               # the last clusters, all of them
def test_outputs_below_the_normal_range(Hq, L, bs):
    """V around the end of bf16's exponents, with logits that rise along the keys so that accumulators are rescaled."""
    q, k, v = syn.make_qkv(syn.AttnConfig("tiny", 1, Hq, Hq, L, 128, bs, 0.3, 0, seed=96, plant_norm=3.0), "cuda")
    k = (k * torch.linspace(0.0, 12.0, L, device="cuda")[:, None]).bfloat16()
    v = (v.abs().double() * 1e-38).bfloat16()
    assert _splits(Hq, L) == ((Hq, L) in ((19, 2080), (37, 192)))
    o = gpu_switch_step(q, k, v, bs, 0.3, 0)[0]
    o_plain, _ = gpu_full(q, k, v)
    ref = torch.softmax(q.double() @ k.double().transpose(-1, -2) / 128 ** 0.5, -1) @ v.double()
    for out in (o, o_plain):   # P in bf16 (2^-9), O in bf16: 2^-9, or half a step of 2^-133
        assert ((out.double() - ref).abs() <= ref * 2.0 ** -7 + 2.0 ** -134).all()
