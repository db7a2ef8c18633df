"""Grids of up to one query tile per SM run on a kernel of their own (one CTA to an SM, two groups of softmax warps): it
must give bitwise what the other kernels give, from the fewest tiles of keys it takes on to rings that wrap around,
whether references stay or move with every tile."""
import pytest
import torch

import paper_2509_24014_b200 as sd
from tests.parity_util import gpu_full, gpu_sparse
from tests.test_gpu_switch_step_stats import gpu_switch_step

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(H, Hkv, L, seed, rising):
    g = torch.Generator(device=DEV).manual_seed(seed)
    q = torch.randn(1, H, L, 128, generator=g, device=DEV).bfloat16()
    k, v = (torch.randn(1, Hkv, L, 128, generator=g, device=DEV).bfloat16() for _ in range(2))
    if rising:   # logits that keep outgrowing the reference
        k = (k * torch.linspace(0.2, 14.0, L, device=DEV)[:, None]).bfloat16()
    return q, k, v


@pytest.mark.parametrize("rising", [False, True])
@pytest.mark.parametrize("L", [256, 257, 300, 384, 449, 640, 700, 1473])   # 4 to 24 tiles, ragged by 1 to 63 keys
def test_dense_equals_the_kernels_of_larger_grids(L, rising):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = (L + 127) // 128
    few, many = 2 * sms // 3 // tiles, sms // tiles + 1
    q, k, v = _inputs(many, many, L, 71, rising)
    o_all, lse_all = gpu_full(q, k, v)                                           # more query tiles than SMs
    o, lse = gpu_full(*(t[:, :few].contiguous() for t in (q, k, v)))
    assert torch.equal(o, o_all[:, :few]) and torch.equal(lse, lse_all[:, :few])


@pytest.mark.parametrize("rising", [False, True])
@pytest.mark.parametrize("most", ["one", "four", "all"])   # blocks of a list at most
@pytest.mark.parametrize("bs,L", [(128, 1280), (64, 1344), (32, 1376), (32, 608), (128, 4736), (128, 8192)])
def test_sparse_equals_the_kernels_of_larger_grids(bs, L, most, rising):
    """Lists of every length, empty ones among them (128-key blocks, 4736 and 8192 tokens: more than the 32 ids fetched at
    once), and lists of a few blocks only. Copies of the same heads make up the larger grid."""
    H, Hkv, nb = (2, 1, L // bs)
    q, k, v = _inputs(H, Hkv, L, 72, rising)
    g = torch.Generator(device=DEV).manual_seed(73)
    keep = torch.rand(H, nb, nb, generator=g, device=DEV) < torch.rand(H, nb, 1, generator=g, device=DEV) * 1.3
    keep &= torch.rand(H, nb, 1, generator=g, device=DEV) < 0.9
    keep[:, 1] = False
    keep[:, 2] = True
    if most != "all":
        keep &= keep.cumsum(-1) <= {"one": 1, "four": 4}[most]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = sms // (H * ((L + 127) // 128)) + 1

    def attend(n):   # n copies of the heads
        row_ptr = torch.zeros(n * H * nb + 1, dtype=torch.int32, device=DEV)
        row_ptr[1:] = keep.repeat(n, 1, 1).sum(-1).flatten().cumsum(0)
        col_idx = keep.repeat(n, 1, 1).flatten(0, 1).nonzero()[:, 1].to(torch.int32).contiguous()
        return gpu_sparse(q.repeat(1, n, 1, 1), k.repeat(1, n, 1, 1), v.repeat(1, n, 1, 1),
                          sd.pattern_from_csr(row_ptr, col_idx, bs, nb, 1, n * H))

    o, o_many = attend(1), attend(copies)                                        # more query tiles than SMs
    assert torch.equal(o_many, o.repeat(1, copies, 1, 1))


@pytest.mark.parametrize("rising", [False, True])
@pytest.mark.parametrize("bs,L", [(32, 256), (32, 288), (32, 1376), (64, 320), (64, 1408), (128, 256), (128, 1408)])
def test_row_statistics_equal_those_of_larger_grids(bs, L, rising):
    """Block scores pooled from the statistics that the pass records (128-key ones span a tile of either group)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    few = sms // ((L + 127) // 128)
    q, k, v = _inputs(few + 2, few + 2, L, 74, rising)
    all_heads = gpu_switch_step(q, k, v, bs, 0.3, 0)
    some = gpu_switch_step(*(t[:, :few].contiguous() for t in (q, k, v)), bs, 0.3, 0)
    for i in (0, 1, 5):   # O, LSE, scores
        assert torch.equal(some[i], all_heads[i][:, :few])
