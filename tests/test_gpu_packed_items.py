"""64- and 32-key blocks: a grid of more query tiles than fit on the device at once, so that CTAs take over further
tiles, with lists of very different lengths, odd unions, empty query blocks and whole runs of tiles without keys."""
import numpy as np
import pytest
import torch

import paper_2509_24014_b200 as sd
from tests.parity_util import check_outputs, gpu_sparse

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("bs,L,Hq,Hkv", [(32, 1056, 80, 16), (64, 1088, 72, 72), (32, 128, 700, 100), (64, 64, 650, 650)])
def test_ctas_that_take_over_further_tiles(bs, L, Hq, Hkv):
    nb = L // bs
    g = torch.Generator(device=DEV).manual_seed(81)
    q = (torch.randn(1, Hq, L, 128, generator=g, device=DEV) * 0.3).bfloat16()
    k = torch.randn(1, Hkv, L, 128, generator=g, device=DEV).bfloat16()
    v = torch.randn(1, Hkv, L, 128, generator=g, device=DEV).bfloat16()
    keep = torch.rand(Hq, nb, nb, generator=g, device=DEV) < torch.rand(Hq, nb, 1, generator=g, device=DEV)
    keep &= torch.rand(Hq, nb, 1, generator=g, device=DEV) < 0.8     # empty query blocks
    keep[torch.arange(Hq, device=DEV) % 7 >= 5] = False              # heads, so runs of tiles, without keys
    keep[0] = True
    counts = keep.sum(-1).flatten()
    row_ptr = torch.zeros(Hq * nb + 1, dtype=torch.int32, device=DEV)
    row_ptr[1:] = counts.cumsum(0)
    col_idx = keep.flatten(0, 1).nonzero()[:, 1].to(torch.int32).contiguous()
    o = gpu_sparse(q, k, v, sd.pattern_from_csr(row_ptr, col_idx, bs, nb, 1, Hq))
    group = Hq // Hkv
    ref = torch.zeros(1, Hq, L, 128, dtype=torch.float64, device=DEV)
    for h in range(Hq):
        s = q[0, h].double() @ k[0, h // group].double().t() / 128 ** 0.5
        mask = keep[h].repeat_interleave(bs, 0).repeat_interleave(bs, 1)
        p = torch.softmax(s.masked_fill(~mask, -float("inf")), -1).nan_to_num(0.0)   # no keys: zeros
        ref[0, h] = p @ v[0, h // group].double()
    ref = ref.cpu().numpy()
    # rows over few keys reach |O| of 4: bf16 rounding alone is 2^-9 of that, the stated 2e-2 is for |O| up to 1
    scale = max(1.0, float(np.abs(ref).max()))
    check_outputs(o.float() / scale, ref / scale, f"block {bs}")
    assert (o[0, 5] == 0).all()


@pytest.mark.parametrize("bs,kept", [(32, (1, 5, 20, 13)), (32, (7, 0, 2, 31)), (64, (3, 16)), (128, (8,))])
def test_lists_that_end_at_the_last_index_of_32_bits(bs, kept):
    """The lists of one query tile as the last entries of a col_idx of 2^31 - 1."""
    L = 32 * bs
    nb, rows, last = 32, 128 // bs, 2 ** 31 - 1
    g = torch.Generator(device=DEV).manual_seed(82)
    q, k, v = (torch.randn(1, 1, L, 128, generator=g, device=DEV).bfloat16() for _ in range(3))
    ids = torch.cat([torch.randperm(nb, generator=g, device=DEV)[:n].sort().values for n in kept]).to(torch.int32)
    ends = torch.zeros(nb + 1, dtype=torch.int64, device=DEV)
    ends[nb - rows + 1:] = torch.tensor(kept, device=DEV).cumsum(0)     # only the last query tile keeps anything
    row_ptr = ends.to(torch.int32)
    want = gpu_sparse(q, k, v, sd.pattern_from_csr(row_ptr, ids, bs, nb, 1, 1))
    col_idx = torch.empty(last, dtype=torch.int32, device=DEV)
    col_idx[last - ids.numel():] = ids
    row_ptr_last = (ends + (last - ids.numel())).to(torch.int32)
    got = gpu_sparse(q, k, v, sd.pattern_from_csr(row_ptr_last, col_idx, bs, nb, 1, 1))
    assert torch.equal(got, want) and bool((want[0, 0, -128:] != 0).any())
