"""Kernels of grids that fit on the device at once are launched so that they may start before the one before them has
ended: chains in which each call reads what the one before it wrote, eagerly, on another stream and as a graph, must
equal the same chain with the device waited for after every call."""
import pytest
import torch

import paper_2509_24014_b200 as sd
from paper_2509_24014_b200 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bs,L", [(32, 96), (64, 448), (128, 640)])
def test_chains_of_dependent_calls(bs, L):
    B, H, dev = 2, 2, "cuda"
    q, k, v = syn.make_qkv(syn.AttnConfig("chain", B, H, H, L, 128, bs, 0.4, 0, seed=91), dev)
    params = sd.make_params(bs, 0.4, 0)
    kp, kg = sd.sparsed_kept_per_row(params, L)
    ws = sd.new_workspace(sd.sparsed_workspace_bytes(sd.OP_SELECT_PATTERN, sd.make_shape(q, k), params), dev)
    pat, row_ptr, col_idx = sd.new_pattern(B, H, L // bs, kp + kg, dev)
    o = [torch.empty_like(q) for _ in range(2)]

    def chain(wait):
        col_idx.zero_()
        x = q
        for i in range(6):
            for call in (lambda: sd.sparsed_select_pattern(x, k, params, pat, ws),      # rewrites the lists ...
                         lambda: sd.sparsed_attn_sparse(x, k, v, o[0], pat, ws),        # ... that this walks
                         lambda: sd.sparsed_attn_full(o[0], k, v, o[1], None, ws)):
                call()
                if wait:
                    torch.cuda.synchronize()
            x = o[1]
        return o[0].clone(), o[1].clone(), col_idx.clone()

    want = chain(True)
    for _ in range(20):
        assert all(torch.equal(a, b) for a, b in zip(chain(False), want))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        got = chain(False)
        s.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            got = chain(False)
    for _ in range(5):
        for t in got:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert sd.sparsed_last_device_status(ws) == (0, 0)
