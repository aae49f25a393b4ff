"""Attention over more K/V buffers than the context's table of tensor maps holds: when a call's own maps make the
table start anew, the call still uses the right ones.  (Forward error of bf16 inputs and a bf16 result, fp32 sums:
2^-9 of the largest output, doubled.)"""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_more_buffers_than_maps_are_kept():
    from paper_2601_12212_b200 import binding
    calls, D, cap, n = 2060, 64, 64, 4  # two maps a call and one of Q: the table of 4096 is full within call 2048
    ctx = binding.Context(1, 1, D, 64, max_batch=1, max_tt=n, max_k=2, max_depth=2)
    gen = torch.Generator(device="cuda").manual_seed(5)
    flat = torch.randn(2 * calls * 8 + cap * D, generator=gen, device="cuda", dtype=torch.bfloat16)
    q = torch.randn(1, n, 1, D, generator=gen, device="cuda", dtype=torch.bfloat16)
    out = torch.zeros(calls, 1, n, 1, D, device="cuda", dtype=torch.bfloat16)
    steps = torch.tensor([[n, 2, 2, 20]], dtype=torch.int32, device="cuda")
    nodes = torch.tensor([n], dtype=torch.int32, device="cuda")
    mask = torch.tensor([[[2 ** (i + 1) - 1, 0] for i in range(n)]], dtype=torch.int64, device="cuda")
    views = [flat[8 * i:8 * i + cap * D] for i in range(2 * calls)]
    for i in range(calls):
        binding.resps_tree_attention(ctx, steps, nodes, 1, q, out[i], None, views[2 * i], views[2 * i + 1], cap * D, cap * D, D,
                                     cap, mask, 1 / math.sqrt(D))
    assert ctx.status() == 0
    seen = torch.ones(n, 20 + n, dtype=torch.bool, device="cuda")
    seen[:, 20:] = torch.tril(seen[:, 20:])
    for i in list(range(0, calls, 97)) + list(range(2040, calls)):
        k, v = (views[j].view(cap, D)[:20 + n].float() for j in (2 * i, 2 * i + 1))
        p = (q[0, :, 0].float() @ k.T / math.sqrt(D)).masked_fill(~seen, float("-inf")).softmax(-1)
        want = p @ v
        assert (out[i, 0, :, 0].float() - want).abs().max() <= 2 ** -8 * want.abs().max()
    ctx.close()
