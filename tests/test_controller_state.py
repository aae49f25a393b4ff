"""A sequence's controller state is written by its own cluster while the next sequence's cluster looks at two words of
it, in no order (csrc/controller.cu).  What is seen may only steer a prefetch: the text is held to that, and on the GPU
the outcome of a sequence does not depend on what its neighbours do."""
import os
import re

import pytest
import torch

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_12212_b200", "csrc", "controller.cu")


def test_the_neighbours_state_only_steers_the_prefetch():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    assert set(re.findall(r"a\.state\[((?:[^][]|\[[^]]*\])*)\]", text)) == {"b", "max(b - 1, 0)"}
    lines = [x.strip() for x in text.splitlines() if re.search(r"\bbeside\b", x)]
    assert lines == ["const resps_controller_state st = a.state[b], beside = a.state[max(b - 1, 0)];",
                     "if (f0 == 0 && vec_w && !(b > 0 && (beside.cache_step == 0 || beside.action < 0))) {"]
    block = text[text.index(lines[1]):]
    block = block[:block.index("if (vec_h)")]
    assert "prefetch" in block


@pytest.mark.gpu
def test_a_sequence_does_not_depend_on_its_neighbours():
    from paper_2601_12212_b200 import binding
    B, W, H, A = 7, 512, 128, 60
    r = dict(generator=torch.Generator(device="cuda").manual_seed(9), device="cuda")
    i32 = dict(dtype=torch.int32, device="cuda")
    w = [torch.randn(H, 3 * W, **r) / (3 * W) ** 0.5, torch.randn(H, **r), torch.randn(H, H, **r) / H ** 0.5, torch.randn(H, **r),
         torch.randn(A, H, **r), torch.randn(A, **r), torch.randint(1, 9, (A, 3), **r).to(torch.int32)]
    hid = [torch.randn(B, W, dtype=torch.bfloat16, **r) for _ in range(3)]
    u = torch.rand(B, dtype=torch.float64, **r)
    # asks: never asked, cache step 0; keeps: steps 1 and 3 (the last of the interval)
    start = torch.tensor([[0, -1, 0, 0], [1, 3, 0, 1], [0, 5, 0, 0], [3, 2, 0, 3], [0, 7, 0, 0], [0, -1, 0, 0], [2, 1, 0, 2]], **i32)

    def run(rows):
        n = len(rows)
        ctx = binding.Context(8, 2, 128, 1000, max_batch=n, max_tt=128, max_k=32, max_depth=8)
        pol = binding.make_policy(*w)
        state, steps = start[rows].clone(), torch.tensor([[1, 1, 1, 100 + i] for i in rows], **i32)
        reward, logits, action = torch.zeros(n, device="cuda"), torch.zeros(n, A, device="cuda"), torch.zeros(n, **i32)
        for _ in range(6):
            binding.resps_controller_step(ctx, pol, *[h[rows].contiguous() for h in hid], W, n, 4, 1.0, u[rows].contiguous(),
                                          None, None, state, steps, reward, logits, action)
        assert ctx.status() == 0
        ctx.close()
        return state, steps, reward, logits, action

    together = run(list(range(B)))
    for b in range(B):
        assert all(torch.equal(x[b:b + 1], y) for x, y in zip(together, run([b])))
