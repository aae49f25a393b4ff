"""The controller step at the edges of its split: hidden units and actions that do not divide by the cluster,
fewer units than CTAs, more actions than threads, features in several parts, unaligned or odd rows."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("temperature", [0.0, 0.7])
@pytest.mark.parametrize("B,W,H,A,shift", [(1, 8, 1, 1, 0), (2, 40, 5, 7, 0), (3, 77, 100, 180, 0), (2, 4096, 64, 513, 0),
                                           (1, 5504, 256, 1024, 0), (2, 6002, 129, 600, 1), (17, 128, 128, 180, 2)])
def test_one_step(B, W, H, A, shift, temperature):
    from paper_2601_12212_b200 import binding
    g = torch.Generator(device="cuda").manual_seed(W + H)
    r = dict(generator=g, device="cuda")
    F = 3 * W
    w1 = torch.empty(H * F + shift, device="cuda")[shift:].view(H, F)   # (16-byte aligned or not)
    w1.copy_(torch.randn(H, F, **r) / F ** 0.5)
    w = [w1, 0.1 * torch.randn(H, **r), torch.randn(H, H, **r) / H ** 0.5, 0.1 * torch.randn(H, **r),
         0.5 * torch.randn(A, H, **r), 0.1 * torch.randn(A, **r)]
    actions = torch.arange(3 * A, dtype=torch.int32, device="cuda").view(A, 3)
    flat = [torch.randn(B * (W + shift) + shift, **r).to(torch.bfloat16)[shift:] for _ in range(3)]
    hid = [h.view(B, W + shift)[:, :W] for h in flat]
    u = torch.rand(B, dtype=torch.float64, **r)
    ctx = binding.Context(8, 2, 128, 1000, max_batch=B, max_tt=128, max_k=32, max_depth=8)
    i32 = dict(dtype=torch.int32, device="cuda")
    state, steps = torch.zeros(B, 4, **i32), torch.tensor([[1, 1, 1, 100 + s] for s in range(B)], **i32)
    state[B - 1] = torch.tensor([1, 0, 0, 2], **i32)                    # the last one keeps its action, if not alone
    if B == 1:
        state.zero_()
    reward, logits, action = torch.zeros(B, device="cuda"), torch.zeros(B, A, device="cuda"), torch.zeros(B, **i32)
    binding.resps_controller_step(ctx, binding.make_policy(*w, actions), *flat, W + shift, B, 4, temperature, u, None, None,
                                  state, steps, reward, logits, action)
    assert ctx.status() == 0
    x = torch.cat([h.double() for h in hid], 1)
    h2 = torch.tanh(torch.tanh(x @ w[0].double().T + w[1]) @ w[2].double().T + w[3])
    want = (h2 @ w[4].double().T + w[5]).cpu().numpy()
    for s in range(B if B == 1 else B - 1):
        np.testing.assert_allclose(logits[s].cpu().numpy(), want[s], atol=3e-4)
        z = logits[s].cpu().numpy().astype(np.float64)
        if temperature:
            p = np.cumsum(np.exp((z - z.max()) / np.float64(np.float32(temperature))))
            choice = min(A - 1, int(np.searchsorted(p, float(u[s]) * p[-1], side="right")))
        else:
            choice = int(z.argmax())
        assert int(action[s]) == choice == int(state[s, 1]) and int(state[s, 0]) == 1
        assert steps[s].tolist() == [3 * choice, 3 * choice + 1, 3 * choice + 2, 100 + s]
    if B > 1:
        assert state[B - 1].tolist() == [2, 0, 0, 2] and steps[B - 1].tolist() == [1, 1, 1, 100 + B - 1]
    ctx.close()
