"""The streaming scan of logits rows: equal ranges of chunks that cut rows anywhere, rows of one chunk and of
many, lists that overflow (equal logits, ascending logits), fewer than k finite logits, negative zeros."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _rows(kind, n, V):
    x = (np.random.default_rng(V + n).normal(size=(n, V)) * 3).astype(np.float32)
    if kind == "equal":
        x[:] = 1.5
        x[:, ::7] = 0.0
    elif kind == "ascending":
        x = np.sort(x, axis=1)
    elif kind == "two values":
        x = np.where(x > 2.0, np.float32(0.0), np.float32(-0.0))
        x[:, V // 2] = 4.0
    elif kind == "few finite":
        keep = x > np.sort(x, axis=1)[:, -4:-3]
        x = np.where(keep, x, -np.inf).astype(np.float32)
    return x


@pytest.mark.parametrize("kind", ["normal", "equal", "ascending", "two values", "few finite"])
@pytest.mark.parametrize("V,batch,d,k,slices", [(64, 1, 1, 32, 0), (8188, 2, 3, 4, 0), (8196, 1, 4, 32, 0), (128256, 1, 2, 10, 0),
                                                (128256, 3, 6, 8, 0), (49160, 5, 8, 32, 0), (40000, 2, 3, 7, 1), (1 << 20, 1, 2, 32, 0)])
def test_rows(kind, V, batch, d, k, slices):
    from paper_2601_12212_b200 import binding
    ctx = binding.Context(8, 8, 128, V, max_batch=batch, max_tt=32, max_k=k, max_depth=d)
    ctx.debug_set(binding.RESPS_DEBUG_SCAN_SLICES, slices)
    rows = int(binding.load().resps_scan_rows(ctx.handle))
    # sequences of different depths: the rows of the batch do not start at multiples of anything
    depth = [max(1, d - s % 3) for s in range(batch)]
    x = np.stack([_rows(kind, d * k, V)] * batch).reshape(batch, d, k, V)
    x = np.ascontiguousarray(np.stack([np.roll(x[s], s, axis=1) for s in range(batch)]))
    steps = torch.tensor([[32, depth[s], k, 5] for s in range(batch)], dtype=torch.int32, device="cuda")
    logits = torch.from_numpy(x).cuda()
    val = torch.zeros(batch, rows, k, device="cuda")
    ids = torch.zeros(batch, rows, k, dtype=torch.int32, device="cuda")
    lse = torch.zeros(batch, rows, dtype=torch.float64, device="cuda")
    for _ in range(2):  # the arrival counters are left as they were found
        binding.resps_row_scan_shard(ctx, steps, batch, logits, d * k * V, k * V, V, d, k, val, ids, lse)
    assert ctx.status() == 0
    for s in range(batch):
        live = [(0, 0)] + [(j, i) for j in range(1, depth[s]) for i in range(k)]
        for r, (level, slot) in enumerate(live):
            row = x[s, level, slot] + np.float32(0.0)
            order = np.argsort(-row, kind="stable")[:k]
            assert np.array_equal(ids[s, r].cpu().numpy(), order), (s, r)
            assert np.array_equal(val[s, r].cpu().numpy(), row[order])
            m = row.max()
            want = float(m) + np.log(np.exp(row.astype(np.float64) - m).sum())
            assert abs(float(lse[s, r]) - want) < 1e-5
    ctx.close()
