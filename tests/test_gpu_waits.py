"""Every device-side wait of the library is bounded: when it runs out the kernel flags
RESPS_STATUS_WAIT_TIMEOUT, finishes its protocol and returns, and the context serves the next call.
Exercised with the test build of the library (millisecond limits; one copy can be left out so that
a wait for it really runs out) on tiny cases: a single CTA, and clusters whose CTAs wait for one another's
results.  Nothing here faults or waits without a limit: the skipped copy is simply never issued, every wait
for it gives up after about a millisecond, every copy that was issued is waited for before the CTA leaves,
and no CTA leaves while another of its cluster may still send to it."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DROP_KEY, DROP_ATTENTION_V, DROP_SCAN_CHUNK = 100, 1, 2


@pytest.fixture(scope="module")
def waitlib():
    """The binding pointed at the test build (its own shared library), restored afterwards."""
    from paper_2601_12212_b200 import binding, build
    path = build.build(wait_test=True)
    saved = (binding._lib, binding.LIB_PATH)
    binding._lib, binding.LIB_PATH = None, path
    binding.load()
    yield binding
    binding._lib, binding.LIB_PATH = saved


def _attention_inputs(binding, synth, n, Hq, Hkv, D, L, cap, T):
    rng = np.random.default_rng(4)
    q = synth.to_bf16_bits(rng.normal(size=(1, T, Hq, D)).astype(np.float32).ravel()).reshape(1, T, Hq, D)
    kc = synth.to_bf16_bits(rng.normal(size=(1, Hkv, cap, D)).astype(np.float32).ravel()).reshape(1, Hkv, cap, D)
    vc = synth.to_bf16_bits(rng.normal(size=(1, Hkv, cap, D)).astype(np.float32).ravel()).reshape(1, Hkv, cap, D)
    masks = np.zeros((1, T, 2), np.uint64)
    for i in range(n):
        masks[0, i, 0] = (1 << (i + 1)) - 1          # a chain
    return q, kc, vc, masks


def test_attention_wait_runs_out_and_the_context_recovers(waitlib):
    import oracle
    from harness import check_attention, u16_to_bf16_cuda, bf16_to_f64
    from paper_2601_12212_b200 import synth
    binding = waitlib
    n, Hq, Hkv, D, L, cap, T = 4, 4, 1, 64, 20, 64, 16       # one work item, one key tile: a single CTA has work
    ctx = binding.Context(Hq, Hkv, D, 100, max_batch=1, max_tt=T, max_k=4, max_depth=4)
    q, kc, vc, masks = _attention_inputs(binding, synth, n, Hq, Hkv, D, L, cap, T)
    steps = torch.tensor([[n, 1, 1, L]], dtype=torch.int32, device="cuda")
    nn = torch.tensor([n], dtype=torch.int32, device="cuda")
    dq, dk, dv = u16_to_bf16_cuda(q), u16_to_bf16_cuda(kc), u16_to_bf16_cuda(vc)
    dm = torch.from_numpy(masks.view(np.int64)).cuda()
    do = torch.zeros_like(dq)

    def call():
        binding.resps_tree_attention(ctx, steps, nn, 1, dq, do, None, dk, dv, Hkv * cap * D, cap * D, D, cap, dm, 0.125)

    ctx.debug_set(DROP_KEY, DROP_ATTENTION_V)     # the V tile is never fetched: whoever waits for it gives up
    call()
    torch.cuda.synchronize()                      # the call returns
    assert ctx.status() & binding.RESPS_STATUS_WAIT_TIMEOUT
    ctx.debug_set(DROP_KEY, 0)
    do.fill_(float("nan"))
    call()                                        # the same context, a complete call
    assert ctx.status() == 0
    ref = oracle.tree_attention(q[0, :n], kc[0], vc[0], L, masks[0, :n], 0.125)
    check_attention(bf16_to_f64(do)[0, :n], ref)
    ctx.close()


# A cluster of eight.  Both cases leave out the first V copy of every CTA that has key tiles in its cluster's first item.
#  meet: one group of 128 rows and nine key tiles, two a CTA: five CTAs wait for the copy; the other three have rows to
#        merge and wait for bytes that nobody sends.
#  free: four groups on two clusters.  The first item of the first cluster has 16 rows, so the CTAs without key tiles have
#        nothing to merge either: they go on to the second item, where the shared memory for it is never released.
CLUSTERS = {"meet": dict(ns=[8], Ls=[530], Hq=16, max_k=4, max_depth=4), "free": dict(ns=[2, 33], Ls=[520, 1000], Hq=8, max_k=2, max_depth=2)}


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("wait", list(CLUSTERS))
def test_cluster_waits_run_out_and_the_context_recovers(waitlib, wait, D):
    import oracle
    from harness import bf16_to_f64, check_attention, u16_to_bf16_cuda
    from paper_2601_12212_b200 import synth
    binding = waitlib
    ns, Ls, Hq, max_k, max_depth = (CLUSTERS[wait][x] for x in ("ns", "Ls", "Hq", "max_k", "max_depth"))
    B, Hkv, cap, T = len(ns), 1, 1088, 40
    ctx = binding.Context(Hq, Hkv, D, 100, max_batch=B, max_tt=T, max_k=max_k, max_depth=max_depth)
    ctx.debug_set(binding.RESPS_DEBUG_ATTN_CLUSTER, 8)
    q, kc, vc, masks = (np.concatenate(x) for x in zip(*(_attention_inputs(binding, synth, n, Hq, Hkv, D, L, cap, T)
                                                         for n, L in zip(ns, Ls))))
    steps = torch.tensor([[n, 1, 1, L] for n, L in zip(ns, Ls)], dtype=torch.int32, device="cuda")
    nn = torch.tensor(ns, dtype=torch.int32, device="cuda")
    dq, dk, dv = u16_to_bf16_cuda(q), u16_to_bf16_cuda(kc), u16_to_bf16_cuda(vc)
    dm = torch.from_numpy(masks.view(np.int64)).cuda()
    do = torch.zeros_like(dq)

    def call():
        binding.resps_tree_attention(ctx, steps, nn, B, dq, do, None, dk, dv, Hkv * cap * D, cap * D, D, cap, dm, 0.125)

    ctx.debug_set(DROP_KEY, DROP_ATTENTION_V)
    call()
    torch.cuda.synchronize()                      # the call returns
    assert ctx.status() & binding.RESPS_STATUS_WAIT_TIMEOUT
    ctx.debug_set(DROP_KEY, 0)
    do.fill_(float("nan"))
    call()                                        # the same context, a complete call
    assert ctx.status() == 0
    for b, (n, L) in enumerate(zip(ns, Ls)):
        check_attention(bf16_to_f64(do)[b, :n], oracle.tree_attention(q[b, :n], kc[b], vc[b], L, masks[b, :n], 0.125))
    ctx.close()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("Hq", [16, 14])             # Q by TMA, by plain loads
@pytest.mark.parametrize("cluster", [1, 2, 8])       # single CTAs, clusters with cut groups, one group a cluster
def test_addresses_begin_where_every_kernel_takes_them_to(waitlib, cluster, Hq, D):
    """The test build's kernels look at what their constant addresses rest on (shared memory at a multiple of 1024,
    tensor memory at column 0) and would set a status bit."""
    from harness import u16_to_bf16_cuda
    from paper_2601_12212_b200 import synth
    binding = waitlib
    n, Hkv, L, cap, T = 5, 2, 1000, 1088, 40
    ctx = binding.Context(Hq, Hkv, D, 100, max_batch=1, max_tt=T, max_k=4, max_depth=4)
    ctx.debug_set(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)
    q, kc, vc, masks = _attention_inputs(binding, synth, n, Hq, Hkv, D, L, cap, T)
    steps, nn = (torch.tensor(x, dtype=torch.int32, device="cuda") for x in ([[n, 1, 1, L]], [n]))
    dq, dk, dv = u16_to_bf16_cuda(q), u16_to_bf16_cuda(kc), u16_to_bf16_cuda(vc)
    dm, do = torch.from_numpy(masks.view(np.int64)).cuda(), torch.zeros_like(dq)
    binding.resps_tree_attention(ctx, steps, nn, 1, dq, do, None, dk, dv, Hkv * cap * D, cap * D, D, cap, dm, 0.125)
    assert ctx.status() == 0 and do[0, :n].abs().max() > 0
    ctx.close()


def test_scan_wait_runs_out_and_the_context_recovers(waitlib):
    import oracle
    binding = waitlib
    V, k = 3 * 8192, 4
    ctx = binding.Context(4, 1, 64, V, max_batch=1, max_tt=8, max_k=k, max_depth=2)
    ctx.debug_set(binding.RESPS_DEBUG_SCAN_SLICES, 1)       # one CTA walks the row's three chunks
    rng = np.random.default_rng(8)
    logits = rng.normal(size=(1, 1, 1, V)).astype(np.float32)
    i32 = dict(dtype=torch.int32, device="cuda")
    steps = torch.tensor([[5, 1, k, 0]], **i32)
    dl = torch.from_numpy(logits).cuda()
    root = torch.tensor([3], **i32)
    outs = [torch.full((1, 8), -7, **i32) for _ in range(4)]
    mask = torch.zeros(1, 8, 2, dtype=torch.int64, device="cuda")
    ret = torch.full((1, 8, 3), -7, **i32)
    nl, nn = torch.zeros(1, **i32), torch.zeros(1, **i32)

    def call():
        binding.resps_tree_expand(ctx, steps, 1, dl, V, V, V, 1, 1, root, *outs, mask, ret, nl, nn)

    ctx.debug_set(DROP_KEY, DROP_SCAN_CHUNK)      # the second chunk is never fetched
    call()
    torch.cuda.synchronize()
    assert ctx.status() & binding.RESPS_STATUS_WAIT_TIMEOUT
    ctx.debug_set(DROP_KEY, 0)
    call()
    assert ctx.status() == 0
    t = oracle.tree_expand(3, logits[0], 5, 1, k, 0, max_tt=8, ret_stride=3)
    assert int(nn[0]) == t.n_nodes == 5
    assert np.array_equal(outs[0].cpu().numpy()[0, :5], t.tokens)
    assert np.array_equal(outs[1].cpu().numpy()[0, :5], t.parent)
    ctx.close()
