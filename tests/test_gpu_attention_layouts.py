"""The ways a layer's attention is laid out (clusters of every size; equal splits in one round of items and in
several; ranges over all groups), forced by the test-only overrides on shapes where each can go wrong: more CTAs than key
tiles, groups whose size does not divide a row tile, a single token, fewer groups than clusters and more."""
import pytest

from test_gpu_edges import _attention_case, _imports

pytestmark = pytest.mark.gpu

SHAPES = [dict(n=7, Hq=12, Hkv=4, D=64, L=5), dict(n=33, Hq=14, Hkv=2, D=128, L=447),
          dict(n=[1, 90, 3], Hq=8, Hkv=8, D=128, L=[0, 1400, 63], B=3),
          dict(n=[20, 128], Hq=16, Hkv=4, D=128, L=[5, 1400], B=2)]  # a cluster: a short item, then a long one


@pytest.mark.parametrize("cluster,equal_splits", [(1, 0), (1, 1000), (2, None), (3, None), (4, None), (6, None), (8, None), (5, None), (7, None)])
@pytest.mark.parametrize("shape", range(len(SHAPES)))
def test_layouts(shape, cluster, equal_splits):
    _, binding, _ = _imports()
    debug = [(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)]
    if equal_splits is not None:
        debug.append((binding.RESPS_DEBUG_ATTN_SINGLE, equal_splits))
    _attention_case(**SHAPES[shape], cap=1664, seed=cluster, poison=True, debug=debug)


@pytest.mark.parametrize("n,Hq,Hkv,L,B", [(12, 16, 2, 900, 1), (1, 8, 1, 2000, 1), ([30, 3], 8, 2, [1000, 700], 2)])
def test_ranges_over_fewer_tiles_than_ctas(n, Hq, Hkv, L, B):
    """15 to 32 key tiles a group, a few groups: most of the 148 CTAs have no range."""
    _, binding, _ = _imports()
    debug = [(binding.RESPS_DEBUG_ATTN_CLUSTER, 1), (binding.RESPS_DEBUG_ATTN_SINGLE, 0)]
    _attention_case(n, Hq, Hkv, 128, L, cap=2048, seed=B, B=B, poison=True, debug=debug)


TILES = [dict(n=[43, 128, 1, 86], Hq=24, Hkv=8, D=128, L=[1000, 63, 1500, 0], B=4),  # 2 row tiles (the second of 1 row), 3, 1, 3
         dict(n=96, Hq=14, Hkv=2, D=64, L=1400),                                      # 6, Q by plain loads
         dict(n=[128, 65, 2, 20], Hq=16, Hkv=1, D=128, L=[130, 1, 5, 1536], B=4)]     # 16, 9, 1, 3


@pytest.mark.parametrize("rounds", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", range(len(TILES)))
def test_equal_splits_in_rounds(shape, rounds):
    _, binding, _ = _imports()
    debug = [(binding.RESPS_DEBUG_ATTN_CLUSTER, 1), (binding.RESPS_DEBUG_ATTN_SINGLE, 1), (binding.RESPS_DEBUG_ATTN_EVEN_ROUNDS, rounds)]
    for cut_for in (0, 12):  # all CTAs; a twelfth of them, so that the rounds are full
        _attention_case(**TILES[shape], cap=1664, seed=rounds, poison=True, debug=debug + [(binding.RESPS_DEBUG_ATTN_ROUNDS, cut_for)])


# Small trees under a context that builds large ones: fewer groups than clusters, so a group is cut over several.
SMALL = [dict(n=5, Hq=16, Hkv=2, D=128, L=1400),                          # 2 groups, 8 clusters
         dict(n=1, Hq=32, Hkv=8, D=64, L=1023),
         dict(n=[5, 18], Hq=16, Hkv=1, D=128, L=[100, 1480], B=2),        # 4 groups of very different lengths
         dict(n=[3, 1, 16, 33], Hq=14, Hkv=2, D=128, L=[0, 7, 640, 1000], B=4),
         dict(n=2, Hq=8, Hkv=1, D=128, L=60)]                             # fewer key tiles than CTAs


@pytest.mark.parametrize("cluster", [2, 3, 4, 6, 8, 5, 7])
@pytest.mark.parametrize("shape", range(len(SMALL)))
def test_a_group_cut_over_several_clusters(shape, cluster):
    _, binding, _ = _imports()
    debug = [(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster), (binding.RESPS_DEBUG_ATTN_SINGLE, 1)]  # cut wherever clusters are left
    _attention_case(**SMALL[shape], cap=1664, seed=shape, poison=True, debug=debug)


def test_cut_groups_keep_values_beyond_fp16():
    _, binding, _ = _imports()
    _attention_case(6, 16, 2, 128, 3000, cap=3200, seed=3, v_scale=3.0e5, debug=[(binding.RESPS_DEBUG_ATTN_CLUSTER, 4)])


@pytest.mark.parametrize("cluster", [5, 7])
def test_groups_cut_over_uneven_clusters_keep_values_beyond_fp16(cluster):
    """The 32 chunks of a partial in shares of 7 and 6, of 5 and 4; two groups in four pieces each."""
    _, binding, _ = _imports()
    _attention_case(6, 16, 2, 128, 4000, cap=4200, seed=cluster, v_scale=3.0e5, debug=[(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)])


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("cluster", [2, 3, 5, 7, 8])
def test_clusters_with_several_items(cluster, D):
    """Trees larger than the context's limits: a cluster takes row tile after row tile, its CTAs' staging is used again
    (full tiles, a tile of 4 rows, a group of a single key tile, which one CTA of the cluster does alone)."""
    _, binding, _ = _imports()
    debug = [(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)]
    _attention_case(n=[128, 33, 3], Hq=8, Hkv=2, D=D, L=[700, 1100, 20], B=3, cap=1280, seed=cluster, poison=True, debug=debug, max_k=2,
                    max_depth=2)
    _attention_case(n=[90, 19], Hq=7, Hkv=1, D=D, L=[300, 64], B=2, cap=448, seed=cluster, poison=True, debug=debug, max_k=2, max_depth=2)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("cluster", [2, 3, 4, 8])
def test_few_key_tiles_in_a_cluster(cluster, D):
    """One to nine key tiles: up to five stay in one CTA; six to eight are a tile a CTA in a cluster of eight, with two,
    one and no CTAs left over, and more a CTA in smaller ones; nine take five CTAs of eight, two each.  The last tile
    full and with a single key."""
    _, binding, _ = _imports()
    for tiles in range(1, 10):
        for last in (1, 64):
            n = 9 if tiles > 1 else 1
            _attention_case(n, 16, 2, D, 64 * (tiles - 1) + last - n, cap=640, seed=tiles, poison=True,
                            debug=[(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)])


@pytest.mark.parametrize("least", [1, 4, 1000])
@pytest.mark.parametrize("cluster", [1, 3, 8])
def test_fewest_key_tiles_of_a_cta(cluster, least):
    """Shares of at least so many key tiles, up to whole groups in one CTA (3, 9 and 23 key tiles; in clusters and in equal
    splits).  Results do not depend on it."""
    _, binding, _ = _imports()
    debug = [(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster), (binding.RESPS_DEBUG_ATTN_MIN_TILES, least)]
    if cluster == 1:
        debug.append((binding.RESPS_DEBUG_ATTN_SINGLE, 1))
    _attention_case(n=[9, 33, 70], Hq=14, Hkv=2, D=128, L=[130, 520, 1400], B=3, cap=1536, seed=least, poison=True, debug=debug)


@pytest.mark.parametrize("cluster", [2, 3, 6, 8])
@pytest.mark.parametrize("n,Hq", [(5, 12), (60, 16)])
def test_clusters_keep_values_beyond_fp16(n, Hq, cluster):
    _, binding, _ = _imports()
    _attention_case(n, Hq, 4, 128, 900, cap=1024, seed=cluster, v_scale=3.0e5, debug=[(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)])


@pytest.mark.parametrize("cap", [1216, 9408])
@pytest.mark.parametrize("n", [12, 40, 128])
def test_trees_of_one_context_in_caches_with_and_without_room(n, cap):
    """The paper's largest action bounds the context; short and long prefixes, small trees and the largest."""
    for L in (1000, cap - 128):
        _attention_case(n, 32, 8, 128, L, cap=cap, seed=n, poison=True, max_k=32, max_depth=8)


def test_replayed_for_small_and_large_trees():
    """One capture of three layers, replayed while the tree shrinks and grows under it: groups are cut, whole and cut
    again.  (bf16 result of fp32 sums: 2^-9 of the largest output, doubled.)"""
    import math

    import torch
    _, binding, _ = _imports()
    hq, hkv, D, cap, T, NL = 32, 8, 128, 6016, 128, 3
    ctx = binding.Context(hq, hkv, D, 1000, max_batch=1, max_tt=T, max_k=32, max_depth=8)
    r = dict(generator=torch.Generator(device="cuda").manual_seed(8), device="cuda", dtype=torch.bfloat16)
    q, k, v = torch.randn(NL, 1, T, hq, D, **r), torch.randn(NL, 1, hkv, cap, D, **r), torch.randn(NL, 1, hkv, cap, D, **r)
    o = torch.zeros_like(q)
    steps, nodes = torch.zeros(1, 4, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    chain = [(1 << (i + 1)) - 1 for i in range(T)]  # node i sees nodes 0 to i
    mask = torch.tensor([[[m & (2 ** 63 - 1) | -(m & 2 ** 63) for m in (c & (2 ** 64 - 1), c >> 64)] for c in chain]], device="cuda")

    def set_tree(n, L):
        steps.copy_(torch.tensor([[n, 8, 32, L]], dtype=torch.int32))
        nodes.fill_(n)

    def layers():
        for i in range(NL):
            binding.resps_tree_attention(ctx, steps, nodes, 1, q[i], o[i], None, k[i], v[i], hkv * cap * D, cap * D, D, cap, mask,
                                         1 / math.sqrt(D))

    set_tree(16, 100)
    layers()
    ctx.attention_replan()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        layers()
    for n, L in ((12, 5800), (128, 5800), (40, 5800), (40, 700), (64, 4000), (3, 5900)):
        set_tree(n, L)
        o.zero_()
        graph.replay()
        graph.replay()
        assert ctx.status() == 0
        seen = torch.ones(n, L + n, dtype=torch.bool, device="cuda")
        seen[:, L:] = torch.tril(seen[:, L:])
        for i in range(NL):
            s = torch.einsum("nhgd,hkd->hgnk", q[i, 0, :n].float().view(n, hkv, hq // hkv, D), k[i, 0, :, :L + n].float())
            p = (s / math.sqrt(D)).masked_fill(~seen, float("-inf")).softmax(-1)
            want = torch.einsum("hgnk,hkd->nhgd", p, v[i, 0, :, :L + n].float()).reshape(n, hq, D)
            assert (o[i, 0, :n].float() - want).abs().max() <= 2 ** -8 * want.abs().max()
    del graph
    ctx.close()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("cluster,equal_splits", [(1, 0), (1, 1), (2, None), (5, None), (8, None)])
def test_an_infinity_in_v_stays_in_its_column(cluster, equal_splits, D):
    """One V of a visible key is infinite: its column is infinite (or not a number) in every row of that KV head, and the
    other columns are what they are without it, also where a partial's scale goes by the row's largest magnitude."""
    import numpy as np
    import torch
    import oracle
    _, binding, synth = _imports()
    from harness import bf16_to_f64, check_attention, u16_to_bf16_cuda
    n, Hq, Hkv, L, cap, T, head, key, col = 12, 16, 2, 900, 1024, 16, 1, 333, 5
    ctx = binding.Context(Hq, Hkv, D, 1000, max_batch=1, max_tt=T, max_k=4, max_depth=4)
    ctx.debug_set(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)
    if equal_splits is not None:
        ctx.debug_set(binding.RESPS_DEBUG_ATTN_SINGLE, equal_splits)
    rng = np.random.default_rng(D + cluster)
    q, kc, vc = (synth.to_bf16_bits(rng.normal(size=s).astype(np.float32).ravel()).reshape(s)
                 for s in ((1, T, Hq, D), (1, Hkv, cap, D), (1, Hkv, cap, D)))
    masks = np.zeros((1, T, 2), np.uint64)
    for i in range(n):
        masks[0, i, 0] = (1 << (i + 1)) - 1
    vc[0, head, key, col] = 0
    want = oracle.tree_attention(q[0, :n], kc[0], vc[0], L, masks[0, :n], 0.125)
    vc[0, head, key, col] = 0x7F80
    dq, dk, dv = u16_to_bf16_cuda(q), u16_to_bf16_cuda(kc), u16_to_bf16_cuda(vc)
    do, dm = torch.zeros_like(dq), torch.from_numpy(masks.view(np.int64)).cuda()
    steps, nn = (torch.tensor(x, dtype=torch.int32, device="cuda") for x in ([[n, 1, 1, L]], [n]))
    binding.resps_tree_attention(ctx, steps, nn, 1, dq, do, None, dk, dv, Hkv * cap * D, cap * D, D, cap, dm, 0.125)
    assert ctx.status() == 0
    got = bf16_to_f64(do)[0, :n]
    rows = slice(head * Hq // Hkv, (head + 1) * Hq // Hkv)
    assert not np.isfinite(got[:, rows, col]).any()
    got[:, rows, col] = want[:, rows, col]
    check_attention(got, want)
    ctx.close()
