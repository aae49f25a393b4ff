"""The ways a layer's attention is laid out (clusters of every size, equal splits, ranges over all groups), forced
by the test-only overrides on shapes where each can go wrong: more CTAs than key tiles, groups whose size does not
divide a row tile, a single token, fewer groups than clusters and more."""
import pytest

from test_gpu_edges import _attention_case, _imports

pytestmark = pytest.mark.gpu

SHAPES = [dict(n=7, Hq=12, Hkv=4, D=64, L=5), dict(n=33, Hq=14, Hkv=2, D=128, L=447),
          dict(n=[1, 90, 3], Hq=8, Hkv=8, D=128, L=[0, 1400, 63], B=3),
          dict(n=[20, 128], Hq=16, Hkv=4, D=128, L=[5, 1400], B=2)]  # a cluster: a short item, then a long one


@pytest.mark.parametrize("cluster,equal_splits", [(1, 0), (1, 1000), (2, None), (3, None), (4, None), (6, None), (8, None)])
@pytest.mark.parametrize("shape", range(len(SHAPES)))
def test_layouts(shape, cluster, equal_splits):
    _, binding, _ = _imports()
    debug = [(binding.RESPS_DEBUG_ATTN_CLUSTER, cluster)]
    if equal_splits is not None:
        debug.append((binding.RESPS_DEBUG_ATTN_SINGLE, equal_splits))
    _attention_case(**SHAPES[shape], cap=1664, seed=cluster, poison=True, debug=debug)
