"""The rerank of the tree build is a selection by a histogram of the scores: the shapes and values at which
it takes another way (the frontiers alone hold fewer than TT-1 candidates; a step of the histogram holds
more candidates than are ranked by counting and is cut again; all of them tie; one candidate, or none)."""
import numpy as np
import pytest

from test_gpu_edges import expand_and_compare

pytestmark = pytest.mark.gpu


def _normal(d, k, V):
    return (np.random.default_rng(d * 100 + k).normal(size=(d, k, V)) * 2).astype(np.float32)


def _equal(d, k, V):
    return np.zeros((d, k, V), np.float32)


def _far_tail(d, k, V):
    """Three likely tokens a row, the rest of its k best 10^6 below: all likely candidates fall into one step."""
    x = _normal(d, k, V)
    x[:, :, 3:] -= 1e6
    return x


def _two_clusters(d, k, V):
    """As above, each cluster equal in itself: the step that is cut again ends in a tie."""
    x = np.zeros((d, k, V), np.float32)
    x[:, :, 3:] = -1e6
    return x


@pytest.mark.parametrize("make", [_normal, _equal, _far_tail, _two_clusters])
@pytest.mark.parametrize("tt,d,k", [(1, 3, 4), (2, 1, 1), (128, 8, 11), (128, 3, 32), (127, 2, 11), (64, 8, 1), (33, 4, 32),
                                    (128, 15, 32)])
def test_rerank_selection(make, tt, d, k):
    expand_and_compare([make(d, k, 64), make(d, k, 64)[:, ::-1].copy()], [(tt, d, k, 5), (max(1, tt - 1), d, k, 6)], [1, 2])
