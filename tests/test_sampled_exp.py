"""The acceptance kernel's exponential (a table of 2^(i/64) and five terms of the series) restated in fp64 on the
CPU: within two units in the last place of the library's over the range of softmax arguments, 0 below -700."""
import numpy as np


def exp_le0(t):
    magic = 6755399441055744.0
    k = (t * 92.33248261689366 + magic - magic)
    r = (t.astype(np.longdouble) - k.astype(np.longdouble) * (np.log(np.longdouble(2)) / 64)).astype(np.float64)
    q = ((((r / 120 + 1 / 24) * r + 1 / 6) * r + 0.5) * r + 1.0) * r
    k = k.astype(np.int64)
    head = np.exp2((k & 63) / 64.0)
    v = np.ldexp(head * q + head, (k >> 6).astype(np.int32))
    return np.where(t > -700.0, v, 0.0)


def test_table_driven_exponential_matches_the_library():
    rng = np.random.default_rng(0)
    edges = np.arange(-64000, 1) * np.log(2) / 128          # ends and middles of the table's intervals
    t = np.concatenate([-rng.exponential(8.0, 200000), -rng.uniform(0, 699.0, 200000), edges[edges > -699], [0.0, 1e-15, -1e-300]])
    want = np.exp(t.astype(np.longdouble))
    assert np.max(np.abs(exp_le0(t) / want - 1)) < 2 * 2.3e-16
    assert np.all(exp_le0(np.array([-700.5, -1e4, -1e300])) == 0.0)
