"""kcore keeps neighbour lists in shared memory where they fit and walks bit rows
where they do not; a warp holds several vertices on larger selections."""
import numpy as np
import pytest

from test_gpu_prune import _planted, _run_both, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_in,n_tau", [(3000, 3000, 3000), (3000, 2079, 3000), (3000, 2085, 3000),
                                          (4097, 3300, 4097), (6000, 1500, 6000), (6000, 3500, 6000), (33, 33, 33)])
def test_core_numbers_of_dense_graphs(env, n, n_in, n_tau):  # noqa: F811
    """Cliques below, at and above the length of a warp's list (about 2080 neighbours
    at these sizes), one and two vertices a warp: every core number against the
    oracle's peeling."""
    torch, _, ctx = env
    rng = np.random.default_rng(n + n_in)
    src4, tgt4 = _planted(rng, n, n_in, 0.03)
    i = rng.permutation(n).astype(np.int64)
    d2 = rng.uniform(1.0, 50.0, n)
    out = _run_both(torch, ctx, (i, i.copy(), d2 * rng.uniform(0.0, 1.0, n), d2), src4, tgt4, 0.45, n_tau)
    assert out["kmax"] >= n_in // 2


@pytest.mark.parametrize("equal", [1, 40])
def test_ratio_order_within_buckets(env, equal):  # noqa: F811
    """Ratios a few ulps apart, `equal` rows to each, share buckets: rank by
    (ratio, i) within a bucket and after the buckets below."""
    torch, _, ctx = env
    rng = np.random.default_rng(equal)
    n = 2000
    src4, tgt4 = _planted(rng, n, 300, 0.03)
    i = rng.permutation(n).astype(np.int64)
    d2 = np.full(n, 8.0, np.float32)
    step = np.arange(n) // equal % 90
    d1 = np.float32(2.0) + step.astype(np.float32) * np.float32(2.0 ** -20)
    d1[::7] = 7.5
    _run_both(torch, ctx, (i, i.copy(), d1, d2), src4, tgt4, 0.45, 1200)
