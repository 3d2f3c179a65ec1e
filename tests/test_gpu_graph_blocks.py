"""graph_build tests every pair of 32-vertex blocks once and writes both words:
selections that end inside, at and after a block, and fewer vertices than the
capacity (the words past the selection are not written)."""
import numpy as np
import pytest

from test_gpu_prune import _planted, _run_both, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_tau", [(31, 3000), (32, 3000), (33, 3000), (64, 64), (95, 97), (1000, 1000), (1025, 4096)])
def test_block_edges(env, n, n_tau):  # noqa: F811
    torch, _, ctx = env
    rng = np.random.default_rng(n)
    # other work on the context's scratch first, so that it does not start as zeros
    big4, tgt4 = _planted(rng, 4000, 3500, 0.03)
    i = rng.permutation(4000).astype(np.int64)
    d = rng.uniform(1.0, 50.0, 4000)
    _run_both(torch, ctx, (i, i.copy(), d * rng.uniform(0.0, 1.0, 4000), d), big4, tgt4, 0.45, 4000)
    src4, tgt4 = _planted(rng, n, n // 2, 0.05)
    i = rng.permutation(n).astype(np.int64)
    d = rng.uniform(1.0, 50.0, n)
    _run_both(torch, ctx, (i, i.copy(), d * rng.uniform(0.0, 1.0, n), d), src4, tgt4, 0.45, n_tau)
