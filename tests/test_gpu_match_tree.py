"""Tree order of the tensor-core matcher: nodes at the size from which a level
takes separate kernels (2048 rows), splits over a cluster's CTAs, and capacities
far above the device counts (levels that hold leaves only)."""
import numpy as np
import pytest

from test_gpu_parity import _pad36, _same_as_exact, ctx, dev, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _rows(rng, n):
    cen = rng.gamma(0.5, 20.0, (40, 33))
    return (cen[rng.integers(0, 40, n)] + rng.normal(0, 2.0, (n, 33))).astype(np.float32)


@pytest.mark.parametrize("shape", [(2047, 2048), (2049, 100), (129, 4097), (16385, 8191), (33000, 2177)])
def test_sizes_around_the_switch(torch_cuda, ctx, shape):  # noqa: F811
    rng = np.random.default_rng(shape[0])
    P, Q = _rows(rng, shape[0]), _rows(rng, shape[1])
    Q[: min(shape) // 2] = P[: min(shape) // 2] + np.float32(0.125)
    assert _same_as_exact(torch_cuda, ctx, P, Q) > 0


def test_equal_projections(torch_cuda, ctx):  # noqa: F811
    """Half of a 20000-row cloud is one descriptor: the split row's key is shared by
    rows on both sides of the split, over all CTAs of a cluster."""
    rng = np.random.default_rng(3)
    P, Q = _rows(rng, 20000), _rows(rng, 9000)
    P[5000:15000] = P[17]
    assert _same_as_exact(torch_cuda, ctx, P, Q) > 0


@pytest.mark.parametrize("count", [(1, 1), (100, 130), (2100, 1500), (5000, 7000)])
def test_counts_below_capacity(torch_cuda, ctx, count):  # noqa: F811
    from paper_2409_15615_gb300 import kmx

    rng = np.random.default_rng(count[0])
    caps = (50000, 40003)
    n = torch_cuda.tensor(count, dtype=torch_cuda.int64, device="cuda")
    full = [_rows(rng, c) for c in caps]
    res = []
    for mode in (kmx.MATCH_FP32_EXACT, kmx.MATCH_BF16_RERANK):
        d = [dev(torch_cuda, _pad36(f)) for f in full]
        corr, n_out = ctx.match(d[0], None, caps[0], d[1], None, caps[1], mode=mode, d_np=n[0:1], d_nq=n[1:2])
        ctx.sync()
        res.append(corr[: int(n_out.item())].cpu().numpy())
    assert len(res[0]) > 0 and np.array_equal(res[0], res[1])
