"""Sizes at which the prefix scan goes from one tile (8192 values) to several, and
at which the exact matcher's chunks grow from one tile pair to four."""
import numpy as np
import pytest

from test_gpu_parity import _gpu_match, _same_as_exact, ctx, dev, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 8190, 8191, 8192, 8193, 16383, 16384, 300001])
def test_scan_tile_edges(torch_cuda, ctx, orc, n):  # noqa: F811
    """Voxelisation numbers its voxels with two scans over the n points; the
    correspondences of a match of n rows against themselves need a third."""
    from paper_2409_15615_gb300 import kmx

    rng = np.random.default_rng(n)
    pts = rng.uniform(-20.0, 20.0, (n, 3)).astype(np.float32)
    ref, ref_assign = orc.voxelize(pts, 0.5)
    out4, n_out, assign = ctx.voxelize(dev(torch_cuda, pts), 0.5, assign=True)
    ctx.sync()
    assert int(n_out.item()) == len(ref)
    assert np.array_equal(out4[: len(ref)].cpu().numpy().view(np.uint32), ref.view(np.uint32))
    assert np.array_equal(assign.cpu().numpy()[:n], ref_assign)
    if n <= 16384:
        F = rng.gamma(0.5, 20.0, (n, 33)).astype(np.float32)
        i, j, d1, _ = _gpu_match(torch_cuda, ctx, F, F, kmx.MATCH_FP32_EXACT)
        assert np.array_equal(i, np.arange(n)) and np.array_equal(j, i) and not d1.any()


# tile pairs: 1, 64, 304 (one per CTA of a 152-SM device), 607, 608, 1216, 2431, 2432
@pytest.mark.parametrize("tiles", [(1, 1), (8, 8), (16, 19), (607, 1), (19, 32), (32, 38), (11, 221), (38, 64)])
def test_chunk_sizes(torch_cuda, ctx, tiles):  # noqa: F811
    rng = np.random.default_rng(tiles[0])
    n = [128 * t - (3 if t > 1 else 0) for t in tiles]
    P, Q = (rng.gamma(0.5, 20.0, (k, 33)).astype(np.float32) for k in n)
    P[rng.random(P.shape) < 0.5] = 0.0
    k = min(n) // 2
    Q[:k] = P[:k] + np.float32(0.25)
    assert _same_as_exact(torch_cuda, ctx, P, Q) > 0
