"""The target side of the tensor-core matcher looks only at target rows that are
some source row's nearest, within the closest such row's distance."""
import numpy as np
import pytest

from test_gpu_parity import _same_as_exact, ctx, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hits", [1, 127, 128, 129, 700])
def test_few_targets_are_nearest(torch_cuda, ctx, hits):  # noqa: F811
    """2500 source rows around `hits` of 3000 target rows: the others are nobody's
    nearest and the compact row tiles end at, before and after a tile's edge.
    Byte equality with the exact path."""
    rng = np.random.default_rng(hits)
    FQ = rng.gamma(0.5, 20.0, (3000, 33)).astype(np.float32)
    at = rng.permutation(3000)[:hits]
    FP = (FQ[at[rng.integers(0, hits, 2500)]] + rng.normal(0, 0.3, (2500, 33))).astype(np.float32)
    assert _same_as_exact(torch_cuda, ctx, FP, FQ) > 0


@pytest.mark.parametrize("copies", [2, 513, 700])
def test_tied_source_rows(torch_cuda, ctx, copies):  # noqa: F811
    """`copies` equal source rows share one target row as their nearest, at
    distance 0 and at a distance: the lowest source row is mutual, also when the
    target row's candidate list overflows (512)."""
    rng = np.random.default_rng(copies)
    FP = rng.gamma(0.5, 20.0, (1500, 33)).astype(np.float32)
    FQ = rng.gamma(0.5, 20.0, (1300, 33)).astype(np.float32)
    FP[40:40 + copies] = FP[40]
    FP[800:800 + copies] = FP[800]
    FQ[11] = FP[40]
    FQ[12] = FP[800] + np.float32(0.25)
    assert _same_as_exact(torch_cuda, ctx, FP, FQ) > 0


def test_one_column_tile_each_way(torch_cuda, ctx):  # noqa: F811
    """One row against one and against 129: bounds that start at infinity."""
    rng = np.random.default_rng(5)
    F = rng.gamma(0.5, 20.0, (130, 33)).astype(np.float32)
    for p, q in ((1, 1), (1, 129), (129, 1), (2, 128)):
        _same_as_exact(torch_cuda, ctx, F[:p], F[130 - q:])
