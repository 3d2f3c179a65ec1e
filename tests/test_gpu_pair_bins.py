"""SPFH bins decided from approximations, with the exact expressions near a
decision: histograms against the FP64 oracle over inputs that reach every
branch (features spread over all bins, near-parallel normals, coplanar points
whose source choice ties, coincident points, normals that are not unit vectors
or zero).  A pair within 1e-5 of a decision in FP64 may move by one bin; FP32
evaluation differs from FP64 by at most a few 1e-6 in each feature here.  And
tiny clouds, where warps hold fewer rows than lanes: the list path and the
list-free path give the same bits."""
import numpy as np
import pytest

from parity_helpers import spfh_allowance

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_15615_gb300 import build, kmx

    build.build()
    ctx = kmx.Context(0)
    yield torch, kmx, ctx
    ctx.close()


def _inputs(case, n=2500):
    rng = np.random.default_rng(len(case))
    p = np.zeros((n, 4), np.float32)
    p[:, :3] = rng.uniform(0, 3, (n, 3))
    nv = rng.standard_normal((n, 3))
    if case in ("near-parallel", "coplanar"):
        nv = np.array([0.0, 0.0, 1.0]) + (1e-3 * nv if case == "near-parallel" else 0.0)
        p[:, 2] = 0.0 if case == "coplanar" else p[:, 2] * 0.05
    if case == "coincident":
        p[n // 2:] = p[: n - n // 2]
    nv = np.broadcast_to(nv, (n, 3)) / np.linalg.norm(nv, axis=-1, keepdims=True)
    if case == "scaled":
        nv = nv * np.array([0.5, 1.0, 1.5])[np.arange(n) % 3][:, None]
    if case == "zero":
        nv = nv * (np.arange(n) % 4 > 0)[:, None]
    n4 = np.zeros((n, 4), np.float32)
    n4[:, :3] = nv
    return p, n4


@pytest.mark.parametrize("case", ["spread", "near-parallel", "coplanar", "coincident", "scaled", "zero"])
def test_spfh_bins(env, orc, case):
    torch, kmx, ctx = env
    p, n4 = _inputs(case)
    n = len(p)
    prm = kmx.params_default(0.1)
    offs, nbr = orc.radius_search(p, prm.r_fpfh)
    fl = np.full(n, 5, np.uint8)
    voffs, vnbr, J, fl2 = orc.valid_filter(offs, nbr, fl, 3)
    sp, npairs, _, n_marg = orc.spfh(p, n4.astype(np.float64), fl2, voffs, vnbr, 11, with_margin=True, band=1e-5)
    d = torch.from_numpy(p).cuda()
    grid = ctx.build_grid(d, prm.r_fpfh)
    res = ctx.fasterpfh(grid, prm, torch.from_numpy(n4).cuda(), torch.from_numpy(fl).cuda(),
                        torch.from_numpy(offs).cuda(), torch.from_numpy(nbr.astype(np.int32)).cuda(), want_spfh=True)
    ctx.sync()
    got = res["spfh"][:n, :33].cpu().numpy().astype(np.float64)
    allow = spfh_allowance(n_marg, npairs)
    assert (np.abs(got - sp).max(1) <= allow + 1e-4).all()
    if case == "spread":
        assert (allow == 0).mean() > 0.8 and (sp > 0).any(0).all()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 9, 10, 27, 28, 100])
def test_small_clouds_equal_the_list_free_path(env, n):
    torch, kmx, ctx = env
    rng = np.random.default_rng(n)
    p = np.zeros((n, 4), np.float32)
    p[:, :3] = rng.uniform(0, 0.5, (n, 3)) * [1, 1, 0.3]
    d = torch.from_numpy(p).cuda()
    prm = kmx.params_default(0.1)
    grid = ctx.build_grid(d, prm.r_fpfh)
    a = ctx.normals(grid, prm, 256 * n)
    b = ctx.fasterpfh(grid, prm, a["normal4"], a["flags"], a["offs"], a["nbr"])
    c = ctx.features(grid, prm)
    ctx.sync()
    nj = int(b["n_valid"].item())
    assert nj == int(c["n_valid"].item())
    assert torch.equal(a["normal4"], c["normal4"]) and torch.equal(a["flags"], c["flags"])
    assert torch.equal(b["valid"][:nj], c["valid"][:nj]) and torch.equal(b["desc"][:nj], c["desc"][:nj])
