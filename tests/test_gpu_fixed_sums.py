"""Scalar products of the FP64 solver added in fixed point: scales at both ends of its range, columns of
very different sizes, columns of zeros, and scales below its range, where the sums are taken in FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_12105_gb300 import api as _api
    return _api


def _t(a, dtype=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device=DEV, dtype=dtype)


@pytest.mark.parametrize("launch", ["graph", "host"])
@pytest.mark.parametrize("nx,ny,k", [
    (19, 7, 1),       # two tiles
    (64, 32, 4),      # a cluster of 16 tiles, eight sums
    (241, 17, 2),     # 17 tiles through global memory: one more than half a warp's addends
    (256, 152, 1),    # 152 tiles: five addends to most lanes
    (256, 152, 3),
    (257, 160, 3),    # 81 tiles of two passes
    (450, 420, 1),    # larger than a resident solve: a tree over the tiles
])
def test_scales(api, nx, ny, k, launch):
    """A right-hand side scaled by a power of two gives the scaled bits as long as the sums stay in range,
    column by column; below it the solve still meets its tolerance; a column of zeros stays zero."""
    from paper_2602_12105_gb300 import meshgen as mg
    rng = np.random.default_rng(5)
    p = mg.config_grid(nx, ny, seed=5, t=None)
    n = p.V.shape[0]
    B = rng.uniform(-1.0, 1.0, (n, k))
    if k > 1:
        B[:, 1] = 0.0
    mesh = api.Mesh(_t(p.F, torch.int32), n)
    mesh.assemble(_t(p.V), 3.0 * p.t)
    opts = api.make_opts(rel_tol=1e-6, launch=launch)
    U, info = mesh.solve(_t(B), opts=opts, info=True)
    assert info["status"] == 0
    # the columns' scales apart from one another (sums of squares from 2^-800 to 2^800)
    s = np.array([2.0 ** e for e in (400, 0, -400, -30)[:k]])
    Us, infos = mesh.solve(_t(B * s), opts=opts, info=True)
    assert torch.equal(Us / _t(s), U) and infos["iterations"] == info["iterations"]
    if k > 1:
        assert float(U[:, 1].abs().max()) == 0.0 and float(Us[:, 1].abs().max()) == 0.0
    # sums of squares around 2^-960 and falling: out of the fixed-point range in the course of the solve
    low = 2.0 ** -486
    Ul, infol = mesh.solve(_t(B * low), opts=opts, info=True)
    assert infol["status"] == 0
    assert max(infol["true_rel_residual"][:k]) <= 1e-6 * (1 + 1e-3)
    mesh.close()
