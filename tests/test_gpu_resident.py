"""Solves of a single mesh in one launch with its rows on chip: the same bits as the multi-CTA kernels
at the edges of the tiling (tile and cluster sizes, ragged passes, the largest mesh, rows with more
entries than fit on chip)."""
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


def _cone(m):
    """A cone: an apex joined to a ring of m vertices (one row of m + 1 entries)."""
    a = 2.0 * np.pi * np.arange(m) / m
    V = np.concatenate([[[0.0, 0.0, 1.0]], np.stack([np.cos(a), np.sin(a), 0.1 * np.sin(3 * a)], 1)])
    i = np.arange(m)
    F = np.stack([np.zeros(m, dtype=np.int64), 1 + i, 1 + (i + 1) % m], 1)
    return V, F.astype(np.int32)


@pytest.mark.parametrize("nx,ny,k", [
    (64, 32, 2),      # 2,048 rows: 16 tiles of 128, the largest cluster of small tiles
    (683, 3, 1),      # 2,049 rows: tiles of 256, the last with one row
    (64, 64, 3),      # 4,096 rows: 16 full tiles, the largest cluster
    (241, 17, 4),     # 4,097 rows: the first mesh whose tiles meet through global memory
    (257, 160, 3),    # 41,120 rows: tiles above 256 rows, a ragged last pass
    (430, 429, 3),    # 184,470 rows: the most rows per SM
    (430, 429, 4),    # the same with the solution outside shared memory
    (0, 300, 3),      # a row of 301 entries: most of its slots outside shared memory
    (0, 3000, 1),     # a row of 3,001 entries
])
def test_resident_solve_same_bits_as_multi_cta(api, nx, ny, k):
    """A single mesh that fits on chip is solved in one launch with one tile per SM (the graph launch
    mode); the host-launched mode runs the multi-CTA kernels on the same tiles. The row arithmetic
    and the order of the sums are the same: the same bits and the same iteration counts, also in a
    second solve on the same buffers, and with a cap on the iterations."""
    from paper_2602_12105_gb300 import _native as N
    from paper_2602_12105_gb300 import meshgen as mg
    rng = np.random.default_rng(11)
    if nx:
        p = mg.config_grid(nx, ny, seed=11, t=None)
        V, F, t = p.V, p.F, 3.0 * p.t
    else:
        V, F = _cone(ny)
        t = 1e-3
    B = rng.uniform(-1.0, 1.0, (V.shape[0], k))
    mesh = api.Mesh(_t(F, torch.int32), V.shape[0])
    mesh.assemble(_t(V), t)
    for kw in ({"rel_tol": 1e-12}, {"rel_tol": 1e-300, "max_iter": 7}):
        Uh, ih = mesh.solve(_t(B), opts=api.make_opts(launch="host", **kw), info=True)
        for _ in range(2):
            U, i = mesh.solve(_t(B), opts=api.make_opts(launch="graph", **kw), info=True)
            assert torch.equal(U, Uh)
            assert i["iterations"] == ih["iterations"] and i["status"] == ih["status"]
            assert i["rel_residual"] == ih["rel_residual"]
    # a non-finite right-hand side is reported
    B[V.shape[0] // 2, 0] = np.inf
    with pytest.raises(N.IgError) as e:
        mesh.solve(_t(B), info=True)
    assert e.value.status == N.IG_ERR_NONFINITE

