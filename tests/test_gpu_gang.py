"""Mixed-precision solves of a group of meshes in one launch (gangs of CTAs that hold their meshes on
chip): the same bits as the multi-CTA kernels at the edges of the tiling, alone and in batches of more
meshes than SMs."""
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


def _mesh(nx, ny, seed=3):
    """A grid, or (nx = 0) a cone whose apex has ny neighbours: V, F, t."""
    from paper_2602_12105_gb300 import meshgen as mg
    if nx:
        p = mg.config_grid(nx, ny, seed=seed)
        return p.V, p.F, 3.0 * p.t
    a = 2.0 * np.pi * np.arange(ny) / ny
    V = np.concatenate([[[0.0, 0.0, 1.0]], np.stack([np.cos(a), np.sin(a), 0.1 * np.sin(3 * a)], 1)])
    i = np.arange(ny)
    return V, np.stack([np.zeros(ny, dtype=np.int64), 1 + i, 1 + (i + 1) % ny], 1).astype(np.int32), 1e-3


@pytest.mark.parametrize("nx,ny,k,precision", [
    (16, 16, 3, "mixed"),       # one full tile
    (257, 1 + 1, 1, "mixed32"),  # 514 rows: three tiles, the last with two rows
    (64, 16, 4, "mixed"),       # 1,024 rows: one full group of four tiles
    (205, 5, 2, "mixed32"),     # 1,025 rows: a second group of one row
    (500, 499, 3, "mixed"),     # tiles of more than 256 rows: a ragged second pass
    (595, 596, 3, "mixed32"),   # the most rows per SM
    (595, 596, 4, "mixed"),     # the same with some slots of a row outside shared memory
    (600, 600, 3, "mixed"),     # too large for a gang: the multi-CTA kernels in both modes
    (0, 2500, 3, "mixed"),      # a row of 2,501 entries
])
def test_single_mesh_same_bits_as_multi_cta(api, nx, ny, k, precision):
    V, F, t = _mesh(nx, ny)
    B = np.random.default_rng(5).uniform(-1.0, 1.0, (V.shape[0], k))
    mesh = api.Mesh(_t(F, torch.int32), V.shape[0])
    mesh.assemble(_t(V), t, precision=precision)
    for kw in ({}, {"max_iter": 5}, {"rel_tol": 1e-14, "max_refine": 2}):
        Uh, ih = mesh.solve(_t(B), opts=api.make_opts(launch="host", **kw), info=True)
        for _ in range(2):
            U, i = mesh.solve(_t(B), opts=api.make_opts(launch="graph", **kw), info=True)
            assert torch.equal(U, Uh)
            assert i == ih


@pytest.mark.parametrize("precision", ["mixed", "mixed32"])
def test_batch_of_more_meshes_than_sms(api, precision):
    """200 meshes of 1 to 21 groups of tiles, some of which are done at once (a zero right-hand side):
    each the same bits as alone, twice."""
    rng = np.random.default_rng(9)
    sizes = [(int(rng.integers(4, 60)), int(rng.integers(4, 60))) for _ in range(188)] + [(150, 141)] * 8 + [(0, 400)] * 4
    items = [_mesh(nx, ny, seed=i) for i, (nx, ny) in enumerate(sizes)]
    Bs = [_t(rng.uniform(-1.0, 1.0, (V.shape[0], 3))) for V, _, _ in items]
    for i in range(0, 200, 17):
        Bs[i].zero_()
    meshes = [api.Mesh(_t(F, torch.int32), V.shape[0]) for V, F, _ in items]
    Vs, ts = [_t(V) for V, _, _ in items], [t for _, _, t in items]
    batch = api.Batch(meshes)
    batch.assemble(Vs, ts, precision)
    Us, infos = batch.solve(Bs, info=True)
    again = batch.solve(Bs)
    for i, (m, V, t, B) in enumerate(zip(meshes, Vs, ts, Bs)):
        U, info = m.solve(B, info=True)
        assert torch.equal(U, Us[i]) and torch.equal(U, again[i]), i
        assert info == infos[i], i
