"""The FP32 SpMV of meshes whose slices share a column pattern (stretches of grid lines), at the sizes
where it changes its path: lines shorter and longer than a slice, no pattern at all (vertices in random
order), tiles in order and in blocks of lines with ragged last blocks."""
import numpy as np
import pytest

import oracle
from gpu_util import rel2

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


@pytest.mark.parametrize("nx,ny,k,shuffle", [
    (31, 40, 3, False),       # no slice lies within one line
    (64, 33, 1, False),       # every slice of a line touches its end
    (129, 70, 4, False),      # half of the slices follow the pattern
    (300, 61, 2, False),
    (300, 61, 3, True),       # random order: no pattern, columns far apart
    (1027, 1023, 3, False),   # blocks of lines, a ragged last block
    (1531, 701, 2, False),    # a line of about two and a half tiles: tiles in order
    (2100, 501, 3, False),    # blocks of lines beside multiples of their width
    (40, 26300, 1, False),    # a large mesh of short lines: tiles in order
])
def test_mixed_solve_on_grids(api, nx, ny, k, shuffle):
    """Mixed precision to 1e-10 against the FP64 path (within 1e-9, as the other mixed tests; small meshes
    also against the oracle's operator), and the same bits in both launch modes."""
    from paper_2602_12105_gb300 import meshgen as mg
    rng = np.random.default_rng(17)
    p = mg.config_grid(nx, ny, seed=17)
    V, F, t = p.V, p.F, p.t
    if shuffle:
        perm = rng.permutation(V.shape[0])
        inv = np.empty_like(perm)
        inv[perm] = np.arange(perm.size)
        V, F = np.ascontiguousarray(V[perm]), np.ascontiguousarray(inv[F].astype(np.int32))
    B = rng.uniform(-1.0, 1.0, (V.shape[0], k))
    mesh = api.Mesh(_t(F, torch.int32), V.shape[0])
    mesh.assemble(_t(V), t)
    U64 = mesh.solve(_t(B), opts=api.make_opts(rel_tol=1e-12)).cpu().numpy()
    mesh.assemble(_t(V), t, precision="mixed")
    U, info = mesh.solve(_t(B), info=True)
    assert info["status"] == 0 and max(info["true_rel_residual"][:k]) <= 1e-10 * (1 + 1e-3)
    assert rel2(U.cpu().numpy(), U64) <= 1e-9
    Uh = mesh.solve(_t(B), opts=api.make_opts(launch="host"))
    assert torch.equal(U, Uh)
    if V.shape[0] < 30000:
        rowptr, col, A, L, M = oracle.operator(V, F, t)
        R = M[:, None] * B
        res = R - oracle.spmv(rowptr, col, A, U.cpu().numpy())
        assert (np.linalg.norm(res, axis=0) / np.linalg.norm(R, axis=0)).max() <= 1e-10 * (1 + 1e-3)
