"""A breakdown of the conjugate gradients inside the FP64 loop (p.q not positive): status, iterations and
iterate of the one-launch solve are those of the multi-CTA loop, with any cap on the iterations."""
import ctypes

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


@pytest.mark.parametrize("k", [1, 2])
@pytest.mark.parametrize("level", [3, 5])  # a cluster; CTAs that meet through global memory
def test_breakdown_in_the_loop(api, level, k):
    from paper_2602_12105_gb300 import _native as N
    from paper_2602_12105_gb300 import meshgen as mg
    V, F = mg.icosphere(level)
    n = V.shape[0]
    mass = 10.0 * n  # of a vertex: sums of squares of M B are in range where those of B . M B are not
    V = V * np.sqrt(mass * n / (4.0 * np.pi))
    B = np.random.default_rng(1).uniform(0.5, 1.0, (n, k))
    # a term of p.q is about mass b^2 = 2^-1078, below half the smallest denormal: 0; one of |M B|^2 is
    # mass^2 b^2 > 2^-1074
    B[:, k - 1] *= 2.0**-539 / np.sqrt(mass)
    mesh = api.Mesh(_t(F, torch.int32), n)
    mesh.assemble(_t(V), 1.0)
    Bd = _t(B)
    for max_iter in (1, 2, 50):
        got = {}
        for launch in ("host", "graph"):
            U = torch.full_like(Bd, 7.0)
            info = N.SolveInfo()
            mesh.ctx.sync_stream()
            st = mesh.ctx.lib.ig_solve(mesh.h, ctypes.c_void_p(Bd.data_ptr()), k, ctypes.c_void_p(U.data_ptr()),
                                       ctypes.byref(api.make_opts(launch=launch, max_iter=max_iter)),
                                       ctypes.byref(info))
            got[launch] = (st, info.iterations, U)
        assert got["host"][0] == N.IG_ERR_NONFINITE
        assert got["graph"][:2] == got["host"][:2]
        assert torch.equal(got["graph"][2], got["host"][2])
    mesh.close()
