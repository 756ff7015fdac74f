"""Which meshes and batches are solved in one launch, by which solves of the public interface, and what a
caller's stream capture gets."""
import os
import subprocess
import sys

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


def _mesh(api, nx, ny):
    """A grid, or (nx = 0) a cone whose apex has ny neighbours."""
    from paper_2602_12105_gb300 import meshgen as mg
    if nx:
        p = mg.config_grid(nx, ny, seed=3)
        V, F, t = p.V, p.F, p.t
    else:
        a = 2.0 * np.pi * np.arange(ny) / ny
        V = np.concatenate([[[0.0, 0.0, 1.0]], np.stack([np.cos(a), np.sin(a), 0.1 * np.sin(3 * a)], 1)])
        i = np.arange(ny)
        F, t = np.stack([np.zeros(ny, dtype=np.int64), 1 + i, 1 + (i + 1) % ny], 1), 1e-3
    return api.Mesh(_t(F, torch.int32), V.shape[0]), _t(V), t


def _solve(api, nx, ny, k, precision, launch="graph"):
    mesh, V, t = _mesh(api, nx, ny)
    B = _t(np.random.default_rng(1).uniform(-1.0, 1.0, (mesh.n, k)))
    mesh.assemble(V, t, precision)
    assert mesh.route() == ("none", 0)
    mesh.solve(B, opts=api.make_opts(launch=launch))
    r = mesh.route()
    mesh.close()
    return r


# the meshes of test_gpu_resident.py, whose bits are compared between the launch modes, and the first
# mesh above the limit (152 SMs x 1,216 rows)
@pytest.mark.parametrize("nx,ny,k,ctas", [
    (64, 32, 2, 16), (683, 3, 1, 9), (64, 64, 3, 16), (241, 17, 4, 17), (257, 160, 3, 81), (430, 429, 3, None),
    (430, 429, 4, None), (0, 300, 3, 3), (0, 3000, 1, 12), (430, 430, 1, 0), (430, 430, 4, 0),
])
def test_route_fp64(api, nx, ny, k, ctas):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip("the sizes are those of 152 SMs")
    route, got = _solve(api, nx, ny, k, "fp64")
    if ctas == 0:
        assert (route, got) == ("graph", 0)
    else:
        assert route == "one_launch" and (got == ctas if ctas else 0 < got <= sms)
    assert _solve(api, nx, ny, k, "fp64", "host") == ("host", 0)


# those of test_gpu_gang.py; the largest gangs have 152 x 4 tiles of 576 rows (350,208), so two of its sizes
# are above them, and test_largest_gangs below compares the bits at the limit
@pytest.mark.parametrize("nx,ny,k,precision,one", [
    (16, 16, 3, "mixed", True), (257, 2, 1, "mixed32", True), (64, 16, 4, "mixed", True), (205, 5, 2, "mixed32", True),
    (500, 499, 3, "mixed", True), (595, 596, 3, "mixed32", False), (595, 596, 4, "mixed", False),
    (591, 592, 3, "mixed32", True), (591, 592, 4, "mixed", True), (591, 593, 4, "mixed", False),
    (600, 600, 3, "mixed", False), (0, 2500, 3, "mixed", True),
])
def test_route_mixed(api, nx, ny, k, precision, one):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip("the sizes are those of 152 SMs")
    route, got = _solve(api, nx, ny, k, precision)
    assert (route == "one_launch" and 0 < got <= sms) if one else (route, got) == ("graph", 0)
    assert _solve(api, nx, ny, k, precision, "host") == ("host", 0)


@pytest.mark.parametrize("k,precision", [(1, "mixed"), (3, "mixed32"), (4, "mixed")])
def test_largest_gangs(api, k, precision):
    """The most rows per SM, with some slots of a row outside shared memory for k = 4: the bits of the
    multi-CTA kernels."""
    mesh, V, t = _mesh(api, 591, 592)
    B = _t(np.random.default_rng(5).uniform(-1.0, 1.0, (mesh.n, k)))
    mesh.assemble(V, 3.0 * t, precision)
    for kw in ({}, {"max_iter": 5}):
        Uh, ih = mesh.solve(B, opts=api.make_opts(launch="host", **kw), info=True)
        U, i = mesh.solve(B, info=True, opts=api.make_opts(**kw))
        assert torch.equal(U, Uh) and i == ih
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert mesh.route()[0] == "one_launch"


def test_route_batches(api):
    ms = [_mesh(api, 40, 30 + i) for i in range(3)]
    batch = api.Batch([m for m, _, _ in ms])
    Bs = [V.clone() for _, V, _ in ms]
    for precision, route in (("mixed", "one_launch"), ("mixed32", "one_launch"), ("fp64", "graph")):
        batch.assemble([V for _, V, _ in ms], [t for _, _, t in ms], precision)
        batch.solve(Bs)
        assert batch.route() == route
        batch.solve(Bs, opts=api.make_opts(launch="host"))
        assert batch.route() == "host"
    assert api.Batch([ms[0][0]]).route() == "none"


@pytest.mark.parametrize("sizes,route", [
    ([(405, 405)] * 4, "one_launch"),             # a few large meshes: gangs one after another
    ([(405, 405)] * 10, "graph"),                 # many: the multi-CTA loop
    ([(405, 405)] + [(220, 186)] * 8, "one_launch"),
    ([(405, 405)] + [(220, 186)] * 40, "graph"),  # CTAs of four workers for all: 41 of them a mesh
    ([(220, 186)] * 60, "one_launch"),            # CTAs of two workers
    ([(590, 590)] * 12, "one_launch"),
])
def test_route_of_large_mixed_batches(api, sizes, route):
    """Batches that the multi-CTA loop solves sooner go there, with the same bits as each mesh alone."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are those of 152 SMs")
    ms = [_mesh(api, nx, ny) for nx, ny in sizes]
    batch = api.Batch([m for m, _, _ in ms])
    Bs = [V.clone() for _, V, _ in ms]
    batch.assemble([V for _, V, _ in ms], [t for _, _, t in ms], "mixed")
    opts = api.make_opts(max_iter=12)
    Us = batch.solve(Bs, opts=opts)
    assert batch.route() == route
    for i in (0, len(ms) - 1):
        U = ms[i][0].solve(Bs[i], opts=opts)
        assert ms[i][0].route()[0] == "one_launch" and torch.equal(U, Us[i])


def _captured(nx, ny, precision, works):
    from paper_2602_12105_gb300 import _native as N
    from paper_2602_12105_gb300 import api
    mesh, V, t = _mesh(api, nx, ny)
    B = V.clone()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        mesh.assemble(V, t, precision)
        U0 = mesh.solve(B)
        U = torch.empty_like(B)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    try:
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            mesh.solve(B, out=U)
        captured = True
    except Exception:  # noqa: BLE001 - an IgError from the call, or torch's at the end of the capture
        captured = False
    assert captured == works
    if works:
        for _ in range(2):
            U.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(U, U0)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        if not works:
            try:
                mesh.solve(B)
            except N.IgError as e:
                assert e.status == N.IG_ERR_CUDA
        assert torch.equal(mesh.solve(B), U0)
    torch.cuda.synchronize()


@pytest.mark.parametrize("nx,ny,precision,works", [
    (40, 30, "fp64", True),    # one cluster: a plain kernel
    (100, 90, "fp64", False),  # the graph of the loop holds a conditional node, which no capture takes
    (40, 30, "mixed", False),
])
def test_solve_under_a_capture(api, nx, ny, precision, works):
    """A captured solve replays with the solve's bits, or the capture is refused; the mesh solves as before
    after either (the refused launch's error may be reported once more first). In a process of its own:
    after a refused capture torch's generator stays in its capture state."""
    code = f"import test_gpu_routes as t; t._captured({nx}, {ny}, {precision!r}, {works})"
    here = os.path.dirname(os.path.abspath(__file__))
    res = subprocess.run([sys.executable, "-c", code], cwd=here, capture_output=True, text=True, timeout=300,
                         env={**os.environ, "PYTHONPATH": os.pathsep.join([here, os.path.dirname(here)])})
    assert res.returncode == 0, res.stderr[-2000:]
