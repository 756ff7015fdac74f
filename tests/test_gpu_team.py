"""One-launch solves of which not every CTA begins in time (other work holds SMs): the CTAs that have begun
solve the mesh, with the same bits. Solves on several streams and threads, beside other kernels."""
import threading

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


def _mesh(api, ctx, nx, ny):
    """A grid, or (nx = 0) a cone whose apex has ny neighbours."""
    from paper_2602_12105_gb300 import meshgen as mg
    if nx:
        p = mg.config_grid(nx, ny, seed=3)
        V, F, t = p.V, p.F, 3.0 * p.t
    else:
        a = 2.0 * np.pi * np.arange(ny) / ny
        V = np.concatenate([[[0.0, 0.0, 1.0]], np.stack([np.cos(a), np.sin(a), 0.1 * np.sin(3 * a)], 1)])
        i = np.arange(ny)
        F, t = np.stack([np.zeros(ny, dtype=np.int64), 1 + i, 1 + (i + 1) % ny], 1), 1e-3
    return api.Mesh(_t(F, torch.int32), V.shape[0], ctx=ctx), _t(V), t


def _hold(streams):
    """Kernels of one block each that hold an SM's shared memory or a part of it for some 5 ms."""
    torch.cuda.synchronize()
    for s in streams:
        with torch.cuda.stream(s):
            torch.cuda._sleep(10_000_000)


def _compare(api, nx, ny, k, precision):
    """With little waiting for the others to begin, and with SMs held by other kernels: the team is whoever
    has begun by then. Returns the sizes of the teams with rows off chip and the whole team's."""
    ctx = api.Context(0)
    mesh, V, t = _mesh(api, ctx, nx, ny)
    B = _t(np.random.default_rng(5).uniform(-1.0, 1.0, (mesh.n, k)))
    mesh.assemble(V, t, precision)
    sizes, others, main = set(), [torch.cuda.Stream() for _ in range(30)], torch.cuda.Stream()
    for kw in ({"rel_tol": 1e-12}, {"rel_tol": 1e-300, "max_iter": 7, "max_refine": 2}):
        Uh, ih = mesh.solve(B, opts=api.make_opts(launch="host", **kw), info=True)
        for begin, held in ((-1, 0), (0, 0), (0, 0), (1, 0), (0, 1), (1, 9), (0, 30), (1, 30), (-1, 30), (-1, 0)):
            ctx.set_wait_limits(begin=begin)
            _hold(others[:held])
            with torch.cuda.stream(main):
                U, i = mesh.solve(B, opts=api.make_opts(**kw), info=True)
                route, ctas = mesh.route()
            torch.cuda.synchronize()
            assert torch.equal(U, Uh) and i == ih
            if (begin, held) == (-1, 0):
                assert route == "one_launch"
                full = ctas
            assert route in ("one_launch", "off_chip") and 0 < ctas <= full
            if route == "off_chip":
                sizes.add(ctas)
    mesh.close()
    return sizes, full


@pytest.mark.parametrize("nx,ny,k", [
    (241, 17, 4),     # 17 tiles of 256 rows
    (257, 160, 3),    # 81 tiles of two passes
    (430, 429, 1), (430, 429, 2), (430, 429, 3),
    (430, 429, 4),    # the solution outside shared memory in the whole team
    (0, 5000, 3),     # a row of 5,001 entries, 20 tiles
])
def test_fewer_ctas_than_tiles_fp64(api, nx, ny, k):
    sizes, full = _compare(api, nx, ny, k, "fp64")
    print(f"{nx}x{ny} k {k}: teams of {sorted(sizes)} of {full} CTAs")
    if ny == 429 and full == torch.cuda.get_device_properties(0).multi_processor_count:
        assert sizes and max(sizes) < full  # a CTA takes an SM's whole shared memory: held SMs are missing


@pytest.mark.parametrize("nx,ny,k,precision", [
    (64, 17, 4, "mixed"),      # two groups of four tiles
    (205, 5, 2, "mixed32"),    # 1,025 rows: a second group of one row
    (300, 211, 3, "mixed"),
    (591, 592, 1, "mixed"), (591, 592, 2, "mixed"), (591, 592, 3, "mixed32"), (591, 592, 4, "mixed"),
    (0, 5000, 3, "mixed"),     # a row of 5,001 entries
])
def test_fewer_ctas_than_groups_mixed(api, nx, ny, k, precision):
    sizes, full = _compare(api, nx, ny, k, precision)
    print(f"{nx}x{ny} k {k}: teams of {sorted(sizes)} of {full} CTAs")
    if ny == 592 and full == torch.cuda.get_device_properties(0).multi_processor_count:
        assert sizes


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("large", [False, True])
def test_batches_of_which_not_every_cta_starts(api, k, large):
    """Batches in CTAs of four workers (a mesh of more than 155,000 rows) and of two, with SMs held: every
    mesh has the bits it has alone."""
    ctx = api.Context(0)
    sizes = [(61 + 3 * i, 40 + i) for i in range(24)] + [(200, 150)] * 6 + ([(450, 430)] * 2 if large else [])
    ms = [_mesh(api, ctx, nx, ny) for nx, ny in sizes]
    batch = api.Batch([m for m, _, _ in ms])
    Vs, ts = [V for _, V, _ in ms], [t for _, _, t in ms]
    Bs = [V[:, :k].contiguous() for V in Vs]
    batch.assemble(Vs, ts, "mixed")
    U0, i0 = batch.solve(Bs, opts=api.make_opts(launch="host"), info=True)
    others, main = [torch.cuda.Stream() for _ in range(30)], torch.cuda.Stream()
    routes = set()
    for begin, held in ((-1, 0), (0, 0), (0, 9), (1, 30), (-1, 30), (-1, 0)):
        ctx.set_wait_limits(begin=begin)
        _hold(others[:held])
        with torch.cuda.stream(main):
            U, i = batch.solve(Bs, info=True)
            routes |= {m.route() for m, _, _ in ms}
        torch.cuda.synchronize()
        assert batch.route() == "one_launch"
        assert all(torch.equal(a, b) for a, b in zip(U, U0)) and i == i0
    print(f"large {large} k {k}: {sorted(routes)}")
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert any(ctas > 0 for _, ctas in routes)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_streams_and_threads(api, precision):
    """Two threads solve and differentiate, each with its own context and stream, while a third stream
    keeps the GPU busy with matrix products: every result has the bits it has alone."""
    jobs = [_mesh(api, api.Context(0), nx, ny) for nx, ny in ((430, 429), (300, 211))]
    want = []
    for mesh, V, t in jobs:
        mesh.assemble(V, t, precision)
        U = mesh.solve(V)
        want.append((U, mesh.adjoint(V, None, True, U, V)[0]))
    torch.cuda.synchronize()
    failed = []

    def work(job, ref):
        try:
            mesh, V, t = job
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(12):
                    mesh.assemble(V, t, precision)
                    U = mesh.solve(V)
                    g = mesh.adjoint(V, None, True, U, V)[0]
                    s.synchronize()
                    if not (torch.equal(U, ref[0]) and torch.equal(g, ref[1])):
                        failed.append("bits")
                mesh.check()
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=(j, r)) for j, r in zip(jobs, want)]
    other = torch.cuda.Stream()
    A = torch.randn(4096, 4096, device=DEV, dtype=torch.bfloat16)
    for th in threads:
        th.start()
    with torch.cuda.stream(other):
        while any(th.is_alive() for th in threads):
            for _ in range(8):
                A @ A
            other.synchronize()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not failed, failed


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_threads_keep_their_route(api, precision):
    """Two threads whose meshes take different amounts of shared memory: no launch is refused for the other
    thread's limit."""
    import ctypes
    jobs = [_mesh(api, api.Context(0), nx, ny) for nx, ny in ((430, 429), (241, 17))]
    for mesh, V, t in jobs:
        mesh.assemble(V, t, precision)
        mesh.solve(V)
    torch.cuda.synchronize()
    routes, go = {0: {}, 1: {}}, threading.Barrier(2)

    def work(i):  # calls of the library alone, so that two of them overlap
        mesh, V, _ = jobs[i]
        opts, U, lib = api.make_opts(max_iter=2, max_refine=1), torch.empty_like(V), mesh.ctx.lib
        B, out, po = ctypes.c_void_p(V.data_ptr()), ctypes.c_void_p(U.data_ptr()), ctypes.byref(opts)
        r, k, n = ctypes.c_int(), mesh.h, {}
        with torch.cuda.stream(torch.cuda.Stream()):
            mesh.ctx.sync_stream()
            go.wait()
            for j in range(6000):
                lib.ig_solve(k, B, 3, out, po, None)
                lib.ig_mesh_route(k, ctypes.byref(r), None)
                n[r.value] = n.get(r.value, 0) + 1
                if j % 200 == 199:
                    torch.cuda.current_stream().synchronize()
        routes[i] = n

    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 1)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert all(set(r) == {3} for r in routes.values()), routes  # IG_ROUTE_ONE_LAUNCH
