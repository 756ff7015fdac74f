"""Waits of the one-launch solves that run out: the solve returns, its result is NaN and its callers can see
that it failed; the next solve of the same mesh is right."""
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


def _ico(api, ctx, level, seed=0):
    from paper_2602_12105_gb300 import meshgen as mg
    V, F = mg.icosphere(level)
    V = mg.radial_perturb(V, 0.02, np.random.default_rng(seed))
    return api.Mesh(_t(F, torch.int32), V.shape[0], ctx=ctx), _t(V)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_wait_that_runs_out_is_seen(api, precision):
    """No polls: in 41 CTAs (FP64) or 11 (mixed) and dozens of meetings some CTA finds a post missing."""
    from paper_2602_12105_gb300 import _native as N
    ctx = api.Context(0)
    mesh, V = _ico(api, ctx, 5)
    mesh.assemble(V, 1e-3, precision)
    U0, info0 = mesh.solve(V, info=True)
    assert mesh.route()[0] == "one_launch" and info0["status"] == 0
    mesh.check()
    ctx.set_wait_limits(meet=0)
    U = mesh.solve(V)  # without info the call itself is asynchronous
    assert torch.isnan(U).any()
    with pytest.raises(N.IgError) as e:
        mesh.check()
    assert e.value.status == N.IG_ERR_CUDA and "given up" in str(e.value)
    with pytest.raises(N.IgError) as e:
        mesh.solve(V, info=True)
    assert e.value.status == N.IG_ERR_CUDA and "given up" in str(e.value)
    gV, _, _ = mesh.adjoint(V, None, True, U0, V)
    assert torch.isnan(gV).any()
    ctx.set_wait_limits()
    assert torch.equal(mesh.solve(V), U0)
    mesh.assemble(V, 1e-3, precision)
    for _ in range(3):
        U, info = mesh.solve(V, info=True)
        assert torch.equal(U, U0) and info == info0


def test_batch_waits_that_run_out(api):
    """A batch whose larger meshes give up: each mesh either gives up or has the bits it has alone."""
    from paper_2602_12105_gb300 import _native as N
    ctx = api.Context(0)
    items = [_ico(api, ctx, level, i) for i, level in enumerate([5, 4, 3, 5, 2, 4] * 4)]
    batch = api.Batch([m for m, _ in items])
    Vs, ts = [V for _, V in items], [1e-3] * len(items)
    batch.assemble(Vs, ts, "mixed")
    U0 = batch.solve(Vs)
    assert batch.route() == "one_launch"
    ctx.set_wait_limits(meet=0)
    Us = batch.solve(Vs)
    given_up = [bool(torch.isnan(U).any()) for U in Us]
    assert any(given_up)
    for U, V0, g, (m, _) in zip(Us, U0, given_up, items):
        if g:
            with pytest.raises(N.IgError):
                m.check()
        else:
            assert torch.equal(U, V0)
    with pytest.raises(N.IgError) as e:
        batch.solve(Vs, info=True)
    assert e.value.status == N.IG_ERR_CUDA
    ctx.set_wait_limits()
    batch.assemble(Vs, ts, "mixed")
    Us, infos = batch.solve(Vs, info=True)
    assert all(torch.equal(a, b) for a, b in zip(Us, U0)) and all(i["status"] == 0 for i in infos)


def test_limits_are_checked(api):
    from paper_2602_12105_gb300 import _native as N
    ctx = api.Context(0)
    with pytest.raises(N.IgError) as e:
        ctx.set_wait_limits(meet=-2)
    assert e.value.status == N.IG_ERR_INVALID_ARG
