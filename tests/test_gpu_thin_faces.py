"""dl/dV and dl/dt of the per-face gradient on meshes of thin faces, with each face's vertices listed from
each of its three corners: against the per-corner formula in extended precision on the same Lambda and U.

The bound is that of the per-corner formula in FP64: its products cancel by the ratio of a face's long to
its short side, so 32 x 2^-53 x ratio of the largest entry. (A form that leaves the short edge out cancels
by the ratio's square.)"""
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


def _grid(ratio, nx=9, ny=11):
    """Cells of 1 x ratio on a smooth height field, turned out of the axes."""
    x, y = np.meshgrid(np.arange(nx, dtype=float), np.arange(ny) * ratio)
    P = np.stack([x, y, 0.2 * np.sin(x) + 0.3 * np.cos(2.0 * y / ratio) * ratio], -1).reshape(-1, 3)
    Q, _ = np.linalg.qr(np.random.default_rng(2).standard_normal((3, 3)))
    v = (np.arange(ny - 1)[:, None] * nx + np.arange(nx - 1)).reshape(-1)
    F = np.stack([v, v + 1, v + nx + 1, v, v + nx + 1, v + nx], 1).reshape(-1, 3)
    return P @ Q.T, F.astype(np.int32)


def _reference(V, F, lam, U, B, t, clamp):
    """sum over faces of grad(w_a area + sum_c omega_c cot_c), corner by corner, and dl/dt with the sum of
    its terms' sizes."""
    V, lam, U, B, t = (np.asarray(a, dtype=np.longdouble) for a in (V, lam, U, B, t))
    P, L, W = V[F], lam[F], U[F]
    d = [P[:, (c + 2) % 3] - P[:, (c + 1) % 3] for c in range(3)]
    N = np.cross(d[1], d[2])
    s = np.sqrt((N * N).sum(1))
    dot = [(d[(c + 1) % 3] * d[(c + 2) % 3]).sum(1) for c in range(3)]
    w_a = (lam * (B - U)).sum(1)[F].sum(1) / 3
    g = np.zeros((F.shape[0], 3, 3), dtype=np.longdouble)
    omega, gt = [], np.zeros(F.shape[0], dtype=np.longdouble)
    for c in range(3):
        a, b = (c + 1) % 3, (c + 2) % 3
        lu = ((L[:, a] - L[:, b]) * (W[:, a] - W[:, b])).sum(1)
        held = np.zeros(F.shape[0], dtype=bool) if clamp is None else -dot[c] / s < clamp
        omega.append(np.where(held, 0, -t / 2 * lu))
        gt += np.where(held, -(clamp or 0.0) / 2 * lu, dot[c] / s / 2 * lu)
    Pv = -sum(omega[c] * dot[c] for c in range(3))
    coef = (w_a / 2 - Pv / s**2) / s
    for c in range(3):
        a, b = (c + 1) % 3, (c + 2) % 3
        g[:, c] = (coef[:, None] * np.cross(N, d[c]) + ((omega[a] - omega[b]) / s)[:, None] * d[c]
                   - (omega[c] / s)[:, None] * (d[b] - d[a]))
    out = np.zeros_like(V)
    np.add.at(out, F, g)
    return out, gt.sum(), np.abs(gt).sum()


@pytest.mark.parametrize("roll", [0, 1, 2])
@pytest.mark.parametrize("clamp", [None, 0.5])
@pytest.mark.parametrize("ratio", [1e-1, 1e-2, 1e-3, 1e-4])
def test_gradient_of_thin_faces(api, ratio, clamp, roll):
    V, F = _grid(ratio)
    F = np.roll(F, roll, axis=1)
    n = V.shape[0]
    rng = np.random.default_rng(3)
    for k in (1, 3, 4):
        # fields that are smooth over the surface, as those of a smoothing step are
        B, G = (V @ rng.standard_normal((3, k)) + 0.3 * ratio * rng.standard_normal((n, k)) for _ in range(2))
        t = 0.3
        mesh = api.Mesh(_t(F, torch.int32), n)
        mesh.set_cot_clamp(clamp)
        mesh.assemble(_t(V), t)
        opts = api.make_opts(rel_tol=1e-12, max_iter=400, launch="host")
        U = mesh.solve(_t(B), opts=opts)
        gV, _, gt = mesh.adjoint(_t(V), _t(B), False, U, _t(G), want_gt=True, opts=opts)
        lam = torch.empty_like(U)  # the Lambda that the gradient read
        mesh.ctx.check(mesh.ctx.lib.ig_solve_end(mesh.h, k, ctypes.c_void_p(lam.data_ptr()), None))
        ref, rt, size = _reference(V, F, lam.cpu().numpy(), U.cpu().numpy(), B, t, clamp)
        bound = 32.0 * 2.0**-53 / ratio
        err = float(np.abs(gV.cpu().numpy() - ref).max() / np.abs(ref).max())
        err_t = float(abs(gt.item() - rt) / size)
        print(f"ratio {ratio} roll {roll} clamp {clamp} k {k}: dl/dV {err:.2e} dl/dt {err_t:.2e} bound {bound:.2e}")
        assert err <= bound and err_t <= bound
        mesh.close()
