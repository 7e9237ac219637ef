"""GPU: right-hand sides beside strong jumps, where the sixth-order kernels leave
faces of the integer path to FP64, against the oracle in every layout (lanes of a
small 1D problem, one thread a face of a batch, 2D tiles along x and y), and the
1D layouts against each other bit for bit.  Tolerance as the parity tests':
1e-12 of each component's largest value for one right-hand side (2D: or the
rounding of its fluxes, as the momentum across the jump's plane is 0 but for the
pressure's rounding).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_26272_gb300 import weno

pytestmark = pytest.mark.gpu

STAGE_TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _euler(x, kind, ratio):
    at = np.where(x < 0.5, ratio, 1.0)
    rho, u, v, p = 1 + 0.2 * np.sin(6 * np.pi * x), 0 * x, 0 * x, 0 * x + 1
    if kind == "pressure":
        p = at
    if kind == "waves":
        u, v = 0.3 * np.sin(2 * np.pi * x + 0.2), 0.4 * np.sin(4 * np.pi * x)
        p = at * (1 + 0.1 * np.sin(8 * np.pi * x))
    if kind == "contact":
        rho, u, v, p = rho * at, 0.5 + 0 * x, 0.1 + 0 * x, 1 + 0.1 * np.sin(4 * np.pi * x)
    return rho, u, v, p


def _check(L, ref, floor=0.0):
    for k in range(ref.shape[1]):
        top = np.abs(ref[:, k]).max() or np.abs(ref).max()
        assert np.abs(L[:, k] - ref[:, k]).max() <= max(STAGE_TOL * top, floor if k in (1, 2) else 0)


CASES = [("pressure", 10.0 ** k) for k in (2, 5, 7, 9, 12, 16, 18)] + \
        [("waves", 1e3), ("waves", 1e6), ("waves", 1e9), ("contact", 1e2)]


@pytest.mark.parametrize("ai,eps", [(True, 1e-40), (True, 1e-12), (False, 1e-40)])
@pytest.mark.parametrize("kind,ratio", CASES)
def test_1d_beside_a_jump_matches_the_oracle(kind, ratio, ai, eps):
    n = 200
    rho, u, _, p = _euler((np.arange(n) + 0.5) / n, kind, ratio)
    U = np.stack([rho, rho * u, p / 0.4 + 0.5 * rho * u * u])[None, :, None, :]
    opt = dict(eps=eps, mu0=1e-40)
    ref = oracle.rhs(oracle.make_grid(nx=n, dx=1.0 / n, ai=int(ai), **opt), np.ascontiguousarray(U))
    out = []
    for nb in (1, 300):  # the lane layout, one thread a face
        d = weno.make_desc(system="euler", ndim=1, nx=n, nbatch=nb, x1=1.0, ai=ai, **opt)
        L = weno.rhs(d, torch.from_numpy(np.ascontiguousarray(np.repeat(U, nb, 0))).cuda()).cpu().numpy()
        assert (L == L[:1]).all()
        _check(L[:1], ref)
        out.append(L[:1])
    assert (out[0] == out[1]).all()


@pytest.mark.parametrize("along", ["x", "y"])
@pytest.mark.parametrize("kind,ratio", CASES)
def test_2d_beside_a_jump_matches_the_oracle(kind, ratio, along):
    nx, ny = 50, 37
    n = nx if along == "x" else ny
    rho, u, v, p = (np.broadcast_to(q[None, :] if along == "x" else q[:, None], (ny, nx))
                    for q in _euler((np.arange(n) + 0.5) / n, kind, ratio))
    if along == "y":
        u, v = v, u
    # (a wave across the jump too)
    other = np.arange(ny)[:, None] / ny if along == "x" else np.arange(nx)[None, :] / nx
    rho = rho * (1 + 0.1 * np.sin(2 * np.pi * other))
    U = np.ascontiguousarray(np.stack([rho, rho * u, rho * v,
                                       p / 0.4 + 0.5 * rho * (u * u + v * v)])[None])
    d = weno.make_desc(system="euler", ndim=2, nx=nx, ny=ny, x1=1.0, y1=1.0)
    g = oracle.make_grid(ndim=2, nx=nx, ny=ny, dx=1.0 / nx, dy=1.0 / ny)
    # eight roundings of each of two faces of the momentum fluxes a direction
    flux = (p + rho * np.maximum(u * u, v * v)).max()
    _check(weno.rhs(d, torch.from_numpy(U).cuda()).cpu().numpy(), oracle.rhs(g, U),
           16 * 2.0 ** -53 * flux * (nx + ny))


@pytest.mark.parametrize("system", ["advection", "burgers"])
def test_scalar_layouts_agree_beside_a_jump(system):
    n = 300
    x = (np.arange(n) + 0.5) / n
    u = np.where((x > 0.2) & (x < 0.4), 1.0, 1e-7 * np.sin(8 * np.pi * x))
    u[x > 0.7] = 0.0
    U = u[None, None, None, :]
    ref = oracle.rhs(oracle.make_grid(system=system, nx=n, dx=1.0 / n), np.ascontiguousarray(U))
    out = []
    for nb in (1, 300):
        d = weno.make_desc(system=system, ndim=1, nx=n, nbatch=nb, x1=1.0)
        L = weno.rhs(d, torch.from_numpy(np.ascontiguousarray(np.repeat(U, nb, 0))).cuda()).cpu().numpy()
        assert (L == L[:1]).all()
        out.append(L[:1])
    assert (out[0] == out[1]).all()
    # each cell to the precision of its own surroundings (the kernel's FP64 path beside the jump)
    near = np.array([np.abs(np.take(u, range(i - 1, i + 2), mode="clip")).max() for i in range(n)])
    flux = near if system == "advection" else np.maximum(near * np.abs(u).max(), near * near)
    tol = STAGE_TOL * flux * n
    assert (np.abs(out[0] - ref)[0, 0, 0] <= np.maximum(tol, 1e-40)).all()
