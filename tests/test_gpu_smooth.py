"""GPU: well-resolved data, where the sixth-order stage kernels take the central
flux of a smooth stencil and its nonlinear term in FP32 instead of the weights,
against the oracle -- smooth everywhere, with a patch of jumps in it (both kinds
of faces in one warp), at rest, and constant.  Tolerance as the
parity tests': 1e-12 of each component's largest value for one right-hand side
(or the rounding of its fluxes).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_26272_gb300 import weno
from paper_2603_26272_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

STAGE_TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _state(kind, nx, ny):
    w = wl.random_smooth_2d(nx=nx, ny=ny, seed=6, amp=0.1)  # up to two periods a side
    U = w["U"].copy()
    if kind == "jumps":
        U[:, :, 20:60, 30:41] *= 1.4
    if kind == "rest":  # a density wave at rest: fields that do not vary at all
        rho = U[:, 0].copy()
        U[:, 1:3] = 0.0
        U[:, 0] = rho
        U[:, 3] = 2.5
    if kind == "constant":
        U[:] = U[:, :, :1, :1]
    return U, w["dx"], w["dy"]


@pytest.mark.parametrize("kind", ["smooth", "jumps", "rest", "constant"])
@pytest.mark.parametrize("ai", [True, False])
def test_smooth_faces_match_the_oracle(ai, kind):
    nx, ny = 203, 190
    U, dx, dy = _state(kind, nx, ny)
    d = weno.make_desc(system="euler", ndim=2, nx=nx, ny=ny, x1=nx * dx, y1=ny * dy, ai=ai,
                       bc_x="periodic", bc_y="periodic")
    g = oracle.make_grid(ndim=2, nx=nx, ny=ny, dx=dx, dy=dy, bc_x="periodic", bc_y="periodic",
                         ai=int(ai))
    L = weno.rhs(d, torch.from_numpy(np.ascontiguousarray(U)).cuda()).cpu().numpy()
    ref = oracle.rhs(g, np.ascontiguousarray(U))
    # or, for a component that hardly changes, the rounding of the fluxes it is the
    # difference of: eight roundings of each of two faces a direction
    floor = 16 * 2.0 ** -53 * 2 * np.abs(U).max() * (1 / dx + 1 / dy)
    for k in range(4):
        tol = max(STAGE_TOL * np.abs(ref[:, k]).max(), floor)
        assert np.abs(L[:, k] - ref[:, k]).max() <= tol
