"""GPU: where the stage kernels change between the integer-pipe reconstruction
(csrc/weno_fixed.cuh, with and without its sensitivity term) and the FP64 one,
every route gives the oracle's right-hand side.

The rule goes by eps and mu_0 (weight_mode: left out at eps <= 2^-126 and
mu_0 <= 2^-100) and, per field, by the largest difference (below mu_0, where
that rule leaves the term out, and below 2^-959: FP64).  Tolerance as the
parity tests': 1e-12 of each component's largest value for one right-hand side.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_26272_gb300 import weno
from paper_2603_26272_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

STAGE_TOL = 1e-12
UP = float(np.nextafter(2.0 ** -126, 1.0))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _data(kind):
    if kind == "2d":  # ragged tiles, jumps and smooth parts
        w = wl.random_smooth_2d(nx=50, ny=37, seed=3)
        U = w["U"].copy()
        U[:, :, 10:20, 12:30] *= 1.7
        return dict(system="euler", ndim=2, nx=50, ny=37, y1=37 * w["dy"], x1=50 * w["dx"]), U
    n = 300
    if kind == "burgers":
        w = wl.burgers_sine(n=n)
        return dict(system="burgers", ndim=1, nx=n), w["U"].copy()
    w = wl.shock_density(n=n)
    return dict(system="euler", ndim=1, nx=n, x0=-5.0, x1=5.0), w["U"].copy()


@pytest.mark.parametrize("ai,eps,mu0,scale", [
    (True, 2.0 ** -126, 2.0 ** -100, 0), (True, UP, 2.0 ** -100, 0), (True, 2.0 ** -126, 2.0 ** -99, 0),
    (True, 1e-40, 1e-40, -300), (True, 1e-40, 1e-40, -130), (True, 1e-40, 1e-40, 300),
    (True, 1e-12, 1e-40, 0), (True, 1e-2, 1e-3, 0), (True, 1e-6, 1e-40, -300), (True, 1e-40, 1e-2, 0),
    (False, 1e-40, 1e-40, 0), (False, 1e-40, 1e-40, -60), (False, 1e-6, 1e-40, 0), (False, 1e-6, 1e-40, 60),
])
@pytest.mark.parametrize("kind", ["1d", "1d_batch", "2d", "burgers"])
def test_every_route_of_the_reconstruction_matches_the_oracle(kind, ai, eps, mu0, scale):
    args, U = _data(kind.split("_")[0])
    if kind == "burgers" and scale:
        pytest.skip("Burgers' flux is not homogeneous of degree one")
    U = np.ascontiguousarray(U) * 2.0 ** scale
    nb = 200 if kind == "1d_batch" else 1  # enough tiles for the one-thread-a-face layout
    d = weno.make_desc(eps=eps, mu0=mu0, ai=ai, nbatch=nb, **{"ny": U.shape[2], **args})
    g = oracle.make_grid(system=args["system"], ndim=args["ndim"], nx=d.nx, ny=d.ny,
                         dx=(d.x1 - d.x0) / d.nx, dy=(d.y1 - d.y0) / d.ny if d.ndim == 2 else 1.0,
                         eps=eps, mu0=mu0, ai=int(ai))
    L = weno.rhs(d, torch.from_numpy(np.repeat(U, nb, axis=0)).cuda()).cpu().numpy()
    ref = oracle.rhs(g, U)
    assert (L == L[:1]).all()
    for k in range(ref.shape[1]):
        top = np.abs(ref[:, k]).max() or np.abs(ref).max()
        assert np.abs(L[:1, k] - ref[:, k]).max() <= STAGE_TOL * top
