"""GPU: data that is cubic about three equal cells but for a fifth difference of
r5.  One smoothness indicator is then 0 and the weights of the other candidates are
what r5 leaves them, below the integer path's units, which leaves those fields to
FP64.  Every layout (lanes of a small 1D problem, one thread a face of a batch, 2D
tiles along x and y, both scalar layouts) against the oracle; the 1D layouts against
each other bit for bit.

Tolerance: 1e-12 of each component's largest value as in the parity tests, 16
roundings of the fluxes at two faces, or 16 times what the oracle's own two orders of
summation differ by (tests/test_oracle_rounding.py; r5 is 2^6 roundings and more, so
that the weights do not hang on those).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_26272_gb300 import weno

pytestmark = pytest.mark.gpu

OPTS = [(True, 1e-40), (False, 1e-40), (True, 1e-12)]
SIZES = [9, 13, 17, 33]
R5 = [2.0 ** -45, 2.0 ** -40]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _plateau(n, r5):
    x = (np.arange(n) + 0.5) / n - 0.5
    h = 1.0 / n
    return 1.1 + 8 * x * (x * x - h * h) * (1 + x * x * (r5 / (960 * h ** 5)))


def _both(g, U):
    with oracle.rounding_variant("reversed"):
        other = oracle.rhs(g, U)
    return oracle.rhs(g, U), other


def _near(L, refs, flux, n):
    ref, other = refs
    for k in range(ref.shape[1]):
        tol = max(1e-12 * np.abs(ref[:, k]).max(), 32 * 2.0 ** -53 * flux * n,
                  16 * np.abs(ref - other)[:, k].max())
        assert np.abs(L[:, k] - ref[:, k]).max() <= tol


def _rhs(d, U):
    return weno.rhs(d, torch.from_numpy(np.ascontiguousarray(U)).cuda()).cpu().numpy()


@pytest.mark.parametrize("ai,eps", OPTS)
@pytest.mark.parametrize("r5", R5)
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("system", ["euler", "advection", "burgers"])
def test_1d(system, n, r5, ai, eps):
    rho = _plateau(n, r5)
    U = rho[None] if system != "euler" else np.stack([rho, 0.7 * rho, 2.5 + 0.245 * rho])
    U = np.ascontiguousarray(U[None, :, None, :])
    ref = _both(oracle.make_grid(system=system, nx=n, dx=1.0 / n, ai=int(ai), eps=eps), U)
    out = []
    for nb in (1, 2000):
        d = weno.make_desc(system=system, ndim=1, nx=n, nbatch=nb, x1=1.0, ai=ai, eps=eps)
        L = _rhs(d, np.repeat(U, nb, 0))
        assert (L == L[:1]).all()
        _near(L[:1], ref, 4.0, n)
        out.append(L[:1])
    assert (out[0] == out[1]).all()


@pytest.mark.parametrize("along", ["x", "y"])
@pytest.mark.parametrize("ai,eps", OPTS)
@pytest.mark.parametrize("r5", R5)
@pytest.mark.parametrize("n", SIZES)
def test_2d(n, r5, ai, eps, along):
    """Lines at rest beside lines that move, which set the speeds: at rest the fluxes of
    equal cells are equal to the last bit (a moving cell's are rounded apart)."""
    m = 22
    rho = np.broadcast_to(_plateau(n, r5), (m, n))
    w = np.where(np.arange(m) < 8, 0.7, 0.0)[:, None] * rho
    U = np.stack([rho, w, 0 * rho, 2.5 + 0.5 * w * w / rho])
    if along == "y":
        U = U[[0, 2, 1, 3]].transpose(0, 2, 1)
    U = np.ascontiguousarray(U[None])
    ny, nx = U.shape[2:]
    d = weno.make_desc(system="euler", ndim=2, nx=nx, ny=ny, x1=nx / n, y1=ny / n, ai=ai, eps=eps)
    g = oracle.make_grid(ndim=2, nx=nx, ny=ny, dx=1.0 / n, dy=1.0 / n, ai=int(ai), eps=eps)
    L = _rhs(d, U)
    still = (slice(None), slice(None), slice(12, None)) if along == "x" else \
        (slice(None), slice(None), slice(None), slice(12, None))
    _near(L[still], [q[still] for q in _both(g, U)], 4.0, n)
