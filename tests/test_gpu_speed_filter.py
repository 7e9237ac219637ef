"""GPU: the speed maxima of eq. (6) on 2D grids large enough that most cells are
filtered by FP32 estimates, where one late cell holds the maxima by a small step,
at ordinary magnitudes and where c^2 is below FP32's normal numbers, and the
maxima that a stage leaves for the next one.

Reference: the same speeds in numpy's FP64.  Tolerance 1e-13: some ten roundings,
amplified by at most E / (E - rho |u|^2 / 2), which is below 20 here except in the
cold states (600, 1e-12).
"""
import numpy as np
import pytest
import torch

from paper_2603_26272_gb300 import weno

pytestmark = pytest.mark.gpu

NX, NY = 1024, 640  # k_alpha: 262144 cells a round


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _alpha(U, gamma):
    rho, mx, my, E = U[0]
    u, v = mx / rho, my / rho
    c = np.sqrt(gamma * (gamma - 1) * (E - 0.5 * (mx * u + my * v)) / rho)
    return np.array([[np.abs(w + k * c).max() for k in (-1, 0, 0, 1)] for w in (u, v)])


# name: rho, speed, rho e, gamma, tolerance
STATES = {
    "ordinary": (1.0, 0.3, 2.5, 1.4, 1e-13),
    "cold_dense": (5e17, 2.8e-18, 1e-20, 1.4, 1e-12),
    "soft_dense": (5e17, 1e-25, 4e-18, 1 + 1e-9, 1e-13),
    "large": (1e-17, 1e16, 4e16, 1.4, 1e-13),
    "tiny": (1e-25, 1e-3, 1e-30, 1.4, 1e-13),
}


@pytest.mark.parametrize("more", [1e-10, 1e-4, 0.3])
@pytest.mark.parametrize("name", STATES)
def test_the_maxima_of_one_late_cell_are_found(name, more):
    rho, w, e, gamma, tol = STATES[name]
    g = np.random.default_rng(3)
    u, v = (w * g.uniform(-0.9, 0.9, (NY, NX)) for _ in range(2))
    ei = e * g.uniform(0.5, 0.999, (NY, NX))
    # a first-round cell each
    ei[0, 5], u[0, 6], u[0, 7], v[0, 8], v[0, 9] = e, w, -w, w, -w
    ei[0, 6:10] = 0.5 * e
    for k, (a, b, f) in enumerate([(0, 0, 1), (1, 0, 0), (0, 1, 0), (1, 0, 1), (0, -1, 1),
                                  (0.995, 0, 1)]):
        j, i = 400 + 40 * k, 77 + 31 * k  # later ones, a step above
        u[j, i], v[j, i] = a * w * (1 + more), b * w * (1 + more)
        ei[j, i] = e * (1 + more) if f else 0.7 * e
    r = np.full((NY, NX), rho)
    U = np.stack([r, r * u, r * v, ei + 0.5 * r * (u * u + v * v)])[None]
    d = weno.make_desc(system="euler", ndim=2, nx=NX, ny=NY, x1=NX / 64, y1=NY / 64, gamma=gamma)
    al, _ = weno.wavespeeds(d, torch.from_numpy(U).cuda())
    ref = _alpha(U, gamma)
    assert np.all(np.abs(al.cpu().numpy()[0] - ref) <= tol * ref.max())


@pytest.mark.parametrize("precision", ["fp64", "fp32_recon"])
@pytest.mark.parametrize("nx,ny", [(96, 96), (1000, 650)])
def test_a_step_leaves_the_maxima_of_its_result(nx, ny, precision):
    """The clock after two steps of one solve: the second dt comes from the maxima
    formed while the first step's last stage wrote its cells."""
    x, y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)
    rho, u, v = 1 + 0.2 * np.sin(7 * x + y), 0.3 * np.cos(5 * y), 0.4 * np.sin(9 * x)
    p = 1 + 4 * np.exp(-400 * ((x - 0.8) ** 2 + (y - 0.9) ** 2))
    U = np.stack([rho, rho * u, rho * v, p / 0.4 + 0.5 * rho * (u * u + v * v)])[None]
    d = weno.make_desc(system="euler", ndim=2, nx=nx, ny=ny, x1=1.0, y1=1.0, precision=precision)
    one = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    two = one.clone()
    dt = weno.step(d, one)[0]
    t, n = weno.solve(d, two, 1e3, max_steps=2, allow_max_steps=True)
    _, second = weno.wavespeeds(d, one)
    a = _alpha(one.cpu().numpy(), 1.4)
    assert n[0] == 2
    assert t[0] == dt + float(second[0])
    al, _ = weno.wavespeeds(d, one)
    assert np.all(np.abs(al.cpu().numpy()[0] - a) <= 1e-13 * a.max())
