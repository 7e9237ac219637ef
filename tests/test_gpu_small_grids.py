"""GPU: the tile the other orders take on grids with few tiles, against those of
larger grids: a problem alone takes the 8x8 tile, the same problem repeated in a
batch one of the large ones (16x15 for the first three sizes, 20x15 for the last
two), and every face is the same arithmetic, so the right-hand sides are equal
bit for bit.
"""
import numpy as np
import pytest
import torch

from paper_2603_26272_gb300 import weno
from paper_2603_26272_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("bc", ["transmissive", "periodic"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (7, 9), (8, 8), (17, 16), (50, 33)])
@pytest.mark.parametrize("order", [4, 8, 10])
def test_small_tile_bitwise_large_tiles(order, nx, ny, bc):
    U = wl.random_smooth_2d(nx=64, ny=64, seed=8)["U"][:, :, :ny, :nx].copy()
    U[:, :, ny // 2:, nx // 2:] *= 1.7
    tiles = -(-nx // 16) * -(-ny // 16)
    copies = torch.cuda.get_device_properties(0).multi_processor_count // tiles + 1
    out = []
    for nb in (1, copies):
        d = weno.make_desc(system="euler", ndim=2, nx=nx, ny=ny, nbatch=nb, x1=nx / 64,
                           y1=ny / 64, order=order, bc_x=bc, bc_y=bc)
        x = torch.from_numpy(np.ascontiguousarray(np.repeat(U, nb, 0))).cuda()
        out.append(weno.rhs(d, x))
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[1], out[0].expand_as(out[1]))
