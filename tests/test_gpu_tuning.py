"""GPU: the tile autotuner keeps one choice per kernel: weights with a sensitivity
term that counts run another kernel than the default ones and are timed on their
own, whichever came first, and a call captured in a graph still takes the choice
made for the other weights on that grid.

A call that times shapes waits for its stream, so an event recorded before it,
behind a kernel of some milliseconds, has passed when it returns; a call that
does not returns while that kernel runs.
"""
import pytest
import torch

from paper_2603_26272_gb300 import weno
from paper_2603_26272_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(autouse=True)
def _no_forced_tile(monkeypatch):
    monkeypatch.delenv("WENO_TILE2D", raising=False)


def _waits(d, U, out, ws):
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)  # about 50 ms
    before = torch.cuda.Event()
    before.record()
    weno.rhs(d, U, out=out, ws=ws)
    waited = before.query()
    torch.cuda.synchronize()
    return waited


def _problem(nx, ny, **opt):
    U = torch.from_numpy(wl.random_smooth_2d(nx=nx, ny=ny, seed=4)["U"].copy()).cuda()
    d = weno.make_desc(system="euler", ndim=2, nx=nx, ny=ny, x1=nx / 64, y1=ny / 64, **opt)
    return d, U, torch.empty_like(U), weno.workspace(d)


@pytest.mark.parametrize("nx,first,second", [(67, {}, {"eps": 1e-6}), (69, {"eps": 1e-6}, {})])
def test_weights_with_another_kernel_are_timed_on_their_own(nx, first, second):
    a, b = _problem(nx, 45, **first), _problem(nx, 45, **second)
    assert _waits(*a) and not _waits(*a)
    assert _waits(*b) and not _waits(*b)
    assert not _waits(*a)


def test_one_kernel_is_timed_once():
    for opt in ({"precision": "fp32_recon"}, {"p": 2.0}):
        a, b = _problem(71, 43, **opt), _problem(71, 43, eps=1e-6, **opt)
        assert _waits(*a) and not _waits(*b)


@pytest.mark.parametrize("nx,first,second", [(73, {}, {"eps": 1e-6}), (75, {"eps": 1e-6}, {})])
def test_capture_takes_the_choice_of_the_other_weights(nx, first, second):
    a, b = _problem(nx, 45, **first), _problem(nx, 45, **second)
    weno.rhs(a[0], a[1], out=a[2], ws=a[3])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        weno.rhs(b[0], b[1], out=b[2], ws=b[3])
    b[2].fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    got = b[2].clone()
    weno.rhs(b[0], b[1], out=b[2], ws=b[3])
    torch.cuda.synchronize()
    assert torch.equal(got, b[2])
