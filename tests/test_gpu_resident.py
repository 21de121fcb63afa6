"""The kernels that take many steps per launch, at the edges of their tiling:
the resident step (tiles exchanging their rims) and the tile sequence of the
row-marching step (tiles waiting for their neighbours), against the batched
solver, which takes a launch per step, bit for bit in FP32; the resident step
in FP64 against the one-thread-per-cell kernel; both replayed from a graph."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    torch.cuda.set_device(0)


# one row or column per tile, one tile more than there are SMs on an axis, tiles of uneven size, the
# largest tiles of the range (x-fluxes in place); then tile sequences: two strips, a clipped last tile,
# tiles of the least height
SIZES = [(152, 1), (1, 153), (3, 305), (31, 33), (62, 31), (97, 620), (257, 509), (512, 512), (612, 617), (700, 610),
         (31, 20000), (5000, 90), (1021, 643), (1500, 601)]


def _problem(nx, ny, xwall, ywall, linear=False):
    xf = I.tanh_faces(nx, 1.5) if xwall else I.uniform_faces(nx)
    yf = I.tanh_faces(ny, 1.5) if ywall else I.uniform_faces(ny)
    bc = (int(xwall),) * 2 + (int(ywall),) * 2
    p = I.Problem(xf=xf, yf=yf, bc=bc, bc_value=(1.2, 0.6, 0.9, 0.7), c=10.0, u=(0.3, -0.2),
                  b=(0.0, 1.0) if linear else (0.0, 0.0, 0.5), alpha=0.02, d=(0.0, 1.0) if linear else (0.0, 1.0, 0.5),
                  dt=I.cfl_dt(xf, yf, 10.0, 0.45))
    xc, yc = p.centres()
    return p, torch.tensor(I.smooth_phi0(xc, yc, seed=nx + 7 * ny), device="cuda")


def _steps(p, phi0, prec, chunks, kernel="auto"):
    from paper_1906_11036_gb300.dugks import Solver

    s = Solver(p, precision=prec, kernel=kernel)
    s.init_phi(phi0)
    for n in chunks:
        s.step(n)
    f = s.save_state()
    s.sync()
    s.close()
    return f


@pytest.mark.parametrize("walls", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_fp32_equals_the_row_marching_step(nx, ny, walls):
    from paper_1906_11036_gb300.dugks import BatchSolver

    p, phi0 = _problem(nx, ny, *walls, linear=nx % 2 == 0)
    b = BatchSolver([p])
    b.init_phi(0, phi0)
    b.step(9)
    ref = b.save_state(0)
    b.sync()
    b.close()
    assert torch.equal(_steps(p, phi0, 32, (4, 5)), ref)


@pytest.mark.parametrize("nx,ny", [(152, 1), (1, 153), (31, 33), (62, 31), (97, 420), (257, 131), (410, 433), (450, 440)])
def test_fp64_matches_the_cell_kernel(nx, ny):
    """FP64 differs from the other kernels only by the order of its operations: 1e-13 after 6 steps
    (each step rounds at 1.1e-16 relative, a few tens of operations deep)."""
    for walls in ((False, False), (True, True)):
        p, phi0 = _problem(nx, ny, *walls, linear=nx % 2 == 0)
        got, ref = _steps(p, phi0, 64, (6,)), _steps(p, phi0, 64, (6,), "naive")
        assert float((got - ref).norm() / ref.norm()) <= 1e-13


@pytest.mark.parametrize("nx,ny,prec", [(70, 45, 32), (70, 45, 64), (900, 700, 32)])
def test_replay_from_a_graph(nx, ny, prec):
    """A captured step call advances the state at every replay as direct calls do."""
    from paper_1906_11036_gb300.dugks import Solver

    p, phi0 = _problem(nx, ny, True, False)
    ref = _steps(p, phi0, prec, (3, 4, 4, 4))
    s = Solver(p, precision=prec)
    stream = torch.cuda.Stream()
    s.set_stream(stream)
    s.init_phi(phi0)
    s.step(3)
    s.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        s.step(4)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(s.save_state(), ref)
    s.sync()
    s.close()


def test_removing_a_source_returns_to_the_plain_step():
    from paper_1906_11036_gb300.dugks import Solver

    p, phi0 = I.cde_source(48)
    phi0 = torch.tensor(phi0, device="cuda")
    s = Solver(p, precision=32)
    s.init_phi(phi0)
    s.step(40)  # more steps than one launch takes with source terms
    a = s.get_phi().double().cpu().numpy()
    s.set_source(())
    s.init_phi(phi0)
    s.step(7)
    f = s.save_state()
    s.sync()
    s.close()
    assert torch.equal(f, _steps(p.with_(source=()), phi0, 32, (7,)))
    exact = p.meta["exact"](40 * p.dt)
    assert np.abs(a - exact).sum() / np.abs(exact).sum() <= 2e-2  # the scheme's own distance on this grid
