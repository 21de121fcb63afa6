"""dJ/du of the checkpointed FP32 gradient against the FP64 gradient of the same
inputs.  dJ/du sees only what differs between the velocities of lam, a thousandth
of lam itself on fine grids, so it shows roundings that lam and dJ/dphi0 hide.

Tolerance 1e-6 of the larger component: every term is a product of at most ten
factors rounded once (6e-8 each, uncorrelated: 2e-7), the cells' own roundings
average out, and the forward run's differ by a few 1e-7 in the FP32 state."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def _wide(ny):
    xf, yf = I.tanh_faces(2048, 2.0), I.tanh_faces(ny, 1.5)
    return I.Problem(xf=xf, yf=yf, bc=(1,) * 4, bc_value=(1.0, 0.5, 0.5, 0.5), c=10.0, u=(0.05, 0.0), b=(0.0, 1.0),
                     alpha=0.01, d=(0.0, 0.0, 1.0), dt=I.cfl_dt(xf, yf, 10.0, 0.4))


CASES = {"periodic_512": lambda: I.burgers(512)[0], "periodic_171x150": lambda: I.burgers(171, 150)[0],
         "walls_2048x128": lambda: _wide(128), "walls_340x360": lambda: I.nonuniform(340, 360)[0]}


@pytest.mark.parametrize("seed", [1, 2, 3])
@pytest.mark.parametrize("kind", ["rows", "tiled"])
@pytest.mark.parametrize("name", list(CASES))
def test_dj_du_of_the_gradient(name, kind, seed):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import Solver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = CASES[name]()
    xc, yc = p.centres()
    area = np.outer(np.diff(p.yf), np.diff(p.xf))
    phi0 = torch.tensor(I.smooth_phi0(xc, yc, seed=seed), device="cuda").float()
    misfit = torch.tensor(area / area.mean() * (I.smooth_phi0(xc, yc, seed=seed + 20) - 0.9), device="cuda").float()
    out = {}
    for prec in (64, 32):
        s = Solver(p, precision=prec)
        s.set_adjoint_kernel(kind)
        out[prec] = s.gradient(phi0.to(s.dtype), 20, misfit.to(s.dtype), checkpoint_every=20, with_u=True)
        s.close()
    (g6, _, u6), (g3, _, u3) = out[64], out[32]
    err = np.abs(np.subtract(u3, u6)).max() / np.abs(u6).max()
    assert float((g3.double() - g6).norm() / g6.norm()) <= 2e-6
    assert err <= 1e-6


@pytest.mark.parametrize("name", ["periodic_512", "walls_2048x128"])
def test_tiled_dj_dphi0_is_as_exact_as_the_row_kernels(name):
    """Both FP32 kernels round lambda_0 the same few times a step, so their distances from 64 bits are the same
    but for the order of their sums: within a quarter."""
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import Solver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = CASES[name]()
    xc, yc = p.centres()
    phi0 = torch.tensor(I.smooth_phi0(xc, yc, seed=1), device="cuda").float()
    misfit = torch.tensor(I.smooth_phi0(xc, yc, seed=21) - 0.9, device="cuda").float()
    g = {}
    for prec, kind in ((64, "tiled"), (32, "tiled"), (32, "rows")):
        s = Solver(p, precision=prec)
        s.set_adjoint_kernel(kind)
        g[prec, kind] = s.gradient(phi0.to(s.dtype), 20, misfit.to(s.dtype), checkpoint_every=20)[0].double()
        s.close()
    ref = g[64, "tiled"]
    tiled, rows = (float((g[32, k] - ref).norm() / ref.norm()) for k in ("tiled", "rows"))
    assert tiled <= 1.25 * rows, (tiled, rows)
