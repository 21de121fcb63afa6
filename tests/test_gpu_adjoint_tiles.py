"""The row-marching FP32 adjoint on a grid large enough that, with walls, its
interior tiles run as a launch of their own: lam and the parameter derivatives
of one step against the FP64 adjoint of the same inputs.  Tolerances as for
the other FP32 adjoint checks: 2e-5 (lam, relative L2), 2e-4 (derivatives)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [(True, True), (True, False), (False, True)])
@pytest.mark.parametrize("nx,ny", [(1404, 1501), (1372, 1489)])  # last strip of 4 columns, of 28; clipped last rows
def test_interior_and_wall_tiles_together(nx, ny, walls):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import Solver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xf = I.tanh_faces(nx, 1.5) if walls[0] else I.uniform_faces(nx)
    yf = I.tanh_faces(ny, 1.5) if walls[1] else I.uniform_faces(ny)
    p = I.Problem(xf=xf, yf=yf, bc=(int(walls[0]),) * 2 + (int(walls[1]),) * 2, bc_value=(1.2, 0.6, 0.9, 0.7), c=10.0,
                  u=(0.3, -0.2), b=(0.0, 0.0, 0.5), alpha=0.02, d=(0.0, 1.0), dt=I.cfl_dt(xf, yf, 10.0, 0.45))
    xc, yc = p.centres()
    phi0 = torch.tensor(I.smooth_phi0(xc, yc, seed=3), device="cuda")
    s64, s32 = Solver(p, precision=64), Solver(p, precision=32)
    s64.init_phi(phi0)
    s64.step(3)
    f = s64.save_state().float()
    # mu: a smooth field seen by every velocity, with an odd part
    g = torch.tensor(I.smooth_phi0(xc, yc, seed=4) - 1.0, device="cuda").float()
    mu = torch.stack([g * (1.0 + 0.05 * i) for i in range(9)])
    lam, da, du = s64.adjoint_step(f.double(), mu.double(), with_u=True)
    got, ga, gu = s32.adjoint_step(f, mu, with_u=True)
    s64.sync()
    s32.sync()
    assert float((got.double() - lam).norm() / lam.norm()) <= 2e-5
    assert abs(float(ga - da)) <= 2e-4 * abs(float(da))
    assert float((gu - du).abs().max()) <= 2e-4 * float(du.abs().max())
    assert np.isfinite(float(ga))
    s64.close()
    s32.close()
