"""The parameter derivatives of one adjoint step are sums over the slots that
the step's own kernels write: neither those of another kernel's earlier step on
the same context nor memory that nothing wrote may enter.  Grids whose
row-marching plan has more slots than the tiled kernel, against a context that
only ever ran the tiled one, bit for bit."""
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("nx,ny", [(512, 512), (340, 360)])
def test_derivatives_do_not_depend_on_the_step_before(nx, ny, walls):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import Solver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p, phi0 = (I.nonuniform if walls else I.burgers)(nx, ny)

    def solver(kind):
        s = Solver(p, precision=32)
        s.set_adjoint_kernel(kind)
        return s

    fresh = solver("tiled")
    fresh.init_phi(torch.tensor(phi0, device="cuda"))
    fresh.step(2)
    f = fresh.save_state()
    gen = torch.Generator(device="cuda").manual_seed(nx + walls)
    mu = torch.randn(f.shape, generator=gen, device="cuda")
    lam, da, du = fresh.adjoint_step(f, mu, with_u=True)
    used = solver("rows")
    used.adjoint_step(f, 1e3 * mu, with_u=True)  # leaves the row-marching kernel's sums behind
    used.set_adjoint_kernel("tiled")
    lam2, da2, du2 = used.adjoint_step(f, mu, with_u=True)
    assert torch.equal(lam, lam2) and torch.equal(da, da2) and torch.equal(du, du2)
    for s in (fresh, used):
        s.sync()
        s.close()
