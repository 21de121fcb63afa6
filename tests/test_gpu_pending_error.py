"""A call that fails on the device reports its error once: the next launch, on
whatever context, does not find it again."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
def test_a_creation_that_does_not_fit_leaves_no_error_behind(dim):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import DugksError, Solver, Solver3

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if dim == 2:
        p, phi0 = I.burgers(64)
        f = np.linspace(0.0, 1.0, 100_001)  # 360 GB a buffer
        large = p.with_(xf=f, yf=f, dt=I.cfl_dt(f, f, p.c, 0.4))
        make = lambda q: Solver(q, precision=32)  # noqa: E731
    else:
        p, phi0 = I.burgers3d(24)
        f = np.linspace(0.0, 1.0, 2_001)  # 480 GB a buffer and more
        large = I.Problem3(**{**p.__dict__, "xf": f, "yf": f, "zf": f, "dt": I.cfl_dt3(f, f, f, p.c, 0.4)})
        make = lambda q: Solver3(q, precision=32)  # noqa: E731
    s = make(p)
    x = torch.as_tensor(phi0, device="cuda").float()
    with pytest.raises(DugksError) as ei:
        make(large)
    assert ei.value.status == 6
    s.init_phi(x)
    s.step(2)
    s.get_phi()
    s.sync()
    s.close()
