"""After a bounded wait has expired no call hands out a result as if nothing
had happened: whatever synchronises returns DUGKS_ERR_TIMEOUT."""
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


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("call", ["get_phi_host", "get_phi", "mass", "gradient"])
def test_results_after_an_expired_wait(call, prec):
    from paper_1906_11036_gb300.dugks import DugksError, Solver

    p, phi0 = I.burgers(40, 30)
    phi0 = torch.tensor(phi0, dtype=torch.float32 if prec == 32 else torch.float64, device="cuda")
    s = Solver(p, precision=prec)
    calls = {"get_phi_host": s.get_phi_host, "get_phi": lambda: s.get_phi(mass=True), "mass": s.mass,
             "gradient": lambda: s.gradient(phi0, 6, phi0, checkpoint_every=3, with_u=True)}
    s.init_phi(phi0)
    s.step(3)
    calls[call]()
    s.wait_timeout_check(2000)
    s.step(3)
    for _ in range(2):
        with pytest.raises(DugksError) as ei:
            calls[call]()
        assert ei.value.status == 7
    s.close()


@pytest.mark.parametrize("nx,ny,prec", [(40, 30, 32), (40, 30, 64), (900, 700, 32)])
def test_many_step_launches_after_an_expired_wait_leave_the_state(nx, ny, prec):
    """The kernels that take many steps per launch end at once where the error word is set already: they
    neither advance the state nor count steps that other tiles would take as done."""
    from paper_1906_11036_gb300.dugks import DugksError, Solver

    p, phi0 = I.burgers(nx, ny)
    s = Solver(p, precision=prec)
    s.init_phi(torch.tensor(phi0, device="cuda"))
    s.step(4)
    before = s.save_state()
    s.wait_timeout_check(2000)
    s.step(6)
    after = s.save_state()
    with pytest.raises(DugksError) as ei:
        s.sync()
    assert ei.value.status == 7
    assert torch.equal(before, after)
    s.close()
