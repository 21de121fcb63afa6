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


TILED = {"resident_fp32": lambda: (I.burgers(70, 45), 32), "resident_fp64": lambda: (I.burgers(64, 64), 64),
         "resident_walls": lambda: (I.nonuniform(330, 517), 32), "resident_source": lambda: (I.cde_source(60), 32),
         "sequence": lambda: (I.burgers(900, 700), 32), "sequence_walls": lambda: (I.nonuniform(1021, 643), 32)}


@pytest.mark.parametrize("name", list(TILED))
def test_a_tile_that_never_answers_ends_the_launch(name):
    """One tile's messages (or its step count) never come: every tile's wait runs out, the launch ends by
    itself, the status says so, and a fresh context computes what one that never failed does."""
    import time

    from paper_1906_11036_gb300.dugks import DugksError, Solver

    (p, phi0), prec = TILED[name]()
    phi0 = torch.tensor(phi0, device="cuda")
    out = []
    for fails in (True, False):
        if fails:
            s = Solver(p, precision=prec)
            s.init_phi(phi0)
            s.step(3)
            s.sync()
            t = time.perf_counter()
            s.tile_timeout_check(2000)
            with pytest.raises(DugksError) as ei:
                s.sync()
            assert ei.value.status == 7 and time.perf_counter() - t < 1.0
            s.step(4)
            with pytest.raises(DugksError) as ei:
                s.get_phi_host()
            assert ei.value.status == 7
            s.close()
        s = Solver(p, precision=prec)
        s.init_phi(phi0)
        s.step(7)
        out.append(s.save_state())
        s.sync()
        s.close()
    assert torch.equal(*out)


def test_no_tiles_to_wait_for():
    from paper_1906_11036_gb300.dugks import DugksError, Solver

    p, _ = I.burgers(40, 30)
    s = Solver(p, precision=32, kernel="naive")
    with pytest.raises(DugksError) as ei:
        s.tile_timeout_check(2000)
    assert ei.value.status == 5
    s.close()
