"""Calls of a few steps on FP32 grids beyond the resident size: whether a call
runs as single launches or as one sequence of tiles, whatever mixture of calls
makes up a run, the state is the same bits; on grids of each class that the
rule tells apart."""
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

# less than 0.6 waves of segments, nearly one, more than one, long segments (periodic, walls)
GRIDS = {"700x600": (700, 600, False), "1024x1000": (1024, 1000, False), "1200x1210": (1200, 1210, True),
         "1500x1501": (1500, 1501, False), "1700x1711": (1700, 1711, True)}


@pytest.mark.parametrize("name", list(GRIDS))
def test_mixed_calls(name):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import Solver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny, walls = GRIDS[name]
    p, phi0 = (I.nonuniform if walls else I.burgers)(nx, ny)
    out = []
    for kernel, calls in (("fused", (31,)), ("auto", (1, 2, 3, 4, 5, 16)), ("auto", (11, 12, 8)), ("auto", (31,))):
        s = Solver(p, precision=32, kernel=kernel)
        s.init_phi(torch.tensor(phi0, device="cuda"))
        for n in calls:
            s.step(n)
        out.append(s.save_state())
        assert s.info()["steps_done"] == 31
        s.sync()
        s.close()
    assert all(torch.equal(out[0], f) for f in out[1:])
