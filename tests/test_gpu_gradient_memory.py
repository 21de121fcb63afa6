"""The gradient on a device that is nearly full: the kept states then lie
without the padding of their rows (a half of it on a grid of 33 columns), and
the results are the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,kernel", [(33, 40000, "auto"), (36, 36000, "fused"), (33, 40000, "naive")])
def test_states_without_padding(nx, ny, kernel):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import Solver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p, phi0 = I.burgers(nx, ny)
    x = torch.tensor(phi0, device="cuda").float()
    g = (x - 0.9) * 1e-3
    steps, every = 100, 10  # 18 kept states: 1.66 GB with padded rows, 0.86 GB without
    s = Solver(p, precision=32, kernel=kernel)
    ref = s.gradient(x, steps, g, checkpoint_every=every, with_u=True)
    s.close()
    s = Solver(p, precision=32, kernel=kernel)
    s.gradient(x, 1, g, checkpoint_every=1, with_u=True)  # its other buffers
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(max(0, free - 1_350_000_000), dtype=torch.uint8, device="cuda")
    left, _ = torch.cuda.mem_get_info()
    if not 1.1e9 < left < 1.6e9:
        pytest.skip(f"{left} bytes left: another process uses this GPU")
    got = s.gradient(x, steps, g, checkpoint_every=every, with_u=True)
    del fill
    torch.cuda.empty_cache()
    s.close()
    assert torch.equal(got[0], ref[0]) and got[1] == ref[1] and np.array_equal(got[2], ref[2])
