"""The row-marching step, a launch per step: kernel "fused" selects it on every
grid, so that it stays tested at the sizes where AUTO takes many steps per
launch.  Against the oracle and, in FP32, bit for bit against AUTO; and AUTO on
the parity cases against the oracle.  Tolerances as in the files the cases
come from."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import test_gpu_parity as parity  # noqa: E402
import test_gpu_sources as sources  # noqa: E402
from oracle import Oracle  # noqa: E402
from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _solver(p, prec, kernel):
    from paper_1906_11036_gb300.dugks import Solver

    s = Solver(p, precision=prec, kernel=kernel)
    if kernel == "fused":
        assert s.info()["block_threads"] == 32  # one warp per (strip, row segment)
    return s


def _run(p, phi0, prec, kernel, chunks):
    s = _solver(p, prec, kernel)
    s.init_phi(torch.tensor(phi0, device="cuda"))
    for n in chunks:
        s.step(n)
    f = s.save_state()
    s.sync()
    s.close()
    return f


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("name", list(sources.CASES))
def test_sources(name, prec):
    p, phi0 = sources.CASES[name]()
    o = Oracle(p)
    ref = o.phi(o.run(o.init(phi0), 30))
    f = _run(p, phi0, prec, "fused", [13, 17])
    assert _rel(f.double().sum(0).cpu().numpy(), ref) <= (1e-12 if prec == 64 else 2e-5)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("name", list(parity.CASES))
def test_auto_on_the_parity_cases(name, prec):
    p, phi0 = parity.CASES[name]()
    o = Oracle(p)
    ref = o.run(o.init(phi0), p.steps, 8)
    assert _rel(_run(p, phi0, prec, "auto", [p.steps]).double().cpu().numpy(), ref) <= parity.TOL[prec] * 5


@pytest.mark.parametrize("name", ["burgers_70x45", "mixed_xwall_33x17", "strips_330x70", "tall_9x300", "large"])
def test_fp32_equals_auto(name):
    p, phi0 = I.nonuniform(900, 700) if name == "large" else parity.CASES[name]()
    assert torch.equal(_run(p, phi0, 32, "fused", [9]), _run(p, phi0, 32, "auto", [1, 4, 4]))


@pytest.mark.parametrize("every", [1, 2, 3, 5, 13])  # without and with scratch states, an uneven last segment
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("walls", [False, True])
def test_gradient(walls, prec, every):
    """Both ways the gradient advances its states: row-marching steps and resident launches.  FP32: the same
    bits; FP64: 1e-11, the order of the operations."""
    p, phi0 = (I.nonuniform if walls else I.burgers)(48, 40)
    xc, yc = p.centres()
    g = torch.tensor(I.smooth_phi0(xc, yc, seed=9) - 1.0, device="cuda")
    x = torch.tensor(phi0, device="cuda")
    out = []
    for kernel in ("fused", "auto"):
        s = _solver(p, prec, kernel)
        out.append(s.gradient(x, 13, g, checkpoint_every=every, with_u=True))
        s.close()
    (g1, a1, u1), (g2, a2, u2) = out
    if prec == 32:
        assert torch.equal(g1, g2) and a1 == a2 and u1 == u2
    else:
        assert float((g1 - g2).norm() / g2.norm()) <= 1e-11 and abs(a1 - a2) <= 1e-11 * abs(a2)
        assert np.abs(np.subtract(u1, u2)).max() <= 1e-11 * np.abs(u2).max()


def test_info_gives_the_grid_that_runs():
    """grid_blocks: 30-column strips times the row segments of the kernel that steps (the tile sequence's with
    AUTO on a large FP32 grid, the row march's own with "fused")."""
    p, _ = I.burgers(900, 700)
    a, f = (_solver(p, 32, k) for k in ("auto", "fused"))
    na, nf = a.info()["grid_blocks"], f.info()["grid_blocks"]
    a.close()
    f.close()
    assert na % 30 == 0 and nf % 30 == 0 and na > nf
