"""A dugks_set_source that finds no memory leaves the context without a source,
not with the buffers it has already given back: the steps that follow are the
plain step's, bit for bit."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [(32, 4096), (64, 2600)])
def test_a_source_that_does_not_fit(prec, n):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import Solver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p, _ = I.burgers(n)
    s = Solver(p, precision=prec)
    fields = torch.zeros(8, n, n, dtype=s.dtype, device="cuda")
    phi0 = torch.rand(n, n, dtype=s.dtype, device="cuda") + 0.5
    rate, power = (ctypes.c_double * 8)(), (ctypes.c_int * 8)(*range(8))

    def source(terms):
        return s.L.dugks_set_source(s.h, terms, rate, power, ctypes.c_void_p(fields.data_ptr()), 0.0)

    s.init_phi(phi0)
    s.step(2)
    ref = s.save_state()
    assert source(1) == 0
    s.step(1)
    s.sync()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(max(0, free - 250_000_000), dtype=torch.uint8, device="cuda")
    left, _ = torch.cuda.mem_get_info()
    if left > 350_000_000:
        pytest.skip(f"{left} bytes left: another process uses this GPU")
    status = source(8)  # eight fields take 0.4 ... 1.2 GB
    del fill
    torch.cuda.empty_cache()
    assert status == 6 and s.info()["nsrc"] == 0
    s.init_phi(phi0)
    s.step(2)
    got = s.save_state()
    s.sync()
    s.close()
    assert torch.equal(got, ref)
