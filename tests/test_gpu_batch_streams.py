"""The batch runs on a stream of its own and hands its results to the caller's.
Neither may overtake the other: memory that queued work of the caller still
reads is not written yet, and what the caller queues on a result runs after it
has been written."""
import pytest

torch = pytest.importorskip("torch")

from paper_1906_11036_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["get_phi", "save_state"])
def test_results_are_ordered_with_the_callers_stream(what):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1906_11036_gb300.dugks import BatchSolver

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p, phi0 = I.burgers(256)
    b = BatchSolver([p])
    b.init_phi(0, phi0)
    b.step(3)
    get = {"get_phi": lambda: b.get_phi(0), "save_state": lambda: b.save_state(0)}[what]
    like = get()
    b.sync()
    # a result that a copy queued behind a long kernel still reads, dropped by the caller
    old = get()
    torch.cuda._sleep(200_000_000)
    seen = old.clone()
    del old
    b.step(1)
    got = [get() for _ in range(3)]
    torch.cuda.synchronize()
    assert torch.equal(seen, like) and not torch.equal(got[0], like)
    assert all(torch.equal(got[0], x) for x in got)
    # memory of the caller's own in the same state
    old = torch.full_like(like, 7.0)
    torch.cuda._sleep(200_000_000)
    seen = old.clone()
    del old
    copy = get().clone()
    torch.cuda.synchronize()
    assert bool((seen == 7.0).all()) and torch.equal(copy, got[0])
    # a result that the batch has not computed yet when the caller reads it
    b.step(2000)
    copy = get().clone()
    b.sync()
    assert torch.equal(copy, get())
    b.close()
