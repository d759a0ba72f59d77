"""A finished request is reported at once: its completion record is never left
unread until the dispatcher's idle sleep of 20 ms runs out."""

import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1806_06698_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def syev3():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06698_gb300 import build, syev3 as mod

    build.build()
    return mod


@pytest.mark.parametrize("sizes", [(7,), (5, 31, 177, 1000)])
def test_no_burst_waits_for_the_idle_sleep(syev3, sizes):
    """20000 bursts of a few hundred microseconds each.  A completion left unread
    makes a burst take the sleep and little more; other delays of that length
    are the machine's, and one is allowed."""
    pool = [torch.from_numpy(inputs.gaussian(n, seed=2500 + n)).cuda() for n in sizes]
    srv = syev3.Server(memory_budget_bytes=64 << 20)
    slept = 0
    for _ in range(20000):
        t0 = time.perf_counter()
        tickets = [srv.submit(A) for A in pool]
        for t in tickets:
            srv.wait(t)
        slept += 0.0195 < time.perf_counter() - t0 < 0.0215
        for t in tickets:
            srv.release(t)
    srv.close()
    assert slept <= 1, f"{slept} of 20000 bursts waited for the dispatcher's sleep to end"
