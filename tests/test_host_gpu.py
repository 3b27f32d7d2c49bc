"""What the calls do on the host: threads, errors, failures that leave nothing behind."""
import threading
import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from test_parity_gpu import sh  # noqa: E402,F401


def test_other_threads_run_while_a_call_waits_for_the_launch_queue(sh):  # noqa: F811
    """A second of work ahead in the stream and more calls than the queue of launches holds: the thread that makes them
    waits, the others do not."""
    x, un, tree = torch.randn((1, 1, 64), device="cuda"), torch.rand((1, 1, 5), device="cuda"), sh.Tree.heap(1)
    sh.spechub_draft_sample(x, un, tree)
    torch.cuda.synchronize()
    took = []

    def calls():
        torch.cuda._sleep(2_000_000_000)   # (clocks: about a second)
        t0 = time.monotonic()
        for _ in range(3000):
            sh.spechub_draft_sample(x, un, tree)
        took.append(time.monotonic() - t0)

    thread, ticks = threading.Thread(target=calls), [time.monotonic()]
    thread.start()
    while thread.is_alive():
        time.sleep(0.002)
        ticks.append(time.monotonic())
    thread.join()
    torch.cuda.synchronize()
    gap = max(b - a for a, b in zip(ticks, ticks[1:]))
    assert took[0] > 0.5, took    # (the calls did wait)
    assert gap < 0.25, (gap, took)
