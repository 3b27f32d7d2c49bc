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


def test_a_refused_launch_leaves_no_error_for_later_calls(sh):  # noqa: F811
    """More CTAs than a grid may have (2^29 + 1 rows on four each) is refused by the host; the next call, whose launches
    are checked by the last error, is not told of it."""
    import ctypes

    from paper_2411_05289_b200 import binding

    lib, x = sh.load_library(), torch.randn((2, 3, 64), device="cuda")
    un, tree, word = torch.rand((2, 3, 5), device="cuda"), sh.Tree.heap(3), torch.zeros(64, device="cuda")
    d, _ = binding._desc(x, tree, 1.0)
    d.batch, d.nodes, d.vocab, d.levels, d.dtype, d.flags = (1 << 29) + 1, 1, 8192, 1, binding.BF16, 4
    d.stride_seq = d.stride_node = 8192
    at = ctypes.c_void_p(word.data_ptr())   # (no kernel runs: nothing is read)
    assert lib.spechub_draft_sample(ctypes.byref(d), at, at, at, None, None, None, None) == -8
    tokens = sh.spechub_draft_sample(x, un, tree)["tokens"]
    sh.spechub_verify_tree_static(x, x, tokens, un, tree)
    torch.cuda.synchronize()


def test_out_of_memory_is_torch_s_own_error(sh):  # noqa: F811
    x, un, tree = torch.zeros((1 << 21, 1, 2), device="cuda"), torch.zeros((1 << 21, 1, 5), device="cuda"), sh.Tree.heap(1)
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction(1e-5)   # no new segment is given out
    try:
        with pytest.raises(torch.cuda.OutOfMemoryError):
            sh.spechub_draft_sample(x, un, tree)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert sh.spechub_draft_sample(x, un, tree)["tokens"].shape == (1 << 21, 1, 2)


def test_temperature_is_whatever_float_takes(sh):  # noqa: F811
    x, un, tree = torch.randn((4, 1, 64), device="cuda"), torch.rand((4, 1, 5), device="cuda"), sh.Tree.heap(1)
    want = sh.spechub_draft_sample(x, un, tree, 0.5)
    for t in ("0.5", b"0.5"):
        got = sh.spechub_draft_sample(x, un, tree, t)
        assert all(torch.equal(want[k], got[k]) for k in want)
