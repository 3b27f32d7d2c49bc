"""Draft statistics of rows that are not whole words (off a 16-byte boundary, or with a remainder), from 16384 ids: records
are written and used, both steps against the oracle; a record that is not the row's leaves the plain call's results, also
where the logit at its argmax is the recorded maximum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from test_parity_gpu import METHODS, gpu_draft_stats, gpu_verify, gpu_verify_stats, padded, random_logits, random_uniforms, sh  # noqa: E402,F401
from test_streaming_gpu import batch_that_streams, check_two_drafts, sample  # noqa: E402

SHAPES = [(16385, "bf16", 0), (16391, "bf16", 64), (16387, "fp32", 0), (16388, "fp32", 8), (33001, "bf16", 0)]


def problem(V, dtype, N=7):
    rng = np.random.default_rng(V)
    B = batch_that_streams(N, V, dtype)
    lp, lq = random_logits(rng, B, N, V, dtype)
    lq[0, 0] = lp[0, 0]                                   # Z_p = Z_q exactly
    lq[0, 1, 16:] = -np.inf
    lq[1, 0, V - 1] = lq[1, 0].max() + 3.0                # the hub in the remainder
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    return rng, B, lp, lq, random_uniforms(rng, B, N)


@pytest.mark.parametrize("V,dtype,pad", SHAPES)
def test_records_are_used(sh, V, dtype, pad):  # noqa: F811
    rng, B, lp, lq, un = problem(V, dtype)
    tq, tree = padded(lq, dtype, pad), sh.Tree.heap(lp.shape[1])
    d = gpu_draft_stats(sh, "spechub", tq, torch.from_numpy(un).cuda(), tree, 0.8)
    assert bool((d["stats"].view(-1, 4)[:, 3] != 0).all())
    for leaves in (False, True):
        check_two_drafts(sh, lp, lq, dtype, pad, 0.8, un, leaves, sample(rng, B, 3, 5), "records", stats=True)
    # a record whose sum is another one is believed: the reported rates are others
    wrong = d["stats"].clone()
    words = wrong.view(-1, 4)
    words[:, 1] = (words[:, 1].contiguous().view(torch.float32) * 1.5).view(wrong.dtype)
    a, und = (padded(lp, dtype, pad), tq), torch.from_numpy(un).cuda()
    plain = gpu_verify(sh, "spechub", *a, d["tokens"], und, tree, 0.8)
    out = gpu_verify_stats(sh, "spechub", *a, wrong, d["tokens"], und, tree, 0.8)
    assert bool(((out["rate"] - plain["rate"]).abs().amax(-1)[2:] > 1e-3).all())


@pytest.mark.parametrize("V,dtype,pad", SHAPES)
def test_foreign_records_leave_the_plain_results(sh, V, dtype, pad):  # noqa: F811
    rng, B, lp, lq, un = problem(V, dtype)
    tp, tq, und, tree = padded(lp, dtype, pad), padded(lq, dtype, pad), torch.from_numpy(un).cuda(), sh.Tree.heap(lp.shape[1])
    for rows in (B, 2):   # streamed, and held in registers
        for m in METHODS:
            a = (tp[:rows], tq[:rows])
            d = gpu_draft_stats(sh, m, a[1], und[:rows], tree, 0.8)
            plain = gpu_verify(sh, m, *a, d["tokens"], und[:rows], tree, 0.8)
            for stats in (torch.zeros_like(d["stats"]), gpu_draft_stats(sh, m, a[1], und[:rows], tree, 0.5)["stats"]):
                out = gpu_verify_stats(sh, m, *a, stats, d["tokens"], und[:rows], tree, 0.8)
                check_plain(m, out, plain, rows)


def check_plain(m, out, plain, rows):
    for key in plain:
        if m == "rrsw" and key in ("beta", "rate"):
            # 1 - q(x1) is Z_q less one term here, a sum of its own there: at most 2^-22 of it apart, and
            # the acceptance ratio and the differences of sums of O(1) with it
            torch.testing.assert_close(out[key], plain[key], rtol=2e-6, atol=2e-6)
        else:
            assert torch.equal(plain[key], out[key]), (m, key, rows)


@pytest.mark.parametrize("V,dtype,pad", SHAPES)
def test_records_of_an_earlier_iteration_leave_the_plain_results(sh, V, dtype, pad):  # noqa: F811
    """The rows' logits are others since the draft step, except at the recorded argmax; or were not finite then."""
    rng, B, lp, lq, un = problem(V, dtype)
    now = workloads.round_to_storage(random_logits(rng, B, lp.shape[1], V, dtype)[1], dtype)
    top = lq.argmax(-1)[..., None]
    np.put_along_axis(now, top, np.take_along_axis(lq, top, -1), -1)
    then = lq.copy()
    then[0, 2, 5], then[1, 1, :], then[1, 2, 7] = np.nan, -np.inf, np.inf
    tp, tq, tthen, und = padded(lp, dtype, pad), padded(now, dtype, pad), padded(then, dtype, pad), torch.from_numpy(un).cuda()
    tree = sh.Tree.heap(lp.shape[1])
    for rows in (B, 2):
        for m in METHODS:
            d = gpu_draft_stats(sh, m, tq[:rows], und[:rows], tree, 0.8)
            a = (tp[:rows], tq[:rows])
            plain = gpu_verify(sh, m, *a, d["tokens"], und[:rows], tree, 0.8)
            assert int((plain["status"] & 1).sum()) == 0
            for old in (tthen, padded(lq, dtype, pad)):
                stats = gpu_draft_stats(sh, m, old[:rows], und[:rows], tree, 0.8)["stats"]
                check_plain(m, gpu_verify_stats(sh, m, *a, stats, d["tokens"], und[:rows], tree, 0.8), plain, rows)
