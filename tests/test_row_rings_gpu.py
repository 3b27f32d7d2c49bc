"""Draft step and leaf rows of one warp each, and those whose passes take their rows from rings of bulk copies (bf16 rows in whole words, CTAs of 64
and 128 threads): rows at which a warp's last chunk is full, one vector long or missing, against the oracle on a sample."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from test_parity_gpu import random_logits, random_uniforms, sh  # noqa: E402,F401
from test_streaming_gpu import check_more_drafts, check_two_drafts, sample  # noqa: E402

# ids a warp's chunk holds: 1024.  64 threads: below 8192 ids and, in many rows, below 40960; 128: more than 592 rows
SIZES = [(4104, 340), (6144, 340), (8192, 90), (8200, 90), (12296, 90), (16384 + 8, 90), (40960, 90), (16384, 340)]


@pytest.mark.parametrize("V,B", SIZES)
def test_two_drafts(sh, V, B):  # noqa: F811
    rng = np.random.default_rng(V)
    N = 7
    lp, lq = random_logits(rng, B, N, V, "bf16")
    lq[0, 0, : V // 2] = -np.inf                          # a warp without a finite logit
    lq[0, 1, :] = -np.inf
    lq[0, 1, V - 1] = 0.0                                 # the last id of the last chunk alone
    lq[1, 0, V - 64:] += 64.0                             # sums that leave the reference behind in the last batch
    lp, lq = workloads.round_to_storage(lp, "bf16"), workloads.round_to_storage(lq, "bf16")
    un = random_uniforms(rng, B, N)
    pick = sample(rng, B, 4, 6)
    for leaves in (False, True):
        check_two_drafts(sh, lp, lq, "bf16", 0, 0.8, un, leaves, pick, "rings")


# one warp per row: bf16 in whole words, below 10240 ids in more than 1184 rows; beside it rows that do not take it
@pytest.mark.parametrize("V,dtype,pad", [(2056, "bf16", 0), (2051, "bf16", 0), (4095, "bf16", 1), (10232, "bf16", 0), (10239, "bf16", 0),
                                         (4104, "fp32", 0), (5001, "fp32", 0)])
def test_rows_of_one_warp(sh, V, dtype, pad):  # noqa: F811
    rng = np.random.default_rng(V + 2)
    B, N = 172, 7
    lp, lq = random_logits(rng, B, N, V, dtype)
    lq[0, 0, : V // 2] = -np.inf
    lq[0, 1, :] = -np.inf
    lq[0, 1, V - 1] = 0.0
    lq[1, 0, V - 64:] += 64.0
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    pick = sample(rng, B, 4, 6)
    check_two_drafts(sh, lp, lq, dtype, pad, 0.8, random_uniforms(rng, B, N), True, pick, "one warp")
    lp, lq = lp[2:, :4], lq[2:, :4]
    lp, lq = np.concatenate([lp, lp[::-1]]), np.concatenate([lq, lq[::-1]])
    B = len(lp)
    un = rng.integers(0, 1 << 24, (B, 4, 7)).astype(np.float32) * np.float32(2.0 ** -24)
    check_more_drafts(sh, 3, True, lp, lq, dtype, pad, 1.0, un, True, sample(rng, B, 4, 6), "one warp")


@pytest.mark.parametrize("V,B", [(8200, 160), (32000, 160), (16384, 620)])
def test_three_drafts(sh, V, B):  # noqa: F811
    rng = np.random.default_rng(V + 1)
    N, k = 4, 3
    lp, lq = random_logits(rng, B, N, V, "bf16")
    un = rng.integers(0, 1 << 24, (B, N, 2 * k + 1)).astype(np.float32) * np.float32(2.0 ** -24)
    for wo in (False, True):
        check_more_drafts(sh, k, wo, lp, lq, "bf16", 0, 1.0, un, True, sample(rng, B, 4, 6), "rings")
