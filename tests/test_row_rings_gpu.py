"""Draft step and leaf rows by the shape of their CTAs: one warp per row; passes that take their rows from rings of bulk
copies (draft step, bf16 rows in whole words of 40960 ids and more, more rows than one wave of CTAs of 128 threads); rows that
come with the next vectors in registers.  Rows at which a warp's last chunk or batch is full, one vector long or missing, and rows that are hard
on sums and references, against the oracle on a sample; the three-method draft step bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from test_compare_gpu import METHODS, bits, separate_draft  # noqa: E402
from test_parity_gpu import random_logits, random_uniforms, sh  # noqa: E402,F401
from test_streaming_gpu import check_more_drafts, check_two_drafts, hard_rows, sample  # noqa: E402

# A chunk of a ring, as a batch of vectors, is 1024 ids of a warp's range.  Seven rows per sequence: 340 sequences fill more than a wave of 64 threads (below
# 40960 ids; below 10240 ids only leaf rows take those, draft steps one warp), 170 more than one of 128, 90 less than that.
SIZES = [(4104, 340), (6144, 340), (10248, 340), (12288, 340), (12296, 340), (16384, 170), (16392, 170), (16416, 170), (40960, 170),
         (40968, 170), (40992, 170),
         (8192, 90), (8200, 90), (16392, 90), (40960, 90)]


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
        check_two_drafts(sh, lp, lq, "bf16", 0, 0.8, un, leaves, pick, "passes")


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


@pytest.mark.parametrize("V,B", [(8200, 160), (32000, 160), (16384, 620), (12296, 620), (16392, 310)])
def test_three_drafts(sh, V, B):  # noqa: F811
    rng = np.random.default_rng(V + 1)
    N, k = 4, 3
    lp, lq = random_logits(rng, B, N, V, "bf16")
    un = rng.integers(0, 1 << 24, (B, N, 2 * k + 1)).astype(np.float32) * np.float32(2.0 ** -24)
    for wo in (False, True):
        check_more_drafts(sh, k, wo, lp, lq, "bf16", 0, 1.0, un, True, sample(rng, B, 4, 6), "rings")


# shifted rows: more than a wave of 128 and of 64 threads, and less
@pytest.mark.parametrize("V,B,dtype", [(16393, 170, "bf16"), (12291, 340, "bf16"), (16393, 90, "bf16"), (16387, 170, "fp32")])
def test_shifted_rows(sh, V, B, dtype):  # noqa: F811
    rng = np.random.default_rng(V + B)
    lp, lq = random_logits(rng, B, 7, V, dtype)
    lq[0, 0, : V // 2] = -np.inf
    lq[1, 0, V - 64:] += 64.0
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    for leaves in (False, True):
        check_two_drafts(sh, lp, lq, dtype, 0, 0.8, random_uniforms(rng, B, 7), leaves, sample(rng, B, 4, 6), "shifted")


# (rows: three per sequence) one warp; 64 threads, leaf rows only and all; 128 threads, more than a wave and less
MANY = [(4104, 410), (9000, 410), (4104, 810), (12296, 810), (16392, 410), (16392, 230), (40968, 410)]


@pytest.mark.parametrize("V,B", MANY)
def test_hard_rows(sh, V, B):  # noqa: F811
    rng = np.random.default_rng(V + B)
    lp, lq = random_logits(rng, B, 3, V, "bf16")
    hard_rows(lp, lq)
    lp, lq = workloads.round_to_storage(lp, "bf16"), workloads.round_to_storage(lq, "bf16")
    un, pick = random_uniforms(rng, B, 3), sample(rng, B, n=6)
    for leaves in (False, True):
        check_two_drafts(sh, lp, lq, "bf16", 0, 1.0, un, leaves, pick, "hard", stats=True)


@pytest.mark.parametrize("V,B", MANY[1:] + [(40960, 800), (40992, 410), (32000, 130), (32000, 90)])
def test_three_methods(sh, V, B):  # noqa: F811
    rng = np.random.default_rng(V + B + 1)
    _, lq = random_logits(rng, B, 3, V, "bf16")
    hard_rows(lq.copy(), lq)
    tq, und = workloads.to_device(workloads.round_to_storage(lq, "bf16"), "bf16", "cuda"), torch.from_numpy(random_uniforms(rng, B, 3)).cuda()
    tree = sh.Tree.heap(3)
    out = sh.mdsd_compare_draft_sample(tq, und, tree, 0.8)
    for m in METHODS:
        one = separate_draft(sh, m, tq, und, tree, 0.8)
        for key in one:
            np.testing.assert_array_equal(bits(out[m][key]), bits(one[key]), err_msg="%s %s" % (m, key))
