"""Rows held in registers (calls whose rows do not fill the GPU, short vocabularies) and streamed rows of any
alignment: the edges of a lane's vectors, of a warp's and a cluster's part, aligned and packed odd rows, both types,
against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import parity  # noqa: E402
import workloads  # noqa: E402
from test_parity_gpu import (METHODS, gpu_draft, gpu_draft_stats, gpu_verify, gpu_verify_stats, padded, random_logits, random_uniforms,  # noqa: E402,F401
                             run_case, sh)


# one warp of 1 / 2 / 4 / 8 vectors per lane, two warps, a CTA, clusters of 2 / 4 / 8 CTAs, each with its neighbours
@pytest.mark.parametrize("pad", [0, 64])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [2, 255, 256, 257, 1025, 2048, 2049, 4097, 16385, 32769, 131071])
def test_edges_of_parts(sh, V, dtype, pad):  # noqa: F811
    rng = np.random.default_rng(V + 3)
    B, N = 2, 3
    lp, lq = random_logits(rng, B, N, V, dtype)
    lq[0, 1] = lp[0, 1]                                      # p = q
    lq[1, 2] = -np.inf; lq[1, 2, V - 1] = 0.0                # one-hot q at the last id
    lp[1, 0, V // 2:] = -np.inf                              # whole parts without mass
    lq[0, 2, V - 1] = lq[0, 2].max() + 6.0                   # the hub is the last id
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    un = random_uniforms(rng, B, N)
    for paper in (False, True):
        run_case(sh, lp, lq, dtype, np.array([1.0, 0.6], np.float32), un, paper, pad_to=pad, label="rowreg V=%d" % V)


@pytest.mark.parametrize("rows", [1, 3, 5, 1183, 2369])
def test_rows_per_cta_and_vectors_per_lane(sh, rows):  # noqa: F811
    """Row counts around a CTA's share of short rows and around one wave (fewer, wider warps from there on)."""
    rng = np.random.default_rng(rows)
    V = 384
    lp, lq = random_logits(rng, rows, 1, V, "fp32", sd=3.0)
    run_case(sh, lp, lq, "fp32", 1.0, random_uniforms(rng, rows, 1), False, label="rowreg rows=%d" % rows)


# streaming kernels on rows of any alignment: warps' ranges that begin and end inside, at and beyond the whole words
@pytest.mark.parametrize("pad", [0, 8, 64])
@pytest.mark.parametrize("V,dtype,B", [(1025, "fp32", 1200), (2049, "bf16", 500), (4105, "bf16", 600), (8199, "fp32", 300), (9001, "bf16", 300),
                                       (8201, "bf16", 790), (8192, "fp32", 790)])
def test_streamed_rows_of_any_alignment(sh, V, dtype, B, pad):  # noqa: F811
    rng = np.random.default_rng(V + pad)
    lp, lq = random_logits(rng, B, 3, V, dtype)
    lq[0, 1] = lp[0, 1]
    lq[1, 2] = -np.inf; lq[1, 2, V - 1] = 0.0
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    un = random_uniforms(rng, B, 3)
    pick = np.unique(np.concatenate([[0, 1, B - 1], rng.integers(0, B, 6)]))
    tp, tq = padded(lp, dtype, pad), padded(lq, dtype, pad)
    und, tree = torch.from_numpy(un).cuda(), sh.Tree.heap(3)
    for m in METHODS:
        d = parity.to_numpy(gpu_draft(sh, m, tq, und, tree, 1.0))
        parity.check_draft(m, lq[pick], 1.0, un[pick], {k: v[pick] for k, v in d.items()}, label="any")
        out = parity.to_numpy(gpu_verify(sh, m, tp, tq, torch.from_numpy(d["tokens"]).cuda(), und, tree, 1.0))
        parity.check_verify(m, lp[pick], lq[pick], 1.0, d["tokens"][pick], un[pick], None,
                            {k: v[pick] for k, v in out.items()}, label="any")


@pytest.mark.parametrize("V,dtype,B", [(8192, "bf16", 199), (8192, "fp32", 101), (128256, "bf16", 13)])
def test_records_of_streamed_draft_rows_read_by_registers(sh, V, dtype, B):  # noqa: F811
    """Between the two steps' limits: the draft step streams its rows and leaves records, the verification holds them
    in registers."""
    rng = np.random.default_rng(V + B)
    lp, lq = random_logits(rng, B, 3, V, dtype)
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    un = random_uniforms(rng, B, 3)
    pick = np.unique(np.concatenate([[0, B - 1], rng.integers(0, B, 6)]))
    tp, tq = padded(lp, dtype, 0), padded(lq, dtype, 0)
    und, tree = torch.from_numpy(un).cuda(), sh.Tree.heap(3)
    for m in METHODS:
        d = gpu_draft_stats(sh, m, tq, und, tree, 1.0)
        out = parity.to_numpy(gpu_verify_stats(sh, m, tp, tq, d["stats"], d["tokens"], und, tree, 1.0))
        d = parity.to_numpy(d)
        parity.check_draft(m, lq[pick], 1.0, un[pick], {k: v[pick] for k, v in d.items()}, label="records")
        parity.check_verify(m, lp[pick], lq[pick], 1.0, d["tokens"][pick], un[pick], None,
                            {k: v[pick] for k, v in out.items()}, label="records")


def test_three_methods_on_more_than_a_wave_of_rows(sh):  # noqa: F811
    """Draft step in CTAs of 64 threads: the three-method call gives the per-method calls' results bit for bit."""
    rng = np.random.default_rng(5)
    B, N, V = 793, 3, 8192
    lp, lq = random_logits(rng, B, N, V, "bf16")
    un = random_uniforms(rng, B, N)
    tq, und, tree = padded(workloads.round_to_storage(lq, "bf16"), "bf16", 0), torch.from_numpy(un).cuda(), sh.Tree.heap(N)
    out = sh.mdsd_compare_draft_sample_stats(tq, und, tree, 1.0)
    for m in METHODS:
        one = gpu_draft_stats(sh, m, tq, und, tree, 1.0)
        assert torch.equal(one["tokens"], out[m]["tokens"]), m
        assert torch.equal(one["stats"], out["stats"]), m
