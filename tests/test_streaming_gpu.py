"""Streaming kernels, on calls with more rows than the kernels that hold rows in registers take: rows that are hard on
their sums and draws, in all row formats, with and without leaf rows, two and more drafts, against the oracle on a
sample of the rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import parity  # noqa: E402
import workloads  # noqa: E402
from test_parity_gpu import (METHODS, gpu_draft, gpu_draft_stats, gpu_verify, gpu_verify_stats, padded, random_logits,  # noqa: E402,F401
                             random_uniforms, sh)

# (V, dtype, ids between row starts are a multiple of pad): whole words and rows of any alignment, both types
FORMATS = [(8192, "bf16", 0), (9001, "bf16", 0), (8192, "fp32", 0), (8201, "fp32", 0)]


def batch_that_streams(nodes, V, dtype):
    """Sequences whose rows are certain to be streamed: a warp holds at most 2048 bf16 or 1024 fp32 ids in registers,
    rows of one or two warps are always held so, and no more than 25 warps per SM are."""
    warps = -(-V // (2048 if dtype == "bf16" else 1024))
    assert warps > 2
    return 25 * 148 // (warps * nodes) + 2


def sample(rng, B, first=8, n=12):
    return np.unique(np.concatenate([np.arange(first), [B - 1], rng.integers(0, B, n)]))


def check_two_drafts(sh, lp, lq, dtype, pad, T, un, leaves, pick, label, stats=False):  # noqa: F811
    """Both steps on all rows, the sequences `pick` against the oracle."""
    N = lp.shape[1]
    tp, tq, und = padded(lp, dtype, pad), padded(lq, dtype, pad), torch.from_numpy(un).cuda()
    tree, kind = sh.Tree.heap(N, leaves_sample=leaves), workloads.paper_node_kind(N) if leaves else None
    for m in METHODS:
        d = (gpu_draft_stats if stats else gpu_draft)(sh, m, tq, und, tree, T)
        if stats:
            out = gpu_verify_stats(sh, m, tp, tq, d["stats"], d["tokens"], und, tree, T)
        else:
            out = gpu_verify(sh, m, tp, tq, d["tokens"], und, tree, T)
        d, out = parity.to_numpy(d), parity.to_numpy(out)
        parity.check_draft(m, lq[pick], T, un[pick], {k: v[pick] for k, v in d.items() if k != "stats"}, label=label)
        parity.check_verify(m, lp[pick], lq[pick], T, d["tokens"][pick], un[pick], kind,
                            {k: v[pick] for k, v in out.items()}, label=label)


def check_more_drafts(sh, k, wo, lp, lq, dtype, pad, T, un, leaves, pick, label):  # noqa: F811
    """RRS / RRSw with k drafts per node, complete k-ary tree of two levels (as test_kary_gpu.check, on a sample)."""
    N = lp.shape[1]
    tree = sh.Tree.kary(k, 2, leaves_sample=leaves)
    kind = np.array([0] + [1] * k, np.uint8) if leaves else None
    tp, tq, und = padded(lp, dtype, pad), padded(lq, dtype, pad), torch.from_numpy(un).cuda()
    d = sh.rrs_draft_sample(tq, und, tree, wo, T)
    out = parity.to_numpy(sh.rrs_verify_tree(tp, tq, d["tokens"], und, tree, wo, T))
    d = {key: v[pick] for key, v in parity.to_numpy(d).items()}
    out = {key: v[pick] for key, v in out.items()}
    lp, lq, un = lp[pick], lq[pick], un[pick]
    od = oracle.rrs_k_draft_batch(k, wo, lq, T, un)
    ov = oracle.rrs_k_verify_batch(k, wo, lp, lq, T, d["tokens"], un, kind)
    for b in range(len(pick)):
        for n in range(N):
            ctx = "%s k=%d wo=%s b=%d n=%d V=%d" % (label, k, wo, pick[b], n, lp.shape[2])
            if tuple(d["tokens"][b, n]) == tuple(od["tokens"][b, n]):
                assert d["status"][b, n] == od["status"][b, n], ctx
            else:   # every draw admissible given the earlier ones
                w, _ = oracle.softmax(lq[b, n], T)
                for i, x in enumerate(d["tokens"][b, n]):
                    lo, hi = oracle.cdf_interval(w, int(x))
                    assert lo - parity.NEAR <= un[b, n, i] <= hi + parity.NEAR, ("draft", ctx, i)
                    if wo:
                        w[x] = 0.0
            token, o_token = int(out["token"][b, n]), int(ov["token"][b, n])
            if kind is not None and kind[n] == 1:
                if token != o_token:
                    lo, hi = oracle.cdf_interval(oracle.softmax(lp[b, n], T)[0], token)
                    assert lo - parity.NEAR <= un[b, n, 2 * k] <= hi + parity.NEAR, ctx
                assert out["status"][b, n] == 0, ctx
                continue
            eps = parity.row_eps(lp[b, n], lq[b, n], T)   # (and the tolerances of parity.check_verify)
            for key, cond in (("beta", ov["cond"][b, n]), ("rate", 1.0)):
                g, o = out[key][b, n], ov[key][b, n]
                assert np.all(np.abs(g - o) <= parity.RTOL * np.abs(o) + parity.FLOOR + eps * cond), (key, ctx, g, o)
            if token == o_token and out["accept_idx"][b, n] == ov["accept_idx"][b, n]:
                assert out["status"][b, n] | 16 == ov["status"][b, n] | 16, ctx
                continue
            bands = [max(parity.NEAR, eps * c) for c in ov["cond"][b, n]] + [parity.NEAR]
            assert any(m <= bd for m, bd in zip(ov["margin"][b, n], bands)), (ctx, token, o_token, ov["margin"][b, n])


def mask_starts(x, V):
    """-inf on the first 300 ids of every 128 vectors and more: whatever CTA shape, some warps' ranges begin with
    ids that are all masked."""
    for s in range(0, V, max(1024, V // 64 // 8 * 8)):
        x[..., s:s + 300] = -np.inf


@pytest.mark.parametrize("leaves", [False, True])
@pytest.mark.parametrize("V,dtype,pad", FORMATS + [(32000, "bf16", 0)])
def test_rows_that_begin_with_masked_ids_and_lie_low(sh, V, dtype, pad, leaves):  # noqa: F811
    """The first ids of warps' ranges are masked and the others lie far below 0: exponentials on the scale of 0 would
    all be 0."""
    rng = np.random.default_rng(V + leaves)
    B = batch_that_streams(3, V, dtype)
    lp, lq = random_logits(rng, B, 3, V, dtype)
    shift = np.float32([-200.0, -85.0])[np.arange(B) % 2][:, None, None]
    lp, lq = lp + shift, lq + shift
    mask_starts(lp, V)
    mask_starts(lq, V)
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    check_two_drafts(sh, lp, lq, dtype, pad, 1.0, random_uniforms(rng, B, 3), leaves, sample(rng, B), "masked")
    B = batch_that_streams(4, V, dtype)
    lp, lq = np.resize(lp, (B, 4, V)), np.resize(lq, (B, 4, V))
    un = rng.integers(0, 1 << 24, (B, 4, 7)).astype(np.float32) * np.float32(2.0 ** -24)
    for wo in (False, True):
        check_more_drafts(sh, 3, wo, lp, lq, dtype, pad, 1.0, un, leaves, sample(rng, B), "masked")


@pytest.mark.parametrize("V,dtype,rows,calls,most", [(128256, "fp32", 1024, 8, 0.0022), (50257, "bf16", 2048, 8, 0.0006)])
def test_draws_take_the_ids_that_fp64_takes(sh, V, dtype, rows, calls, most):  # noqa: F811
    """Draws by the prefix sums of whole rows: an id of the flat tail weighs 1e-6 of its row, a few fp32 roundings of the
    row's mass.  What is left are the roundings of the masses themselves (0.0016 and 0.0003 of the draws; with prefixes
    and targets in fp32 too, 0.0030 and 0.0012): the limits lie between the two."""
    leaf = sh.Tree.heap(1)
    leaf.node_kind = torch.ones(1, dtype=torch.uint8, device="cuda")
    off = n = 0
    for call in range(calls):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(1000 + call * rows)
        prior = -1.2 * torch.log1p(torch.randperm(V, generator=gen, device="cuda").float())
        logits = torch.randn((rows, V), generator=gen, device="cuda") + prior
        logits = logits.to(torch.bfloat16 if dtype == "bf16" else torch.float32)
        un = torch.randint(0, 1 << 24, (rows, 1, 5), generator=gen, device="cuda").float() * 2.0 ** -24
        cdf = logits.double().softmax(1).cumsum(1)
        x = logits[:, None, :]
        drafts = sh.rrs_draft_sample(x, un, sh.Tree.heap(1), False)["tokens"][:, 0]
        bonus = sh.rrs_verify_tree(x, x, drafts[:, None].contiguous(), un, leaf, False)["token"][:, 0]
        for u, got in ((0, drafts[:, 0]), (1, drafts[:, 1]), (4, bonus)):
            want = torch.searchsorted(cdf, un[:, 0, u:u + 1].double() * cdf[:, -1:], right=True)[:, 0].clamp(max=V - 1)
            off += int((got != want).sum())
            n += rows
    assert off <= most * n, (off, n)


@pytest.mark.parametrize("V,dtype", [(8192, "bf16"), (9001, "bf16"), (8192, "fp32")])
def test_verification_with_leaf_rows_reads_what_the_kernel_before_it_wrote(sh, V, dtype):  # noqa: F811
    """Logits, drafts and uniforms overwritten by kernels of the same stream right before the call, in buffers that the
    call before it read: every call sees the new values."""
    rng = np.random.default_rng(V)
    B, tree = batch_that_streams(3, V, dtype), sh.Tree.heap(3, leaves_sample=True)
    sets = []
    for _ in range(3):
        lp, lq = random_logits(rng, B, 3, V, dtype)
        tp, tq, un = padded(lp, dtype, 0), padded(lq, dtype, 0), torch.from_numpy(random_uniforms(rng, B, 3)).cuda()
        sets.append((tp, tq, un))
    for m in METHODS:
        drafts = [gpu_draft(sh, m, tq, un, tree, 1.0)["tokens"] for _, tq, un in sets]
        want = [parity.to_numpy(gpu_verify(sh, m, tp, tq, d, un, tree, 1.0)) for (tp, tq, un), d in zip(sets, drafts)]
        tp, tq, un, d = *(t.clone() for t in sets[0]), drafts[0].clone()
        got = []
        for i in range(9):
            for buf, new in zip((tq, un, d, tp), (sets[i % 3][1], sets[i % 3][2], drafts[i % 3], sets[i % 3][0])):
                buf.copy_(new)
            got.append(gpu_verify(sh, m, tp, tq, d, un, tree, 1.0))
        for i, out in enumerate(got):
            for key, v in parity.to_numpy(out).items():
                np.testing.assert_array_equal(v.view(np.int32), want[i % 3][key].view(np.int32), err_msg="%s %s" % (m, key))


@pytest.mark.parametrize("B", [2, 600])
@pytest.mark.parametrize("V,dtype", [(8192, "bf16"), (8201, "fp32")])
def test_second_drafts_from_next_to_nothing(sh, V, dtype, B):  # noqa: F811
    """Nearly all mass on one id and 2^-120 of it on three others: they are what is left to draw from."""
    rng = np.random.default_rng(V + B)
    lq = np.full((B, 3, V), -np.inf, np.float32)
    lq[:, :, 6000] = 4.0
    lq[:, :, [100, 3000, 8000]] = 4.0 - 83.2
    lq = workloads.round_to_storage(lq, dtype)
    un, pick = random_uniforms(rng, B, 3), sample(rng, B, first=2)
    tq, und = padded(lq, dtype, 0), torch.from_numpy(un).cuda()
    for m in METHODS:
        d = parity.to_numpy(gpu_draft(sh, m, tq, und, sh.Tree.heap(3), 1.0))
        parity.check_draft(m, lq[pick], 1.0, un[pick], {k: v[pick] for k, v in d.items()}, label="next to nothing")
        assert int(d["status"].max()) == 0, m


def test_draws_from_rows_with_ids_of_no_normal_exponential(sh):  # noqa: F811
    """Uniforms of 0 on rows whose first ids lie just below 2^-126 of the top: together they have mass, each alone has
    none in fp32.  Draws go to an id that has some, and no row is flagged."""
    rng = np.random.default_rng(77)
    for V, dtype, B in ((8192, "bf16", batch_that_streams(3, 8192, "bf16")), (9001, "fp32", batch_that_streams(3, 9001, "fp32")),
                        (8192, "bf16", 4), (9001, "fp32", 4)):
        lp, lq = random_logits(rng, B, 3, V, dtype)
        for x in (lp, lq):
            x[...] = np.minimum(x, 7.0)
            x[:, :, :4096] = -80.0     # log2(e) * -80 = -115.4; the reference of the row is 11 = rint(log2(e) * 7.5)
            x[:, :, 5000] = 7.5        # the maximum
        lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
        un = random_uniforms(rng, B, 3)
        un[:, :, [0, 1, 4]] = 0.0
        for leaves in (False, True):
            check_two_drafts(sh, lp, lq, dtype, 0, 1.0, un, leaves, sample(rng, B, first=min(B, 8)), "below normal")
        tq, und = padded(lq, dtype, 0), torch.from_numpy(un).cuda()
        all3 = sh.mdsd_compare_draft_sample(tq, und, sh.Tree.heap(3), 1.0)
        assert all(int(all3[m]["tokens"].min()) >= 0 and int(all3[m]["status"].max()) == 0 for m in METHODS)
        un = np.zeros((B, 4, 7), np.float32)
        un[:, :, 3:6] = 0.5
        lp, lq = np.resize(lp, (B, 4, V)), np.resize(lq, (B, 4, V))
        for wo in (False, True):
            for leaves in (False, True):
                check_more_drafts(sh, 3, wo, lp, lq, dtype, 0, 1.0, un, leaves, sample(rng, B, first=min(B, 8)), "below normal")


def hard_rows(lp, lq):
    """The first eight sequences' rows become what is hard on sums, references and draws."""
    V = lp.shape[2]
    lq[0, 0] = lp[0, 0]                                                  # p = q
    lq[0, 1] = -np.inf; lq[0, 1, V - 1] = 0.0                            # one-hot q at the last id
    lq[0, 2] = -60.0; lq[0, 2, V // 2] = 0.0                             # nearly
    lp[1, 0, :V // 2] = -np.inf; lq[1, 0, V // 2:] = -np.inf             # disjoint
    lp[1, 1] = np.round(lp[1, 1] * 2) / 2; lq[1, 1] = np.round(lq[1, 1] * 2) / 2   # ties
    lq[1, 2] = 0.0                                                       # uniform: the hub is id 0
    lp[2, 0, 3] = np.nan                                                 # flagged rows
    lq[2, 1, 9] = np.inf
    lq[2, 2] = -np.inf
    lp[3, 0, :V // 2] -= 300.0; lq[3, 0, :V // 2] -= 300.0               # sums leave the range of their first reference
    lq[3, 1, ::2] -= 250.0
    lp[3, 2, :V // 3] = -np.inf; lp[3, 2, V // 3:V // 2] -= 400.0
    lq[4, 0, :100] += 300.0
    lq[4, 1, V - 50:] += 280.0; lp[4, 1, V - 50:] += 280.0
    lq[4, 2, 1000:1010] += 200.0
    lq[5, 0, 7] = lq[5, 0].max() + 9.0                                   # peaked
    lq[5, 1, V - 1] = lq[5, 1].max() + 6.0                               # the hub is the last id


# many rows, and rows for CTAs of 512 and of 256 threads
SHAPES = [f + (None,) for f in FORMATS] + [(32000, "bf16", 0, 240), (32000, "bf16", 0, 450), (32003, "bf16", 0, 240), (32003, "bf16", 0, 450),
                                           (16384, "fp32", 0, 240), (16384, "fp32", 0, 450), (16387, "fp32", 0, 240),
                                           (16387, "fp32", 0, 450), (8201, "fp32", 64, None)]


@pytest.mark.parametrize("leaves", [False, True])
@pytest.mark.parametrize("V,dtype,pad,rows", SHAPES)
def test_hard_rows_two_drafts(sh, V, dtype, pad, rows, leaves):  # noqa: F811
    rng = np.random.default_rng(V + leaves)
    B = rows // 3 if rows else batch_that_streams(3, V, dtype)
    assert B >= batch_that_streams(3, V, dtype) - 1
    lp, lq = random_logits(rng, B, 3, V, dtype)
    hard_rows(lp, lq)
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    un, pick = random_uniforms(rng, B, 3), sample(rng, B, n=6)
    for stats in (False, True):
        check_two_drafts(sh, lp, lq, dtype, pad, 1.0, un, leaves, pick, "hard", stats=stats)


@pytest.mark.parametrize("k", [3, 4])
@pytest.mark.parametrize("V,dtype,pad,rows", SHAPES)
def test_hard_rows_more_drafts(sh, V, dtype, pad, rows, k):  # noqa: F811
    rng = np.random.default_rng(V + k)
    N = k + 1
    B = -(-rows // N) if rows else batch_that_streams(N, V, dtype)
    lp, lq = random_logits(rng, B, N, V, dtype)
    hard_rows(lp, lq)
    lp, lq = workloads.round_to_storage(lp, dtype), workloads.round_to_storage(lq, dtype)
    un = rng.integers(0, 1 << 24, (B, N, 2 * k + 1)).astype(np.float32) * np.float32(2.0 ** -24)
    for wo in (False, True):
        for leaves in (False, True):
            check_more_drafts(sh, k, wo, lp, lq, dtype, pad, 1.0, un, leaves, sample(rng, B, n=6), "hard")


@pytest.mark.parametrize("k", [3, 4])
@pytest.mark.parametrize("V", [8192, 32000, 131080])
def test_hard_rows_more_drafts_resident(sh, V, k):  # noqa: F811
    """The exponentials kept on chip (asked for), one CTA per row and clusters."""
    rng = np.random.default_rng(V + k)
    B, N = 8, k + 1
    lp, lq = random_logits(rng, B, N, V, "bf16")
    hard_rows(lp, lq)
    lp, lq = workloads.round_to_storage(lp, "bf16"), workloads.round_to_storage(lq, "bf16")
    un = rng.integers(0, 1 << 24, (B, N, 2 * k + 1)).astype(np.float32) * np.float32(2.0 ** -24)
    sh.set_row_split(8)
    try:
        for wo in (False, True):
            for leaves in (False, True):
                check_more_drafts(sh, k, wo, lp, lq, "bf16", 0, 1.0, un, leaves, np.arange(B), "resident")
    finally:
        sh.set_row_split(0)


@pytest.mark.parametrize("V,dtype,B", [(8192, "bf16", 310), (8192, "fp32", 160)])
def test_streamed_records_of_other_logits_or_another_temperature_are_refused(sh, V, dtype, B):  # noqa: F811
    """Both steps stream their rows; verification checks the records as test_draft_stats_gpu has it on few rows."""
    rng = np.random.default_rng(V)
    assert B >= batch_that_streams(3, V, dtype) - 1
    tree, tq = sh.Tree.heap(3), []
    for _ in range(2):
        lp, lq = random_logits(rng, B, 3, V, dtype)
        tq.append(padded(lq, dtype, 0))
    tp, un = padded(lp, dtype, 0), torch.from_numpy(random_uniforms(rng, B, 3)).cuda()
    for m in METHODS:
        d = gpu_draft_stats(sh, m, tq[0], un, tree, 1.0)
        for stats in (gpu_draft_stats(sh, m, tq[1], un, tree, 1.0)["stats"], gpu_draft_stats(sh, m, tq[0], un, tree, 0.7)["stats"],
                      torch.zeros_like(d["stats"])):
            out = gpu_verify_stats(sh, m, tp, tq[0], stats, d["tokens"], un, tree, 1.0)
            assert bool(((out["status"] & 64) != 0).all()) and bool((out["token"] == -1).all()), m
        out = gpu_verify_stats(sh, m, tp, tq[0], d["stats"], d["tokens"], un, tree, 1.0)
        assert int((out["status"] & 64).max()) == 0, m
