"""What a decoding loop or a study has this library do, as cases that can be timed.

A decoding iteration of multi-draft speculative decoding has two steps on the same tree of nodes: the
draft step samples every node's drafts from the draft logits, verification tests them against the
target logits, draws residual and bonus tokens and walks the tree.  A case names

    call     "step"    both, the drafts of the first handed to the second
             "draft"   the draft step alone
             "verify"  verification alone, the drafts already in hand (drawn by somebody else's code)
    method   "spechub", "rrs", "rrsw", or "compare" (the three from shared reads of the logits)
    k, levels          complete k-ary tree: 2 drafts per node unless RRS / RRSw are asked for more
    batch, vocab       sequences; token ids per row
    pad                row starts are a multiple of this many ids apart (1: rows are packed)
    dtype              of the logits: "bf16", or "fp32" from a model whose head returns fp32
    leaves             the last level only draws the bonus token from p (no drafts below it)
    handover           the draft call leaves its per-row statistics for the verification call
    probabilities      verification also reports acceptance probabilities and rates; without, decisions only
    temperature        0 means: every sequence has its own, from 0.6 to 1.0
    sigma              noise between draft and target logits
    adversarial        share of rows that are p = q, one-hot, disjoint, near-uniform or full of ties
"""
import math

import torch

import paper_2411_05289_b200 as sh
from paper_2411_05289_b200.binding import alloc_verify_outputs

METHODS = ("spechub", "rrs", "rrsw")


def _case(name=None, call="step", method="spechub", batch=1, levels=3, k=2, vocab=32000, pad=1, dtype="bf16",
          leaves=False, handover=True, probabilities=False, temperature=1.0, sigma=1.0, adversarial=0.0):
    c = dict(call=call, method=method, batch=batch, levels=levels, k=k, vocab=vocab, pad=pad, dtype=dtype, leaves=leaves,
             handover=handover, probabilities=probabilities, temperature=temperature, sigma=sigma,
             adversarial=adversarial)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # one user at a terminal: 7 nodes of a 32000-id vocabulary, where latency is all that counts
        _case("one_sequence_step", "step", "spechub", 1, 3, vocab=32000, temperature=0.6, sigma=1.5),
        # one user, deep tree, 128256 ids; the drafts come from a draft model that samples by itself
        _case("one_sequence_verify_128k", "verify", "spechub", 1, 5, vocab=128256, handover=False, temperature=0.6),
        # a study on many small independent instances: 1000 trees of 3 nodes, V = 1000, fp32
        _case("small_vocab_step_fp32", "step", "spechub", 1000, 2, vocab=1000, dtype="fp32", handover=False),
        # an ordinary serving batch: 64 sequences of 7 nodes
        _case("batch64_step", "step", "spechub", 64, 3, vocab=32000, sigma=1.5),
        # a busy server with deeper trees whose leaves carry no drafts, sampling without replacement
        _case("batch256_leaves_rrsw_step", "step", "rrsw", 256, 4, vocab=32000, leaves=True, temperature=0.6, sigma=0.5),
        # the headline verification: 256 sequences of 31 nodes, 128256 ids, with all probabilities
        _case("batch256_verify_128k", "verify", "spechub", 256, 5, vocab=128256, probabilities=True),
        # its draft step
        _case("batch256_draft_128k", "draft", "spechub", 256, 5, vocab=128256),
        # the baseline method on a middling batch, drafts in hand, with probabilities (an ablation)
        _case("batch64_rrs_verify_128k", "verify", "rrs", 64, 5, vocab=128256, handover=False, probabilities=True),
        # a head that returns fp32 logits; requests of a server carry their own temperatures
        _case("fp32_step_128k", "step", "spechub", 32, 4, vocab=128256, dtype="fp32", temperature=0.0),
        # a vocabulary of an odd number of ids in packed rows: most rows start off a 16-byte boundary
        _case("odd_vocab_step", "step", "spechub", 64, 4, vocab=50257, leaves=True),
        # three drafts per node, ternary tree of 40 nodes, Algorithm 1 without replacement
        _case("three_drafts_rrsw_step", "step", "rrsw", 256, 4, 3, vocab=32000, handover=False, sigma=1.5),
        # the three methods side by side on the largest input, a tenth of its rows degenerate
        _case("compare_verify_152k", "verify", "compare", 1024, 5, vocab=152064, probabilities=True, adversarial=0.1),
    ]


def draw(rng):
    method = rng.choice(("spechub", "spechub", "spechub", "rrs", "rrsw", "compare"))
    k = rng.choice((3, 4)) if method in ("rrs", "rrsw") and rng.random() < 0.3 else 2
    levels = rng.randint(2, 5) if k == 2 else rng.randint(2, 4 if k == 3 else 3)
    nodes = (k ** levels - 1) // (k - 1)
    vocab = int(math.exp(rng.uniform(math.log(1000), math.log(152064))))
    vocab -= vocab % rng.choice((1, 1, 8, 64, 64))
    pad = rng.choice((1, 1, 64))
    dtype = rng.choice(("bf16", "bf16", "bf16", "fp32"))
    # ids in all rows together: some way below the largest listed case, by how often a row is read
    most = (1 << 28 if k > 2 else 1 << 29 if method == "compare" or dtype == "fp32" else 1 << 30) // (nodes * vocab)
    batch = max(1, min(1024, most, int(math.exp(rng.uniform(0.0, math.log(1025))))))
    call = rng.choice(("step", "step", "draft", "verify"))
    return _case(None, call, method, batch, levels, k, vocab, pad, dtype, leaves=rng.random() < 0.4,
                 handover=rng.random() < 0.6, probabilities=call == "verify" and rng.random() < 0.6,
                 temperature=rng.choice((0.0, 0.6, 1.0)), sigma=rng.choice((0.5, 1.0, 1.5)),
                 adversarial=rng.choice((0.0, 0.0, 0.0, 0.1)))


def _nodes(case):
    return (case["k"] ** case["levels"] - 1) // (case["k"] - 1)


def _degenerate(lp, lq, share, gen):
    """Some rows of the chunk become p = q, one-hot (hard, soft), disjoint, near-uniform or full of ties."""
    rows, V = lp.shape
    kind = torch.randint(0, 6, (rows,), generator=gen, device=lp.device)
    kind[torch.rand(rows, generator=gen, device=lp.device) >= share] = -1
    at = [torch.nonzero(kind == j).flatten() for j in range(6)]
    lq[at[0]] = lp[at[0]]
    for j, low in ((1, -math.inf), (2, -60.0)):
        hot = torch.randint(0, V, (len(at[j]),), generator=gen, device=lp.device)
        lq[at[j]] = low
        lq[at[j], hot] = 0.0
    if len(at[3]):
        tp, tq = lp[at[3]].topk(min(64, V // 4)).indices, lq[at[3]].topk(min(64, V // 4)).indices
        lq[at[3]] = lq[at[3]].scatter(1, tp, -math.inf)
        lp[at[3]] = lp[at[3]].scatter(1, tq, -math.inf)
    lq[at[4]] = torch.randn((len(at[4]), V), generator=gen, device=lp.device) * 0.01
    lp[at[5]] = torch.round(lp[at[5]] * 2.0) / 2.0
    lq[at[5]] = torch.round(lq[at[5]] * 2.0) / 2.0


def _sample(lq, T, k, gen):
    """Drafts of the rows by perturbed maxima (Gumbel): k ids without replacement, one more that is
    independent of them per further draft, and the hub (lowest id of the largest logit)."""
    V = lq.shape[1]
    ids = torch.arange(V, device=lq.device)
    hub = torch.where(lq == lq.amax(1, keepdim=True), ids, V).amin(1)
    score = lq / T[:, None]
    free = []
    for _ in range(k - 1):
        free.append((score - torch.rand(lq.shape, generator=gen, device=lq.device).clamp_(1e-30).log_().neg_().log_()).argmax(1))
    score -= torch.rand(lq.shape, generator=gen, device=lq.device).clamp_(1e-30).log_().neg_().log_()
    without = []
    for _ in range(k):
        best, x = score.max(1)
        taken = torch.stack(without, 1) if without else x[:, None] - 1
        spare = (ids[None, :k] != taken[:, :, None]).all(1).to(torch.int8).argmax(1)  # nothing left to draw from
        x = torch.where(best == -math.inf, spare, x)
        without.append(x)
        score.scatter_(1, x[:, None], -math.inf)
    return without, [without[0]] + free, hub


def prepare(case, seed):
    dev = "cuda"
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    B, N, V, k = case["batch"], _nodes(case), case["vocab"], case["k"]
    wide = -(-V // case["pad"]) * case["pad"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    target = torch.empty((B * N, wide), dtype=dt, device=dev)[:, :V]
    draft = torch.empty((B * N, wide), dtype=dt, device=dev)[:, :V]
    # u = (integer of 24 bits) / 2^24, one per draft, one per test, one for the residual draw
    uniforms = torch.randint(0, 1 << 24, (B, N, 2 * k + 1), generator=gen, device=dev).to(torch.float32) * 2.0 ** -24
    T = case["temperature"]
    if T == 0.0:
        T = 0.6 + 0.4 * torch.rand(B, generator=gen, device=dev)
    row_T = (T if isinstance(T, torch.Tensor) else torch.full((B,), T, device=dev)).repeat_interleave(N)
    # a row: Zipf-shaped prior over a permutation of the ids plus noise; small vocabularies have no prior
    small = V < 4096
    prior = -1.2 * torch.log1p(torch.randperm(V, generator=gen, device=dev).to(torch.float32)) * (not small)
    tokens = {m: torch.empty((B * N, k), dtype=torch.int32, device=dev) for m in METHODS}
    chunk = max(1, (1 << 28) // V)
    for r0 in range(0, B * N, chunk):
        r1 = min(B * N, r0 + chunk)
        lp = torch.randn((r1 - r0, V), generator=gen, device=dev) * (2.0 if small else 1.0) + prior
        lq = lp + torch.randn((r1 - r0, V), generator=gen, device=dev) * case["sigma"]
        if case["adversarial"] > 0:
            _degenerate(lp, lq, case["adversarial"], gen)
        target[r0:r1] = lp
        draft[r0:r1] = lq
        if case["call"] == "verify":
            lq.copy_(draft[r0:r1])
            without, free, hub = _sample(lq, row_T[r0:r1], k, gen)
            tokens["rrs"][r0:r1] = torch.stack(free, 1)
            tokens["rrsw"][r0:r1] = torch.stack(without, 1)
            if k == 2:  # (x, hub), or (hub, x) with x from the other ids
                tokens["spechub"][r0:r1] = torch.stack((without[0], torch.where(without[0] == hub, without[1], hub)), 1)
    target, draft = target.view(B, N, V), draft.view(B, N, V)
    tree = sh.Tree.heap(N, leaves_sample=case["leaves"]) if k == 2 else sh.Tree.kary(k, case["levels"], case["leaves"])
    out = [alloc_verify_outputs(B, N, tree.levels, torch.device(dev, torch.cuda.current_device()), k)
           for _ in (METHODS if case["method"] == "compare" else "1")]
    s = dict(case=case, target=target, draft=draft, uniforms=uniforms, T=T, tree=tree,
             out=dict(zip(METHODS, out)) if case["method"] == "compare" else out[0])
    if case["call"] == "verify":
        s["tokens"] = {m: t.view(B, N, k) for m, t in tokens.items()}
        if case["method"] != "compare":
            s["tokens"] = s["tokens"][case["method"]]
        if case["handover"]:  # the records that the draft step of this iteration left
            s["stats"] = _draft(dict(s, case=dict(case)))["stats"]
    return s


def _draft(s):
    c, a = s["case"], (s["draft"], s["uniforms"], s["tree"])
    if c["method"] == "compare":
        return (sh.mdsd_compare_draft_sample_stats if c["handover"] else sh.mdsd_compare_draft_sample)(*a, s["T"])
    if c["method"] == "spechub":
        return (sh.spechub_draft_sample_stats if c["handover"] else sh.spechub_draft_sample)(*a, s["T"])
    return (sh.rrs_draft_sample_stats if c["handover"] else sh.rrs_draft_sample)(*a, c["method"] == "rrsw", s["T"])


def _verify(s, tokens, stats):
    c = s["case"]
    a = (s["target"], s["draft"]) + ((stats,) if c["handover"] else ()) + (tokens, s["uniforms"], s["tree"])
    kw = dict(out=s["out"], probabilities=c["probabilities"])
    if c["method"] == "compare":
        return (sh.mdsd_compare_verify_tree_stats if c["handover"] else sh.mdsd_compare_verify_tree)(*a, s["T"], **kw)
    if c["method"] == "spechub":
        return (sh.spechub_verify_tree_stats if c["handover"] else sh.spechub_verify_tree)(*a, s["T"], **kw)
    return (sh.rrs_verify_tree_stats if c["handover"] else sh.rrs_verify_tree)(*a, c["method"] == "rrsw", s["T"], **kw)


def run(s):
    c, d, v = s["case"], None, None
    if c["call"] != "verify":
        d = _draft(s)
    if c["call"] == "step":
        v = _verify(s, {m: d[m]["tokens"] for m in METHODS} if c["method"] == "compare" else d["tokens"], d.get("stats"))
    elif c["call"] == "verify":
        v = _verify(s, s["tokens"], s.get("stats"))
    # the records of draft statistics are the library's own, for its verification alone; beta and rate are
    # written only where probabilities were asked for
    left_out = ("stats",) if c["probabilities"] else ("stats", "beta", "rate")
    pick = lambda o: o and {n: pick(x) if isinstance(x, dict) else x for n, x in o.items() if n not in left_out}  # noqa: E731
    return {"draft": pick(d), "verify": pick(v)}


def work(case):
    """Every logit of the tensors that the call takes, the uniforms, drafts and outputs, once each.  Of a
    row of q or p, an exponential, a product and a sum per id; verification compares the two: about 8 more."""
    B, N, V, k = case["batch"], _nodes(case), case["vocab"], case["k"]
    size = 2 if case["dtype"] == "bf16" else 4
    methods = 3 if case["method"] == "compare" else 1
    verifying = (k ** (case["levels"] - 1) - 1) // (k - 1) if case["leaves"] else N
    q_rows = verifying if case["call"] == "verify" else N
    p_rows = 0 if case["call"] == "draft" else N
    small = N * 4 * (2 * k + 1)
    if case["call"] != "verify":
        small += methods * N * 4 * (k + 1) + (12 * N if case["method"] in ("spechub", "compare") else 0)
    if case["call"] != "draft":
        small += methods * (N * 4 * (k + 4 + (2 * k + 1 if case["probabilities"] else 0)) + 8 + 8 * case["levels"])
    flops = 3 * (q_rows + p_rows) * V + (8 * methods * verifying * V if p_rows else 0)
    return {"bytes": B * ((q_rows + p_rows) * V * size + small), "flops": B * flops}


def tolerance(case):
    """Sums of up to 152064 fp32 terms: 1e-5, twice for the exponent's own rounding at T = 0.6; an acceptance
    probability whose numerator is a difference of nearly equal probabilities carries more (some 1e-3, in one of a
    hundred thousand rows).  A draw whose uniform lies within fp32 rounding of an edge between two ids may take
    the neighbour (2e-4 of the drafts at V = 32000, T = 0.6; up to 5e-3 on the flattest rows of 128256 ids and
    more), and the probability reported for that pair of drafts is then the neighbour's."""
    if case["call"] == "verify":
        return {"rel": 2e-5, "max": 5e-3, "differ": 1e-2}
    return {"rel": 3e-3, "max": 0.5, "differ": 1e-2}
