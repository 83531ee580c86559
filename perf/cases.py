"""What the speed of this framework is measured on: draft + verify steps and the calls around them, as a serving program
issues them through `paper_2402_14160_b200.step` and `paper_2402_14160_b200.api`.

A case names a path and its sizes.  Rows are Gaussian logits made on the GPU from the seed (target = draft + noise, as
in `workloads`), in the storage type of the case.  The paths:

  c        one RSD step with constant branching factors: Gumbel-Top-k over the parent rows, then the walk (RsdCStep)
  s        one RSD step with Stochastic Beam Search, rows of all levels ready (RsdSStep: rsd_sbs_draft_tree + walk)
  levels   the same with one rsd_sbs_step call per level, as an autoregressive drafter needs it
  cold     path c with sampling temperatures for drafter and target, and the picks' log-probabilities returned
  warped   path s on rows that go through rsd_filter_rows first (top-k / nucleus sampling)
  filter   rsd_filter_rows alone (a sampler's logit warping)
  rule     the walk under one of the baseline verification rules over trees of independent draws
  residual rsd_resample_residual alone, with the residual distribution returned
"""
import torch

from paper_2402_14160_b200 import api
from paper_2402_14160_b200 import step as rsd_step

ELEM = {"f32": 4, "bf16": 2}
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # one request, a small tree: what a single user waits for; launches and the walk's latency decide
        dict(name="c_one_f32", path="c", batch=1, vocab=32000, dtype="f32", branching="2,2,2", sigma=2.0, noise=0.5),
        # a small serving batch in fp32
        dict(name="c_batch_f32", path="c", batch=64, vocab=32000, dtype="f32", branching="3,2,2,1", sigma=2.0, noise=1.0),
        # beam-search trees over rows that are log-probabilities already
        dict(name="s_logprob_f32", path="s", batch=32, vocab=32000, dtype="f32", width=6, depth=6, logprob=True, sigma=2.0, noise=0.7),
        # a large batch at OPT's vocabulary
        dict(name="c_opt_bf16", path="c", batch=256, vocab=50272, dtype="bf16", branching="4,2,2,1,1", sigma=3.0, noise=0.5),
        # full serving load: 1024 sequences, 64 drafted nodes each
        dict(name="s_serving_bf16", path="s", batch=1024, vocab=32000, dtype="bf16", width=8, depth=8, logprob=False, sigma=2.0, noise=0.8),
        # one request with an autoregressive drafter: eight small drafting launches and a walk
        dict(name="levels_one_bf16", path="levels", batch=1, vocab=32000, dtype="bf16", width=4, depth=4, logprob=False, sigma=2.0, noise=0.8),
        # an autoregressive drafter, a moderate batch, a large vocabulary
        dict(name="levels_large_vocab_bf16", path="levels", batch=32, vocab=128000, dtype="bf16", width=6, depth=5, logprob=False, sigma=2.0,
             noise=0.7),
        # nucleus sampling (top-p 0.95 at temperature 1): every draft and target row is filtered before the step
        dict(name="warped_topp_bf16", path="warped", batch=64, vocab=32000, dtype="bf16", width=5, depth=5, top_k=0, top_p=0.95, sigma=2.0,
             noise=0.7),
        # top-k and top-p on one row per request, as a plain sampler does
        dict(name="filter_rows_f32", path="filter", batch=32, rows=1, vocab=32000, dtype="f32", top_k=50, top_p=0.9, temp_t=1.0, sigma=3.0),
        # temperature 0.3 over a vocabulary with one added token (rows off every vector boundary), log-probabilities returned
        dict(name="cold_odd_bf16", path="cold", batch=64, vocab=32001, dtype="bf16", branching="3,2,1", temp_d=0.3, temp_t=0.3, sigma=2.0,
             noise=0.5),
        # multi-round rejection sampling with the paper's own last draw, to compare acceptance on equal inputs
        dict(name="rule_multiround_bf16", path="rule", batch=128, vocab=32000, dtype="bf16", branching="4,2,2", rule="multiround", gamma=1.0,
             top1=True, sigma=2.0, noise=0.7),
        # the residual of a few rejected tokens, returned whole
        dict(name="residual_f32", path="residual", batch=256, vocab=32000, dtype="f32", rejected=3, sigma=2.0, noise=0.7),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _tree_sizes(case):
    """(parent rows, nodes with the root, levels)"""
    if "branching" in case:
        sizes = [1]
        for b in _branching(case):
            sizes.append(sizes[-1] * b)
        return sum(sizes[:-1]), sum(sizes), len(sizes) - 1
    return 1 + case["width"] * (case["depth"] - 1), 1 + case["width"] * case["depth"], case["depth"]


def _branching(case):
    return [int(b) for b in case["branching"].split(",")]


def draw(rng):
    """One more case: the listed paths at sizes over their whole ranges."""
    path = rng.choice(["c", "c", "s", "s", "levels", "cold", "warped", "filter", "rule", "residual"])
    dtype = rng.choice(["f32", "bf16"])
    vocab = _log_int(rng, 2000, 131072)
    if path in ("warped", "filter"):
        vocab = min(vocab, 50000 if dtype == "f32" else 100000)   # the filter keeps a row on chip
    align = rng.choice([1, 8, 16, 32, 64])                        # model vocabularies are mostly padded, not always
    vocab = max(2000, vocab // align * align)
    case = dict(path=path, vocab=vocab, dtype=dtype, sigma=rng.choice([1.5, 2.0, 3.0]))
    if path in ("c", "cold", "rule"):
        levels, cap = rng.randint(1, 5), 60
        sizes, bs = [1], []
        for _ in range(levels):
            b = rng.randint(1, 4)
            if sum(sizes) + sizes[-1] * b > cap:
                b = 1
            bs.append(b)
            sizes.append(sizes[-1] * b)
        case["branching"] = ",".join(str(b) for b in bs)
    if path in ("s", "levels", "warped"):
        case.update(width=rng.randint(2, 8), depth=rng.randint(2, 8))
    if path in ("s", "levels"):
        case["logprob"] = dtype == "f32" and rng.random() < 0.5
    if path == "cold":
        case.update(temp_d=rng.choice([0.3, 0.7]), temp_t=rng.choice([0.3, 0.7]))
    if path in ("warped", "filter"):
        case.update(top_k=rng.choice([0, 0, 50, 200]), top_p=rng.choice([0.8, 0.9, 0.95]))
    if path == "filter":
        case.update(rows=rng.choice([1, 1, 5, 9]), temp_t=rng.choice([0.7, 1.0]))
    if path == "rule":
        case.update(rule=rng.choice(["multiround", "kseq"]), gamma=rng.choice([1.5, 2.0]), top1=rng.random() < 0.5)
    if path == "residual":
        case["rejected"] = rng.randint(0, 4)
    if path != "filter":
        case["noise"] = rng.choice([0.5, 0.7, 1.0])
    # batch: 1 .. 1024 with at most 4 GB of rows (half the largest listed case), a quarter of it where every row is
    # also rewritten
    per_seq = _row_count(case) * vocab * ELEM[dtype]
    most = (1 if path in ("warped", "filter", "rule", "residual", "cold") else 4) * 10 ** 9
    case["batch"] = _log_int(rng, 1, max(1, min(1024, most // per_seq)))
    return case


def _row_count(case):
    if case["path"] == "filter":
        return case["rows"]
    if case["path"] == "residual":
        return 2
    p, n, _ = _tree_sizes(case)
    return p + n


def _rows(case, gen, n_draft, n_target):
    """Draft [B, n_draft, V] and target [B, n_target, V] rows; target = draft + noise."""
    B, V, dt = case["batch"], case["vocab"], DTYPE[case["dtype"]]
    draft = torch.empty((B, n_draft, V), dtype=dt, device="cuda") if n_draft else None
    target = torch.empty((B, n_target, V), dtype=dt, device="cuda")
    per = max(n_draft, n_target)
    chunk = max(1, min(B, (1 << 26) // (per * V)))
    for b in range(0, B, chunk):
        n = min(chunk, B - b)
        base = torch.randn((n, per, V), generator=gen, device="cuda").mul_(case["sigma"])
        if case.get("logprob"):
            base = torch.log_softmax(base, dim=-1)
        if n_draft:
            draft[b:b + n].copy_(base[:, :n_draft])
        if "noise" in case:
            base.add_(torch.randn((n, per, V), generator=gen, device="cuda"), alpha=case["noise"])
        target[b:b + n].copy_(base[:, :n_target])
    return draft, target


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    path, B, V = case["path"], case["batch"], case["vocab"]
    st = dict(case=case, seed=seed & 0xFFFFFFFF)
    if path == "filter":
        _, st["target"] = _rows(case, gen, 0, case["rows"])
        st["out"] = dict(rows=torch.empty_like(st["target"]), kept=torch.empty((B, case["rows"]), dtype=torch.int32, device="cuda"),
                         status=torch.empty((B,), dtype=torch.int32, device="cuda"))
        return st
    if path == "residual":
        draft, target = _rows(case, gen, 1, 1)
        st["draft"], st["target"] = draft[:, 0], target[:, 0]
        st["node"] = torch.zeros((B,), dtype=torch.int32, device="cuda")
        k = case["rejected"]
        st["rejected"] = None
        if k:   # tokens that a drafter proposes (without replacement) and that the target model rejects: q(x) < p(x)
            logp, logq = torch.log_softmax(st["draft"].float(), dim=-1), torch.log_softmax(st["target"].float(), dim=-1)
            noise = -torch.log(-torch.log(torch.rand((B, V), generator=gen, device="cuda").clamp_(1e-7, 1 - 1e-7)))
            noise.add_(logp).masked_fill_(logq >= logp, float("-inf"))
            st["rejected"] = torch.topk(noise, k, dim=-1).indices.to(torch.int32).contiguous()
        return st
    P, N1, L = _tree_sizes(case)
    st["draft"], st["target"] = _rows(case, gen, P, N1)
    if path in ("c", "cold", "rule"):
        st["step"] = rsd_step.RsdCStep(B, V, _branching(case))
    else:
        st["step"] = rsd_step.RsdSStep(B, V, case["width"], case["depth"], draft_is_logprob=bool(case.get("logprob")),
                                       rows_ready=path != "levels")
    if path == "warped":
        for name in ("draft", "target"):
            rows = st[name]
            st["warp_" + name] = dict(rows=torch.empty_like(rows), kept=torch.empty(rows.shape[:2], dtype=torch.int32, device="cuda"),
                                      status=torch.empty((B,), dtype=torch.int32, device="cuda"))
    if path == "rule":   # the baselines' children are independent draws from their parent's row
        step = st["step"]
        tok = torch.full((B, N1), -1, dtype=torch.int32, device="cuda")
        for r in range(P):
            k, first = step.k_per_row[r], step.child_base[r]
            probs = torch.softmax(st["draft"][:, r].float(), dim=-1)
            tok[:, first:first + k] = torch.multinomial(probs, k, replacement=True, generator=gen).to(torch.int32)
        st["token"] = tok
    return st


def run(st):
    case, seed = st["case"], st["seed"]
    path = case["path"]
    if path == "filter":
        return api.rsd_filter_rows(st["target"], case["top_k"], case["top_p"], temperature=case["temp_t"], out=st["out"])
    if path == "residual":
        return api.rsd_resample_residual(st["draft"], st["target"], st["rejected"], st["node"], seed, 0, want_residual=True)
    step = st["step"]
    if path == "cold":
        drafted = api.rsd_gumbel_topk_draft(st["draft"], step.k_per_row, step.rng_node, seed, 0, max_k=step.max_k, want_values=True,
                                            child_base=step.child_base, node_token=step.token, temperature=case["temp_d"])
        walked = api.rsd_verify_tree(st["draft"], st["target"], step.parent, step.token, step.L, seed, 0,
                                     draft_temperature=case["temp_d"], target_temperature=case["temp_t"])
        return dict(drafted=drafted, walked=walked)
    if path == "rule":
        return api.rsd_verify_tree_rule(st["draft"], st["target"], step.parent, st["token"], step.L,
                                        api.RULE_MULTIROUND if case["rule"] == "multiround" else api.RULE_KSEQ, case["gamma"],
                                        api.FINAL_GUMBEL_TOP1 if case["top1"] else api.FINAL_INVERSE_CDF, seed, 0)
    draft, target = st["draft"], st["target"]
    out = {}
    if path == "warped":
        for name in ("draft", "target"):
            out["warp_" + name] = api.rsd_filter_rows(st[name], case["top_k"], case["top_p"], out=st["warp_" + name])
        draft, target = st["warp_draft"]["rows"], st["warp_target"]["rows"]
    out["walked"] = step.run(draft, target, seed, 0)
    out["token"] = step.token
    if path == "c":
        out["drafted"] = step.draft_out
    else:
        out["parent"] = step.parent
        out["count"] = step.count
        out["beam"] = step.state[(case["depth"] - 1) % 2] if path == "levels" else step.tree_out
    return out


def work(case):
    """Rows read once and rows written once.  A walk reads the target rows it visits: the root's and about a third of a
    level's further ones on these inputs (the drafter's rows are counted where they are drafted from)."""
    row = case["vocab"] * ELEM[case["dtype"]]
    B, V, path = case["batch"], case["vocab"], case["path"]
    if path == "filter":
        n = B * case["rows"]
        return {"bytes": 2 * n * row, "flops": 4 * n * V}
    if path == "residual":
        n = B * (2 if case["rejected"] else 1)
        return {"bytes": n * row + B * V * 4, "flops": 4 * (n + B * case["rejected"]) * V}
    P, N1, L = _tree_sizes(case)
    visited = 1 + L / 3
    if path == "rule":
        return {"bytes": 2 * B * visited * row, "flops": 8 * B * visited * V}
    if path == "warped":
        return {"bytes": 2 * B * (P + N1) * row, "flops": 8 * B * (P + visited) * V}
    return {"bytes": B * (P + visited) * row, "flops": 4 * B * (P + visited) * V}


def tolerance(case):
    """Tokens, nodes, lengths and flags are decisions: sums in another order flip one only where its margin is within
    fp32 rounding (about one last draw in several thousand), so a few in a thousand of the values may differ, or those of
    one sequence.  Log-probabilities, perturbed values and residual probabilities are fp32 sums and fast exponentials;
    against the same path in double the largest relative error seen is 2.4e-7 (2-norm) and 1.3e-5 (single value)."""
    return {"rel": 1e-6, "max": 5e-5, "differ": min(0.01, max(0.002, 1.01 / case["batch"]))}
