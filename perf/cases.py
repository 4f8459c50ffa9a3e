"""The work whose speed is watched: listed cases and draws from the ranges they stand for.

Every case is one call sequence that a decoding loop built on this library makes once per step, through
`paper_2408_15562_b200.binding.Context`:

  step     `verify_step`: attention of one layer, acceptance, compaction, on device buffers
  paged    the same step on a cache of 128-row blocks: `tree_attn_paged`, `tree_accept`, `kv_compact_paged`,
           the tree's K/V rows living in the cache
  host     `verify_step_host`: the step from pinned host buffers
  lm_head  `lm_head_accept` and `kv_append`: the target's vocabulary product with the acceptance behind it,
           then the accepted K/V rows written into the cache
  draft    one draft phase: `draft_expand` level by level, then `tree_build`
  sampler  `feature_sampler`: the draft model's input synthesis on the frontier rows

Sizes are those of the workloads in `synth.WORKLOADS`, of the tests and of the benchmark, or generic.
Inputs follow `synth`'s recipe (logits ~ N(0, sigma^2), draft distribution softmax(logits + N(0, 1)), siblings drawn
from it without replacement, trees cut from a top-k expansion), with the random numbers made on the GPU.
"""
import math

import numpy as np
import torch

from paper_2408_15562_b200 import binding, synth

D = synth.HEAD_DIM
SAMPLED_ROWS = 3          # draft rows a sampling walk reads: about the mean accepted length of these inputs


def listed():
    return [
        # Smallest step: one greedy sequence, short context, a tree of 26 nodes, small vocabulary: launches and latency.
        dict(name="step_tiny_greedy", kind="step", batch=1, hq=32, hkv=32, lo=256, hi=256, nodes=26, depth=4, branch=3,
             tree="bfs", vocab=32000, sampling=0, temp=1.0, sigma=2.0, layers=1),
        # The ordinary interactive step: one sampled sequence, four query heads per KV head, 2K context, large vocabulary.
        dict(name="step_gqa4_2k_sample", kind="step", batch=1, hq=32, hkv=8, lo=2048, hi=2048, nodes=60, depth=6, branch=10,
             tree="pruned", vocab=128256, sampling=1, temp=1.0, sigma=3.0, layers=1),
        # Every query head with its own KV head (52 of them), 4K context: the KV cache is what is read.
        dict(name="step_mha52_4k_sample", kind="step", batch=1, hq=52, hkv=52, lo=4096, hi=4096, nodes=60, depth=6, branch=10,
             tree="pruned", vocab=32000, sampling=1, temp=1.0, sigma=3.0, layers=1),
        # Long context with eight query heads per KV head: the attention is a contraction.
        dict(name="step_gqa8_8k_sample", kind="step", batch=1, hq=64, hkv=8, lo=8192, hi=8192, nodes=60, depth=6, branch=10,
             tree="pruned", vocab=128256, sampling=1, temp=1.0, sigma=3.0, layers=1),
        # A server's batch: 16 ragged sequences, half greedy and half sampled, the accepted rows compacted in 32 layers.
        dict(name="step_batch16_ragged", kind="step", batch=16, hq=32, hkv=8, lo=512, hi=4096, nodes=60, depth=6, branch=10,
             tree="pruned", vocab=128256, sampling=8, temp=1.0, sigma=3.0, layers=32),
        # A paged cache, trees beyond 64 nodes, a vocabulary that is no multiple of four, tree rows in the cache.
        dict(name="paged_batch4_wide_tree", kind="paged", batch=4, hq=32, hkv=8, lo=300, hi=3000, nodes=130, depth=8, branch=10,
             tree="pruned", vocab=50257, sampling=2, temp=0.8, sigma=3.0, layers=4),
        # A caller whose logits and draft rows are on the host: the step end to end over the host link.
        dict(name="host_gqa4_2k_sample", kind="host", batch=1, hq=32, hkv=8, lo=2048, hi=2048, nodes=60, depth=6, branch=10,
             tree="pruned", vocab=128256, sampling=1, temp=1.0, sigma=3.0, layers=1),
        # Vocabulary product and acceptance of one sampled sequence: the matrix is streamed once.
        dict(name="lm_head_60_rows_sample", kind="lm_head", batch=1, hidden=4096, hkv=8, lo=2048, hi=2048, nodes=60, depth=6,
             branch=10, tree="pruned", vocab=128256, sampling=1, temp=1.0, sigma=3.0, layers=32),
        # The same for a server's batch of 16, half of it greedy: 960 rows, where the product is a contraction.
        dict(name="lm_head_960_rows_mixed", kind="lm_head", batch=16, hidden=4096, hkv=8, lo=512, hi=4096, nodes=60, depth=6,
             branch=10, tree="pruned", vocab=128256, sampling=8, temp=1.0, sigma=3.0, layers=4),
        # Draft phase of one sequence (five levels of ten by ten, small vocabulary): a chain of small launches.
        dict(name="draft_batch1", kind="draft", batch=1, vocab=32000, levels=5, top_k=10, width=10, nodes=60),
        # The same for a batch of 16 at a large vocabulary: every level reads 82 MB of log-probabilities.
        dict(name="draft_batch16", kind="draft", batch=16, vocab=128256, levels=5, top_k=10, width=10, nodes=60),
        # Input synthesis of one draft level, ten frontier rows: three matrices are streamed once.
        dict(name="sampler_10_rows", kind="sampler", rows=10, hidden=4096, inter=14336),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "paged", "lm_head", "lm_head", "draft", "draft", "sampler", "host"])
    if kind == "sampler":
        hidden = 8 * _log(rng, 128, 1024)
        return dict(kind=kind, rows=_log(rng, 1, 128), hidden=hidden, inter=8 * int(hidden * rng.uniform(2.5, 4.0) / 8))
    if kind == "draft":
        k = rng.choice([4, 5, 8, 10, 16])
        return dict(kind=kind, batch=_log(rng, 1, 16), vocab=rng.choice([32000, 32001, 50257, 128256, 151936]),
                    levels=rng.randint(3, 4 if k == 16 else 6), top_k=k, width=k, nodes=rng.randint(24, 64))
    batch = _log(rng, 1, {"host": 2, "paged": 8}.get(kind, 16))
    lo = _log(rng, 64, 4096)
    hi = min(8192 if batch == 1 else 4096, int(lo * rng.uniform(1.0, 4.0)))
    hi = max(lo, min(hi, 65536 // batch))
    case = dict(kind=kind, batch=batch, lo=lo, hi=hi, nodes=rng.randint(65, 256) if kind == "paged" else _log(rng, 8, 60),
                depth=rng.randint(4, 8), branch=rng.choice([3, 4, 8, 10]), tree="pruned",
                vocab=rng.choice([32000, 32001, 50257, 128256]), sampling=rng.choice([0, batch // 2, batch, batch]),
                temp=rng.choice([0.6, 0.8, 1.0, 1.0]), sigma=3.0)
    if kind == "lm_head":
        return dict(case, hidden=8 * _log(rng, 128, 512), hkv=8, layers=4)
    hq, hkv = rng.choice([(32, 32), (32, 8), (52, 52), (64, 8), (28, 4), (40, 10)])
    if batch > 4 and hkv > 10:
        hq, hkv = 32, 8
    return dict(case, hq=hq, hkv=hkv, layers=rng.choice([1, 1, 4]))


# ---- inputs ---------------------------------------------------------------------------------------------------


def _tree_inputs(case, seed):
    """Prefix lengths and parents (host arrays), the same for every kind that has a tree."""
    rng = np.random.default_rng([seed, 17])
    B, N = case["batch"], case["nodes"]
    prefix = rng.integers(case["lo"], case["hi"] + 1, size=B).astype(np.int32)
    parents = []
    for _ in range(B):
        if case["tree"] == "bfs":
            p = synth.bfs_tree(N, case["branch"])
        else:
            p = synth.pruned_tree(rng, N, case["depth"], case["branch"])
        if len(p) < N:                      # the expansion was smaller than the budget: the rest hangs on the root
            p = np.concatenate([p, np.zeros(N - len(p), np.int32)])
        parents.append(p)
    return prefix, np.stack(parents).astype(np.int32)


def _draft_side(case, gen, logits, parent):
    """Draft distribution, draft tokens, temperatures and uniforms for logits [B][N][V] on the GPU.

    Sequence b samples iff b >= batch - sampling.  A greedy sequence's children are the best tokens of the noisy
    logits; a sampled sequence's are drawn one after another without replacement from the draft row (the m largest
    of log q + Gumbel noise, in that order)."""
    B, N, V = logits.shape
    n_sampling = case["sampling"]
    draft = torch.empty_like(logits) if n_sampling else None
    tokens = np.zeros((B, N), np.int32)
    for b in range(B):
        noisy = torch.randn((N, V), generator=gen, device="cuda").add_(logits[b])
        sampled = b >= B - n_sampling
        if n_sampling:
            draft[b] = torch.softmax(noisy, -1)
        if sampled:
            noisy -= torch.log(-torch.log(torch.rand((N, V), generator=gen, device="cuda").clamp_(1e-12, 1 - 6e-8)))
        children = synth.children_lists(parent[b])
        top = noisy.topk(min(V, max(len(c) for c in children) or 1), dim=-1).indices.cpu().numpy()
        for i, c in enumerate(children):
            tokens[b, c] = top[i, :len(c)]
    temp = torch.zeros(B)
    temp[B - n_sampling:] = case["temp"]
    uniforms = torch.rand((B, N + 1), generator=gen, device="cuda").clamp_(max=1 - 6e-8) if n_sampling else None
    return draft, torch.from_numpy(tokens).cuda(), temp.cuda(), uniforms


def _bf16(gen, shape, scale=1.0):
    out = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    out.normal_(0.0, scale, generator=gen)
    return out


def _logits(case, gen):
    return torch.randn((case["batch"], case["nodes"], case["vocab"]), generator=gen, device="cuda").mul_(case["sigma"])


def _results(batch, nodes):
    i32 = dict(dtype=torch.int32, device="cuda")
    return dict(path=torch.empty((batch, nodes), **i32), n_acc=torch.empty((batch,), **i32),
                bonus=torch.empty((batch,), **i32), new_len=torch.empty((batch,), **i32))


def _max_len(case, nodes):
    return -(-(case["hi"] + nodes) // 64) * 64


def _prepare_step(case, seed, gen, host):
    B, N, V, hq, hkv, layers = (case[k] for k in ("batch", "nodes", "vocab", "hq", "hkv", "layers"))
    prefix, parent = _tree_inputs(case, seed)
    s = dict(parent=torch.from_numpy(parent).cuda(), prefix=torch.from_numpy(prefix).cuda(), q=_bf16(gen, (B, N, hq, D)),
             tree_k=_bf16(gen, (B, hkv, N, D)), tree_v=_bf16(gen, (B, hkv, N, D)), logits=_logits(case, gen))
    s["draft"], s["tokens"], s["temp"], s["uniforms"] = _draft_side(case, gen, s["logits"], parent)
    max_len = _max_len(case, N)
    s["cache"] = _bf16(gen, (layers, 2, B, hkv, max_len, D))
    for b, L in enumerate(prefix.tolist()):      # the target's forward has left the tree's rows behind the prefix
        s["cache"][0, 0, b, :, L:L + N] = s["tree_k"][b]
        s["cache"][0, 1, b, :, L:L + N] = s["tree_v"][b]
    s["out"] = torch.empty_like(s["q"])
    s.update(_results(B, N))
    s["ctx"] = binding.Context(hq, hkv, V, max_len, max_nodes=N, n_layers=layers, max_batch=B)
    if host:
        for k, t in s.items():
            if isinstance(t, torch.Tensor) and k != "cache":
                s[k] = t.cpu().pin_memory()
    return s


def _prepare_paged(case, seed, gen):
    B, N, V, hq, hkv, layers = (case[k] for k in ("batch", "nodes", "vocab", "hq", "hkv", "layers"))
    prefix, parent = _tree_inputs(case, seed)
    s = dict(parent=torch.from_numpy(parent).cuda(), prefix=torch.from_numpy(prefix).cuda(), q=_bf16(gen, (B, N, hq, D)),
             logits=_logits(case, gen))
    s["draft"], s["tokens"], s["temp"], s["uniforms"] = _draft_side(case, gen, s["logits"], parent)
    per_seq = -(-(case["hi"] + N) // 128)
    n_blocks = B * per_seq
    table = np.random.default_rng([seed, 23]).permutation(n_blocks).astype(np.int32).reshape(B, per_seq)
    s["table"] = torch.from_numpy(table).cuda()
    s["pool"] = _bf16(gen, (layers, 2, n_blocks, hkv, 128, D))
    s["out"] = torch.empty_like(s["q"])
    s.update(_results(B, N))
    s["ctx"] = binding.Context(hq, hkv, V, per_seq * 128, max_nodes=N, n_layers=layers, max_batch=B)
    return s


def _prepare_lm_head(case, seed, gen):
    B, N, V, H, hkv, layers = (case[k] for k in ("batch", "nodes", "vocab", "hidden", "hkv", "layers"))
    prefix, parent = _tree_inputs(case, seed)
    s = dict(parent=torch.from_numpy(parent).cuda(), prefix=torch.from_numpy(prefix).cuda(), hidden=_bf16(gen, (B, N, H)),
             weight=_bf16(gen, (V, H), case["sigma"] / math.sqrt(H)))
    logits = torch.empty((B, N, V), dtype=torch.float32, device="cuda")
    for b in range(B):
        logits[b] = s["hidden"][b] @ s["weight"].T
    s["draft"], s["tokens"], s["temp"], s["uniforms"] = _draft_side(case, gen, logits, parent)
    s["logits"] = logits.zero_() if case["sampling"] else None     # an all-greedy batch wants no logits
    max_len = _max_len(case, N)
    s["cache"] = _bf16(gen, (layers, 2, B, hkv, max_len, D))
    s["tree_kv"] = _bf16(gen, (layers, 2, B, hkv, N, D))
    s.update(_results(B, N))
    s["ctx"] = binding.Context(hkv, hkv, V, max_len, max_nodes=N, n_layers=layers, max_batch=B)
    return s


def _draft_frontiers(case):
    """(frontier nodes, first candidate index) of every level."""
    got, base = [], 0
    for level in range(case["levels"]):
        f = 1 if level == 0 else case["width"]
        got.append((f, base))
        base += f * case["top_k"]
    return got, base


def _prepare_draft(case, seed, gen):
    B, V, k, width = case["batch"], case["vocab"], case["top_k"], case["width"]
    levels, cap = _draft_frontiers(case)
    i32, f32 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.float32, device="cuda")
    s = dict(levels=levels, cand=(torch.empty((B, cap), **i32), torch.empty((B, cap), **i32), torch.empty((B, cap), **f32)),
             root=torch.randint(V, (B,), generator=gen, device="cuda").to(torch.int32),
             logprobs=[torch.log_softmax(torch.randn((B, f, V), generator=gen, **f32) * 3.0, -1) for f, _ in levels],
             frontier=[(torch.full((B, 1), -1, **i32), torch.zeros((B, 1), **f32))] +
                      [(torch.empty((B, width), **i32), torch.empty((B, width), **f32)) for _ in levels],
             tree=tuple(torch.empty((B, case["nodes"]), **i32) for _ in range(3)) + (torch.empty((B,), **i32),),
             anc=torch.empty((B, case["nodes"]), dtype=torch.int64, device="cuda"), top_k=k, width=width, nodes=case["nodes"])
    s["ctx"] = binding.Context(32, 8, V, 256, max_nodes=64, max_batch=B)
    return s


def _prepare_sampler(case, seed, gen):
    R, H, I = case["rows"], case["hidden"], case["inter"]
    bf = dict(dtype=torch.bfloat16, device="cuda")
    s = dict(f=_bf16(gen, (R, H)), e=_bf16(gen, (R, H)), up=_bf16(gen, (I, H), H ** -0.5), gate=_bf16(gen, (I, H), H ** -0.5),
             down=_bf16(gen, (H, I), I ** -0.5), inter=torch.empty((R, I), **bf), eta=torch.empty((R, H), **bf))
    need = binding.load().fspad_feature_sampler_workspace_bytes(R, H, I)
    s["work"] = torch.empty((need,), dtype=torch.uint8, device="cuda")
    s["ctx"] = binding.Context(8, 8, 128, 256, max_nodes=64)
    return s


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind in ("step", "host"):
        s = _prepare_step(case, seed, gen, kind == "host")
    else:
        s = {"paged": _prepare_paged, "lm_head": _prepare_lm_head, "draft": _prepare_draft,
             "sampler": _prepare_sampler}[kind](case, seed, gen)
    s["kind"] = kind
    return s


# ---- one pass --------------------------------------------------------------------------------------------------


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "step":
        ctx.verify_step(s["cache"], s["q"], s["tree_k"], s["tree_v"], s["parent"], s["prefix"], s["logits"], s["draft"],
                        s["tokens"], s["temp"], s["uniforms"], s["out"], s["path"], s["n_acc"], s["bonus"], s["new_len"])
        return s["out"], s["path"], s["n_acc"], s["bonus"], s["new_len"], s["cache"]
    if kind == "host":
        ctx.verify_step_host(s["cache"], s["q"], s["tree_k"], s["tree_v"], s["parent"], s["prefix"], s["logits"], s["draft"],
                             s["tokens"], s["temp"], s["uniforms"], s["out"], s["path"], s["n_acc"], s["bonus"], s["new_len"])
        return s["out"], s["path"], s["n_acc"], s["bonus"], s["new_len"], s["cache"]
    if kind == "paged":
        ctx.tree_attn_paged(s["q"], s["pool"][0, 0], s["pool"][0, 1], s["table"], None, None, s["parent"], s["prefix"], s["out"])
        ctx.tree_accept(s["logits"], s["draft"], s["tokens"], s["parent"], s["temp"], s["uniforms"], s["path"], s["n_acc"],
                        s["bonus"])
        ctx.kv_compact_paged(s["pool"], s["table"], s["path"], s["n_acc"], s["prefix"], s["new_len"])
        return s["out"], s["path"], s["n_acc"], s["bonus"], s["new_len"], s["pool"]
    if kind == "lm_head":
        ctx.lm_head_accept(s["hidden"], s["weight"], s["draft"], s["tokens"], s["parent"], s["temp"], s["uniforms"], s["logits"],
                           s["path"], s["n_acc"], s["bonus"])
        ctx.kv_append(s["cache"], s["tree_kv"], s["path"], s["n_acc"], s["prefix"], s["new_len"])
        return s["logits"], s["path"], s["n_acc"], s["bonus"], s["new_len"], s["cache"]
    if kind == "draft":
        for level, (_, base) in enumerate(s["levels"]):
            cand, logp = s["frontier"][level]
            ctx.draft_expand(s["logprobs"][level], logp, cand, s["top_k"], s["width"], base, *s["cand"],
                             *s["frontier"][level + 1])
        ctx.tree_build(*s["cand"], s["root"], s["nodes"], s["tree"], s["anc"])
        return s["tree"], s["anc"], s["cand"], s["frontier"][1:]
    ctx.feature_sampler(s["f"], s["e"], s["up"], s["gate"], s["down"], s["inter"], s["eta"], s["work"])
    return s["eta"], s["inter"]


# ---- what a pass cannot do without ----------------------------------------------------------------------------


def work(case):
    kind = case["kind"]
    if kind == "sampler":
        R, H, I = case["rows"], case["hidden"], case["inter"]
        return {"bytes": 3 * 2 * H * I + 2 * R * (3 * H + I), "flops": 3 * 2 * R * H * I}
    if kind == "draft":
        levels, cap = _draft_frontiers(case)
        return {"bytes": case["batch"] * (sum(f for f, _ in levels) * case["vocab"] * 4 + cap * 12), "flops": 0}
    B, N, V = case["batch"], case["nodes"], case["vocab"]
    L = (case["lo"] + case["hi"]) / 2
    moved = 2 * SAMPLED_ROWS * D * 2 * case["hkv"] * 2 * case["layers"] * B              # accepted rows, read and written
    draft = case["sampling"] * SAMPLED_ROWS * V * 4
    if kind == "lm_head":
        H = case["hidden"]
        logits = B * N * V * 4 if case["sampling"] else 0
        return {"bytes": 2 * V * H + 2 * B * N * H + logits + draft + moved, "flops": 2 * B * N * V * H}
    attn = B * (2 * case["hkv"] * (L + N) * D * 2 + 2 * N * case["hq"] * D * 2)
    return {"bytes": attn + B * N * V * 4 + draft + moved, "flops": 4 * B * N * case["hq"] * (L + 8) * D}


def tolerance(case):
    # Whole numbers (paths, tokens, counts) are the same; moved cache rows are copies.  The rest is about four times the
    # error against the same operation in 64 bits: attention and Feature Sampler round to bf16 what was accumulated in
    # 32 bits, from operands (probabilities, gated product) that are bf16 themselves: 2.3e-3, largest element 1.0e-2;
    # the vocabulary product is a 32-bit sum of 4096 products: 4.4e-6, largest element 1.6e-5.
    if case["kind"] == "draft":
        return "exact"
    if case["kind"] == "lm_head":
        return {"rel": 2e-5, "max": 8e-5, "differ": 0.0}
    return {"rel": 9e-3, "max": 4e-2, "differ": 0.0}
