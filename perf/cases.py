"""What a program built on this library has it do: the workloads whose speed is tracked.

A case is a dict of plain values:
  kind      "decode"    n free-running decoding steps (Amphista.step) from the end of a prompt already in the cache
            "calls"     the same step as its three calls (draft, verify_tree, accept) with pinned host buffers and a
                        synchronise per step: a server that streams every step's tokens to a client
            "answer"    prompts of one or more sequences prefilled, then n steps: one turn of a conversation, or of a batch
            "prefill"   one prompt through the target and the adaptation layers
            "project"   the projection primitive on its own (project_noalloc), as a chain over several layers' weights
  model     the widths (WIDTHS below), with "layers" target layers
  nodes     nodes of the candidate tree, root included
  ctx       prompt tokens (of the longest sequence of a batch)
  batch     sequences side by side
  steps     decoding steps of one pass
  rank      rank of the drafting vocabulary heads (0: full matrices)
  temperature  0: greedy, else sampling

The widths, trees, contexts and batch sizes are those of the shape table, the benchmark and its sweep (trees of 16 to
128 nodes, contexts of 256 to 8192 tokens, batches up to 8).  Everything goes through the public binding.
"""
import math
import random
from types import SimpleNamespace

import torch

from paper_2406_13170_b200 import Amphista, project_noalloc

DEVICE = "cuda:0"

#         d_model, heads, head_dim, d_ffn, vocab, dtype, candidates kept per drafting head
WIDTHS = {
    "tiny": (256, 4, 64, 688, 1000, "fp32", (4, 2, 2, 1)),
    "small_bf16": (512, 4, 128, 1408, 2048, "bf16", (6, 5, 4, 3)),
    "7b": (4096, 32, 128, 11008, 32000, "bf16", (10, 10, 10, 10)),
    "13b": (5120, 40, 128, 13824, 32000, "bf16", (10, 10, 10, 10)),
    "33b": (6656, 52, 128, 17920, 32000, "bf16", (10, 10, 10, 10)),
}
LAYERS = {"tiny": 2, "small_bf16": 3, "7b": 32, "13b": 40, "33b": 60}
K, N_SAL = 4, 2


def _case(kind, model, layers, nodes, ctx, batch=1, steps=0, rank=0, temperature=0.0, name=None):
    c = dict(kind=kind, model=model, layers=layers, nodes=nodes, ctx=ctx, batch=batch, steps=steps, rank=rank,
             temperature=temperature)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the benchmark's own workload: one user, greedy, 64-node tree behind a 512-token prompt
        _case("decode", "7b", 32, 64, 512, steps=12, name="decode_7b"),
        # the largest tree, low-rank drafting heads, a document in the context
        _case("decode", "7b", 32, 128, 2048, steps=6, rank=256, name="decode_7b_tree128_lr256"),
        # long context, a tree whose size is not a multiple of anything
        _case("decode", "7b", 32, 43, 7900, steps=6, name="decode_7b_ctx7900"),
        # the next larger model
        _case("decode", "13b", 40, 64, 1024, steps=6, name="decode_13b"),
        # a chat server: tokens handed over after every step, small tree
        _case("calls", "7b", 32, 26, 700, steps=8, name="calls_7b"),
        # four conversations side by side, ragged prompts, prefill included
        _case("answer", "7b", 32, 64, 300, batch=4, steps=16, name="answer_7b_batch4"),
        # eight short requests at a sampling temperature
        _case("answer", "7b", 32, 48, 130, batch=8, steps=8, temperature=0.7, name="answer_7b_batch8_sampled"),
        # time to the first token: the benchmark's prompt, and a long ragged one
        _case("prefill", "7b", 32, 64, 512, name="prefill_7b"),
        _case("prefill", "7b", 32, 64, 1900, name="prefill_7b_1900"),
        # the small shapes: latency and launches
        _case("answer", "small_bf16", 3, 32, 48, steps=8, name="answer_small_bf16"),
        _case("answer", "tiny", 2, 16, 32, steps=8, name="answer_tiny_fp32"),
        # the projection primitive: odd row count, four layers' q / k / v, output and down projections
        _case("project", "7b", 4, 37, 0, name="project_7b"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the same ranges: any kind, odd sizes, fewer layers where the pass would otherwise be the largest."""
    kind = rng.choice(["decode", "decode", "calls", "answer", "answer", "prefill", "project"])
    if kind == "project":
        return _case("project", rng.choice(["7b", "13b"]), rng.randint(2, 4), rng.randint(1, 64), 0)
    model = rng.choice(["tiny", "small_bf16", "7b", "7b", "13b", "33b"])
    small = model in ("tiny", "small_bf16")
    layers = LAYERS[model] if small else _log_int(rng, 2, 32 if model == "7b" else 16)
    nodes = rng.randint(5, 24 if model == "tiny" else 60) if small else _log_int(rng, 16, 128)
    temperature = rng.choice([0.0, 0.0, 0.7])
    rank = 256 if not small and rng.random() < 0.2 else 0
    if kind == "prefill":
        return _case(kind, model, layers, nodes, _log_int(rng, 8, 400) if small else _log_int(rng, 20, 1900), rank=rank,
                     temperature=temperature)
    if kind == "answer":
        batch = rng.randint(1, 8)
        while batch * ((max(nodes, 16) + 15) // 16 * 16) > 512:
            batch -= 1
        return _case(kind, model, layers, nodes, _log_int(rng, 8, 300), batch=batch, steps=rng.randint(4, 8), rank=rank,
                     temperature=temperature)
    ctx = _log_int(rng, 16, 400) if small else _log_int(rng, 256, 7900 if layers <= 16 else 3000)
    return _case(kind, model, layers, nodes, ctx, steps=rng.randint(3, 8), rank=rank, temperature=temperature)


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
def _shape(case):
    d, heads, dh, ffn, vocab, dtype, topk = WIDTHS[case["model"]]
    return SimpleNamespace(name=case["model"], n_layers=case["layers"], d_model=d, n_heads=heads, head_dim=dh, d_ffn=ffn,
                           vocab=vocab, dtype=dtype, K=K, n_sal=N_SAL, aeb_layers=1, lm_rank=case["rank"],
                           use_sampled_token=True, topk=topk, n_nodes=case["nodes"], rms_eps=1e-6, rope_theta=10000.0)


def _tree(nodes, widths):
    """The `nodes` best root-to-node paths when rank r of head k is right with probability 0.8 * 0.85^k * 2^-r / 2."""
    paths, level = [], [((), 1.0)]
    for k in range(K):
        level = [(p + (r,), s * 0.8 * 0.85 ** k * 0.5 ** (r + 1)) for p, s in level for r in range(widths[k])]
        level = sorted(level, key=lambda e: (-e[1], e[0]))[:nodes]
        paths += level
    paths = sorted(paths, key=lambda e: (-e[1], len(e[0]), e[0]))[: nodes - 1]
    paths = sorted((p for p, _ in paths), key=lambda p: (len(p), p))
    index = {(): 0, **{p: i + 1 for i, p in enumerate(paths)}}
    return SimpleNamespace(n_nodes=len(index), parent=[-1] + [index[p[:-1]] for p in paths],
                           depth=[0] + [len(p) for p in paths], rank=[0] + [p[-1] for p in paths])


def _weights(sh, gen):
    """Random weights that decode as trained ones do: a confident next token, and drafts that are often but not always right.

    The residual stream keeps the token's embedding (every linear map is N(0, 1 / fan_in), the ones that write to the
    residual stream damped by the depth, as models are initialised for training); the target's vocabulary head carries
    the embedding of each token's predecessor in a random cyclic order, so the next token has a clear margin over the rest of
    the vocabulary.  Drafting head k carries the k-th predecessor: its best candidate is right for about 3 tokens in 4 at
    depth 1 and half of them at depth 4, the second candidate for half of the rest, else it is wrong."""
    dt = torch.float32 if sh.dtype == "fp32" else torch.bfloat16
    d, F, V = sh.d_model, sh.d_ffn, sh.vocab

    def normal(*shape, std):
        return torch.empty(shape, dtype=dt, device=DEVICE).normal_(0.0, std, generator=gen)

    w = {"tok_emb": normal(V, d, std=1.0)}

    def layer(pre, depth):
        out = 1.0 / math.sqrt(2 * depth)
        for n in ("attn_norm", "ffn_norm"):
            w[pre + n] = (1.0 + normal(d, std=0.05))
        for n in ("wq", "wk", "wv"):
            w[pre + n] = normal(d, d, std=d ** -0.5)
        w[pre + "wo"] = normal(d, d, std=out * d ** -0.5)
        w[pre + "w_gate"] = normal(F, d, std=d ** -0.5)
        w[pre + "w_up"] = normal(F, d, std=d ** -0.5)
        w[pre + "w_down"] = normal(d, F, std=out * F ** -0.5)

    for i in range(sh.n_layers):
        layer(f"layers.{i}.", sh.n_layers)
    w["final_norm"] = 1.0 + normal(d, std=0.05)
    order = torch.randperm(V, generator=gen, device=DEVICE)              # token order[i] is followed by order[i + 1]
    place = torch.empty_like(order)
    place[order] = torch.arange(V, device=DEVICE)

    def before(k):                                                        # the token k places before each token
        return order[(place - k) % V]

    w["lm_head"] = w["tok_emb"][before(1)] * d ** -0.5
    for s in range(1, sh.n_sal + 1):
        fc = normal(d, 2 * d, std=(2 * d) ** -0.5)
        fc[:, d:] += torch.eye(d, dtype=dt, device=DEVICE)
        w[f"draft.fc{s}"] = fc
        layer(f"draft.sal{s}.", sh.n_sal)
    for k in range(K):
        w[f"draft.mlp.{k}.w"] = normal(d, d, std=d ** -0.5)
        w[f"draft.mlp.{k}.b"] = normal(d, std=0.5)
    w["draft.pe"] = normal(K, d, std=0.5)
    for n in ("wq", "wk", "wv", "wo"):
        w[f"draft.aeb.0.{n}"] = normal(d, d, std=d ** -0.5)
    for k in range(K):
        head = w["tok_emb"][before(k + 1)] * d ** -0.5
        lot = torch.rand(V, generator=gen, device=DEVICE)
        right = (0.75, 0.65, 0.55, 0.5)[k]
        second = torch.nonzero((lot >= right) & (lot < right + (1 - right) / 2)).flatten()
        wrong = torch.nonzero(lot >= right + (1 - right) / 2).flatten()
        other = torch.randperm(V, generator=gen, device=DEVICE)[: second.numel()]
        head[other] += head[second] * 1.25                                # another token comes first
        head[wrong] = normal(wrong.numel(), d, std=d ** -0.5)
        if sh.lm_rank:
            a = normal(sh.lm_rank, d, std=d ** -0.5)
            w[f"draft.lm_head.{k}.a"] = a
            w[f"draft.lm_head.{k}.b"] = ((head.float() @ a.float().T) * (d / sh.lm_rank)).to(dt)
        else:
            w[f"draft.lm_head.{k}"] = head
    return w


def _prompts(case, vocab, gen):
    """Token ids; the sequences of a batch are of different lengths, the first one the longest."""
    n = case["ctx"]
    lens = [max(1, n - (b * n * 5) // 43) for b in range(case["batch"])]
    return [torch.randint(0, vocab, (m,), generator=gen, device=DEVICE).tolist() for m in lens]


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    if case["kind"] == "project":
        d, _, _, F, _, _, _ = WIDTHS[case["model"]]
        rows, cap = case["nodes"], (case["nodes"] + 15) // 16 * 16
        calls = []
        for _ in range(case["layers"]):
            for n_seg, out, inner in ((3, d, d), (1, d, d), (1, d, F)):
                x = torch.empty(cap, inner, dtype=torch.bfloat16, device=DEVICE).normal_(0.0, 1.0, generator=gen)
                ws = [torch.empty(out, inner, dtype=torch.bfloat16, device=DEVICE).normal_(0.0, inner ** -0.5, generator=gen)
                      for _ in range(n_seg)]
                calls.append((x, ws, torch.empty(rows, n_seg * out, device=DEVICE)))
        return SimpleNamespace(case=case, calls=calls, status=torch.zeros(1, dtype=torch.int32, device=DEVICE))
    sh = _shape(case)
    B, n = case["batch"], case["steps"]
    tree = _tree(case["nodes"], sh.topk)
    cap = (case["ctx"] + n * (K + 1) + tree.n_nodes + 127) // 128 * 128
    model = Amphista(sh, tree, _weights(sh, gen), device=DEVICE, max_ctx=cap, max_batch=B, temperature=case["temperature"],
                     seed=seed)
    s = SimpleNamespace(case=case, shape=sh, tree=tree, model=model, prompts=_prompts(case, sh.vocab, gen))
    s.tokens = torch.zeros(max(n, 1), B, K + 1, dtype=torch.int32, device=DEVICE)
    s.counts = torch.zeros(max(n, 1), B, dtype=torch.int32, device=DEVICE)
    if case["kind"] in ("decode", "calls"):
        # the prompt is in the cache; its last row is what the first draft reads
        s.root = model.prefill(s.prompts[0])
        rows = (case["ctx"] - 1) % 512 + 1
        s.pending = model.get_tensor("hidden", (rows, sh.d_model))[-1:].clone()
    if case["kind"] == "calls":
        s.tokens, s.counts = s.tokens.cpu().pin_memory(), s.counts.cpu().pin_memory()
        s.path = torch.zeros(n, K + 1, dtype=torch.int32).pin_memory()
        s.next_root = torch.zeros(n, dtype=torch.int32).pin_memory()
        s.keep = torch.full((tree.n_nodes,), -1, dtype=torch.int32).pin_memory()      # every drafted token stays
    return s


# ---------------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------------
def run(s):
    case = s.case
    if case["kind"] == "project":
        for x, ws, y in s.calls:
            project_noalloc(x, ws, case["nodes"], True, y, s.status)
        return [y for _, _, y in s.calls]
    m, sh, B = s.model, s.shape, case["batch"]
    if case["kind"] == "prefill":
        root, n = m.prefill(s.prompts[0]), case["ctx"]
        rows, last = (n - 1) % 512 + 1, sh.n_layers - 1
        out = {"root": root, "hidden": m.get_tensor("hidden", (rows, sh.d_model)), "logits": m.get_tensor("logits", (rows, sh.vocab)),
               "k": m.get_tensor(f"kv.k.{last}", (n, sh.d_model)), "v": m.get_tensor(f"kv.v.{last}", (n, sh.d_model))}
        if n > 1:
            out["sal_k"], out["sal_v"] = (m.get_tensor(f"sal{N_SAL}.{c}", (n - 1, sh.d_model)) for c in "kv")
        return out
    roots = []
    if case["kind"] == "answer":
        roots = [m.prefill(p, seq=b) for b, p in enumerate(s.prompts)]
    else:
        m.set_state(case["ctx"], s.root, s.pending, [s.root])             # back to the end of the prompt
    for i in range(case["steps"]):
        if case["kind"] == "calls":
            m.draft()
            m.verify_tree(s.keep)
            m.accept(s.tokens[i], s.counts[i], s.path[i], s.next_root[i])
            m.synchronize()
        else:
            m.step(s.tokens[i], s.counts[i])
    out = {"roots": roots, "tokens": s.tokens, "counts": s.counts}
    if case["kind"] == "calls":
        out["path"], out["next_root"] = s.path, s.next_root
    # Per sequence: the last step's logits (the target's after the tree's root, all drafting heads'), and the last layer's
    # keys and values of the prompt and of at least one token per step.  The other tree rows belong to speculated tokens of low
    # rank: which of two nearly equal candidates takes such a place is a matter of rounding, so their logits are not results.
    for b, p in enumerate(s.prompts):
        rows, last = len(p) + case["steps"], sh.n_layers - 1
        out[f"logits{b}"] = m.get_tensor(f"logits#{b}", (1, sh.vocab))
        out[f"draft{b}"] = m.get_tensor(f"d_logits#{b}", (K, sh.vocab))
        out[f"k{b}"] = m.get_tensor(f"kv.k.{last}#{b}", (rows, sh.d_model))
        out[f"v{b}"] = m.get_tensor(f"kv.v.{last}#{b}", (rows, sh.d_model))
    return out


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct implementations may be apart
# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    d, _, _, F, V, dtype, _ = WIDTHS[case["model"]]
    esz = 4 if dtype == "fp32" else 2
    L, N, B, S, r = case["layers"], case["nodes"], case["batch"], case["steps"], case["rank"]
    if case["kind"] == "project":
        w = L * (3 * d * d + d * d + d * F)
        acts = L * N * (2 * d + F)
        return {"bytes": 2.0 * (w + acts) + 4.0 * L * N * 5 * d, "flops": 2.0 * w * N}
    layer = 4 * d * d + 3 * d * F
    target, sal = L * layer, N_SAL * (layer + 2 * d * d)
    heads_w = K * (d * d + d) + 4 * d * d + K * (r * (d + V) if r else V * d)
    head = V * d
    lens = [max(1, case["ctx"] - (b * case["ctx"] * 5) // 43) for b in range(B)]
    bytes_, flops = 0.0, 0.0
    if case["kind"] in ("prefill", "answer"):
        for n in lens:                            # every weight once per prompt, the keys and values written once
            bytes_ += esz * (target + sal + head + 2 * n * d * (L + N_SAL))
            flops += 2.0 * n * (target + sal) + 2.0 * head + 2.0 * n * n * d * (L + N_SAL)
        if case["kind"] == "prefill":
            rows = (case["ctx"] - 1) % 512 + 1    # hidden rows and logits of the last pass are results
            bytes_ += 4.0 * rows * (d + V) + 4.0 * 4 * case["ctx"] * d
            flops += 2.0 * head * (rows - 1)
    for i in range(S):                            # about 2.5 tokens are accepted per step
        live = sum(n + 2.5 * i + N for n in lens)
        bytes_ += esz * (target + sal + heads_w + head + 2 * live * d * (L + N_SAL)) + 4.0 * B * (N + K) * V
        flops += 2.0 * B * (N * (target + head) + 2.5 * sal + K * d * V) + 4.0 * N * live * d * L
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times what was measured: the projection against 64-bit sums 2.1e-6 (largest difference 8e-6); bf16 models,
    the fused kernels against the separate ones (sums in another order, other places of rounding to bf16): logits 2.2e-3,
    drafting logits 4.5e-3, keys and values 3.2e-3 (largest differences 3e-2); 32-bit models against 64 bits 3e-7.  The
    vocabulary heads' margins (see _weights) are far beyond these, so tokens and counts do not move."""
    if case["kind"] == "project":
        return {"rel": 1e-5, "max": 4e-5}
    if WIDTHS[case["model"]][5] == "fp32":
        return {"rel": 4e-6, "max": 4e-5}
    return {"rel": 1.8e-2, "max": 0.12}
