"""amph_step keeps a bounded set of captured schedules, one per combination of attention grids.  Lengths that come back must
find the right one, more combinations than are kept must still be right, and so must every sequence length a kept schedule is
replayed at: the emitted tokens equal those of a context that launches its kernels one by one (bit for bit the same kernels)."""
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu


def _decode(model, prompts, steps):
    tok = torch.zeros(model.B, model.shape.K + 1, dtype=torch.int32, device="cuda:0")
    n = torch.zeros(model.B, dtype=torch.int32, device="cuda:0")
    out = [model.prefill(p, seq=b) for b, p in enumerate(prompts)]
    for _ in range(steps):
        model.step(tok, n)
        torch.cuda.synchronize()
        out += tok.flatten().tolist() + n.tolist()
    return out


# fp32 caches: every sequence's own split count is part of the combination, 25 of them for two sequences (more than are kept);
# bf16 caches: one launch sized for the longest sequence
@pytest.mark.parametrize("name,lengths", [("tiny", (20, 150, 280, 410, 540)), ("small_bf16", (60, 300, 700))])
def test_lengths_that_come_back(name, lengths):
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape(name)
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    texts = {n: inputs.make_prompt(shape.with_(prompt_len=n), seed=n).tolist() for n in lengths}
    graphs = Amphista(shape, topo, w, max_batch=2, max_ctx=1024)
    plain = Amphista(shape, topo, w, max_batch=2, max_ctx=1024, flags=2)
    pairs = [(a, b) for a in lengths for b in lengths]
    for a, b in pairs + pairs[:3] + pairs[-2:]:
        prompts = [texts[a], texts[b]]
        assert _decode(graphs, prompts, 2) == _decode(plain, prompts, 2), (a, b)
    graphs.close()
    plain.close()


def test_eight_sequences_of_different_lengths():
    """Eight sequences with a split count each: combinations that differ in one of them only are different schedules."""
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("tiny")
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    texts = {n: inputs.make_prompt(shape.with_(prompt_len=n), seed=n).tolist() for n in (20, 150, 280)}
    graphs = Amphista(shape, topo, w, max_batch=8, max_ctx=512)
    plain = Amphista(shape, topo, w, max_batch=8, max_ctx=512, flags=2)
    for longer in (None, 0, 7, 3, 0, None):
        prompts = [texts[280 if b == longer else 150 if b % 2 else 20] for b in range(8)]
        assert _decode(graphs, prompts, 2) == _decode(plain, prompts, 2), longer
    graphs.close()
    plain.close()


def test_context_grows_past_the_prefetch_helper():
    """20 MB of keys and values per layer: below, a step's schedule has a prefetch helper per layer, above, none; first the
    verification pass crosses the line, then the draft."""
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16")
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    n = (20 << 20) // (4 * shape.d_model) - shape.n_nodes - 12
    prompt = inputs.make_prompt(shape.with_(prompt_len=n), seed=1).tolist()
    outs = []
    for flags in (0, 2):                              # 2: kernels launched one by one
        m = Amphista(shape, topo, w, max_ctx=n + 256, flags=flags)
        outs.append(_decode(m, [prompt], 14))
        m.close()
    assert outs[0] == outs[1]


@pytest.mark.parametrize("batch", [1, 3])
def test_results_reach_whatever_arrays_a_step_is_given(batch):
    """Device arrays, other device arrays, pinned and pageable host arrays, one of the two, none: each call's results arrive where
    that call asked for them, and nowhere else."""
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16")
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompts = [inputs.make_prompt(shape.with_(prompt_len=n), seed=n).tolist() for n in (40, 130, 17)[:batch]]
    K = shape.K
    make = {"device": lambda s: torch.full(s, -7, dtype=torch.int32, device="cuda:0"),
            "pinned": lambda s: torch.full(s, -7, dtype=torch.int32).pin_memory(), "pageable": lambda s: torch.full(s, -7, dtype=torch.int32),
            "none": lambda s: None}
    kinds = [("device", "device"), ("device", "device"), ("pinned", "pinned"), ("device", "pinned"), ("none", "none"), ("device", "none"),
             ("pageable", "device"), ("none", "device"), ("device", "device")]

    def run(flags):
        m = Amphista(shape, topo, w, max_batch=batch, max_ctx=512, flags=flags)
        for b, p in enumerate(prompts):
            m.prefill(p, seq=b)
        outs = []
        for kt, kn in kinds:
            t, n = make[kt]((batch, K + 1)), make[kn]((batch,))
            m.step(t, n)
            m.synchronize()
            outs.append((t, n))
        torch.cuda.synchronize()
        m.close()
        return [(None if t is None else t.tolist(), None if n is None else n.tolist()) for t, n in outs]

    assert run(0) == run(2)                       # 2: kernels launched one by one, results copied


@pytest.mark.parametrize("batch", [1, 3])
def test_results_reach_arrays_at_any_byte(batch):
    """Device arrays that do not start at a multiple of four bytes: results arrive by copy."""
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16")
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    K = shape.K
    outs = []
    for shifts in (((0, 0), (0, 0), (0, 0), (0, 0)), ((1, 0), (0, 2), (3, 1), (0, 0))):
        m = Amphista(shape, topo, w, max_batch=batch, max_ctx=512)
        for b in range(batch):
            m.prefill(inputs.make_prompt(shape, seed=b).tolist(), seq=b)
        got = []
        for st, sn in shifts:
            t = torch.zeros(4 * batch * (K + 1) + 4, dtype=torch.uint8, device="cuda:0")
            n = torch.zeros(4 * batch + 4, dtype=torch.uint8, device="cuda:0")
            m.step(t[st:], n[sn:])
            m.synchronize()
            got.append((t[st:].cpu()[:4 * batch * (K + 1)].clone().view(torch.int32).tolist(), n[sn:].cpu()[:4 * batch].clone().view(torch.int32).tolist()))
        m.close()
        outs.append(got)
    assert outs[0] == outs[1]
    assert all(1 <= c <= K + 1 for _, n in outs[0] for c in n)


def test_helper_launches_follow_the_context():
    """The schedule that a step replays has a helper for every layer of a pass that may read at most 20 MB of keys and values per
    layer, and none for the others: counted from the kernels that ran, with lengths that come back."""
    from paper_2406_13170_b200 import Amphista
    from torch.profiler import ProfilerActivity, profile
    shape = inputs.get_shape("small_bf16")
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    limit, N = (20 << 20) // (4 * shape.d_model), shape.n_nodes
    m = Amphista(shape, topo, w, max_ctx=limit + N + 64)
    root = m.prefill(inputs.make_prompt(shape.with_(prompt_len=limit + 1), seed=1).tolist())
    pending = torch.ones(1, shape.d_model)
    both, draft, none = shape.n_sal + shape.n_layers, shape.n_sal, 0
    for n, want in ((limit - N, both), (limit - N + 1, draft), (limit, draft), (limit + 1, none), (limit - N, both), (limit, draft)):
        m.set_state(n, root, pending, [root])
        m.step()                                  # captures the schedule, or finds it
        m.set_state(n, root, pending, [root])
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            m.step()
            torch.cuda.synchronize()
        names = [e.key for e in prof.key_averages() for _ in range(e.count)]
        if not any("accept_compact_kernel" in k for k in names):
            pytest.skip("the profiler records no kernels here")
        assert sum("tc_prefetch_pair_kernel" in k for k in names) == want, n
    m.close()
