"""A context is reused for several sequences, and the path is deterministic: the same inputs give bit-identical
tokens, logits and cache rows from run to run, with the CUDA-graph replay of amph_step and with its kernels launched
one by one (split-K partial sums are always added in a fixed order; there are no floating-point atomics)."""
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu


def _run(model, shape, prompt, steps, use_step):
    K, V, d = shape.K, shape.vocab, shape.d_model
    root = model.prefill(prompt)
    out_tok = torch.zeros(K + 1, dtype=torch.int32, device="cuda:0")
    out_n = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    toks = [root]
    for _ in range(steps):
        if use_step:
            model.step(out_tok, out_n)
        else:
            model.draft()
            model.verify_tree()
            model.accept(out_tok, out_n)
        torch.cuda.synchronize()
        toks += out_tok[: int(out_n[0])].tolist()
    C, root, _ = model.get_state()
    kv = model.get_tensor("kv.k.0", (C, d)).clone()
    dl = model.get_tensor("d_logits", (K, V)).clone()
    return toks, C, root, kv, dl


@pytest.mark.parametrize("name", ["tiny", "small_bf16"])
def test_reuse_and_bitwise_determinism(name):
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape(name)
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0")
    p1 = inputs.make_prompt(shape).tolist()
    p2 = [(t * 7 + 3) % shape.vocab for t in p1[: len(p1) // 2]]
    m = Amphista(shape, topo, w)
    a = _run(m, shape, p1, 4, use_step=True)
    b = _run(m, shape, p2, 3, use_step=True)          # a second sequence in the same context (prefill resets it)
    m.reset()
    c = _run(m, shape, p1, 4, use_step=True)          # the first one again, after an explicit reset
    assert a[0] == c[0] and a[1:3] == c[1:3]
    assert torch.equal(a[3], c[3]) and torch.equal(a[4], c[4])
    assert b[0] != a[0]
    m.close()
    # kernels launched one by one (no graph), phases called separately: same bits
    m2 = Amphista(shape, topo, w, flags=2)
    e = _run(m2, shape, p1, 4, use_step=False)
    assert e[0] == a[0] and e[1:3] == a[1:3]
    assert torch.equal(e[3], a[3]) and torch.equal(e[4], a[4])
    m2.close()


def test_a_tap_is_not_overwritten_by_what_torch_has_queued():
    """get_tensor's result may sit in a block of torch's pool that kernels queued on torch's stream still write."""
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16")
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    m = Amphista(shape, topo, inputs.make_weights(shape, seed=0, device="cuda:0"))
    n = 48
    m.prefill(inputs.make_prompt(shape.with_(prompt_len=n)).tolist())
    want = m.get_tensor("logits", (n, shape.vocab)).clone()
    for cycles in (1, 100_000_000):                    # the second time about 50 ms (the first one loads the kernels)
        torch.cuda.synchronize()
        busy = torch.empty(n, shape.vocab, device="cuda:0")
        torch.cuda._sleep(cycles)
        busy.fill_(7.0)
        block = busy.data_ptr()
        del busy
        got = m.get_tensor("logits", (n, shape.vocab))
        assert got.data_ptr() == block
        torch.cuda.synchronize()
        assert torch.equal(got, want)
        del got
    m.close()


def test_two_contexts_on_two_streams_at_once():
    """Every projection and attention CTA takes tensor memory, several kernels of a context are resident at a time, and two contexts
    share the SMs: each gives what it gives alone.  (Passes of up to 64 rows, of more, and prompts of both.)"""
    from paper_2406_13170_b200 import Amphista
    steps = 12

    def build(n_nodes, n, heads):
        shape = inputs.get_shape("small_bf16").with_(d_model=heads * 128, n_heads=heads, n_nodes=n_nodes, topk=(16, 16, 16, 16), prompt_len=n)
        w = inputs.make_weights(shape, seed=n, device="cuda:0", init="fan_in")
        m = Amphista(shape, inputs.make_tree(n_nodes, shape.topk), w, max_ctx=n + steps * (shape.K + 1) + n_nodes + 8)
        out = torch.zeros(steps, shape.K + 2, dtype=torch.int32, device="cuda:0")
        return m, shape, inputs.make_prompt(shape).tolist(), out

    def enqueue(c, i):
        c[0].step(c[3][i, : c[1].K + 1], c[3][i, c[1].K + 1 :])

    def results(c):
        c[0].synchronize()
        return [c[3].clone(), c[0].get_tensor("logits", (c[1].n_nodes, c[1].vocab)), c[0].get_tensor("kv.k.2", (c[0].get_state()[0], c[1].d_model))]

    pair = [build(64, 300, 4), build(100, 50, 8)]
    torch.cuda.synchronize()
    alone = []
    for c in pair:
        c[0].prefill(c[2])
        for i in range(steps):
            enqueue(c, i)
        alone.append(results(c))
    for c in pair:
        c[0].prefill(c[2])
    for i in range(steps):
        for c in pair:
            enqueue(c, i)
    for c, want in zip(pair, alone):
        for a, b in zip(results(c), want):
            assert torch.equal(a, b)
        c[0].close()
