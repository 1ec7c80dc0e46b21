"""The number of KV splits per head falls as a launch carries more row blocks.  Sequences decoded side by side (1 to 7 splits,
depending on how many there are) must agree with each decoded alone in a context of its own (one per 128 keys, up to 7)."""
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,dh,nodes,batch", [(16, 64, 64, 8), (16, 64, 100, 4), (8, 128, 33, 5), (8, 128, 128, 4), (8, 128, 64, 1)])
def test_side_by_side_equals_alone(heads, dh, nodes, batch):
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16").with_(d_model=heads * dh, n_heads=heads, head_dim=dh, n_layers=2, n_nodes=nodes, topk=(16, 16, 16, 16))
    topo = inputs.make_tree(nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    lens = [900, 64, 127, 513, 700, 1, 640, 300][:batch]
    prompts = [inputs.make_prompt(shape.with_(prompt_len=n), seed=5 + i).tolist() for i, n in enumerate(lens)]
    many = Amphista(shape, topo, w, max_batch=batch, max_ctx=1152)
    one = Amphista(shape, topo, w, max_ctx=1152, flags=128)              # prompts in single chunks of 128 rows
    for b, p in enumerate(prompts):
        many.prefill(p, seq=b)
    many.draft()
    N, V, d = topo.n_nodes, shape.vocab, shape.d_model
    toks = torch.randint(0, V, (batch, N), dtype=torch.int32, generator=torch.Generator().manual_seed(1)).cuda()
    many.verify_tree(toks)
    many.synchronize()
    for b, p in enumerate(prompts):
        one.reset()
        one.prefill(p)
        root = torch.tensor([many.get_state(b)[1]], dtype=torch.int32, device="cuda:0")
        one.set_tensor("root", root)                                     # the greedy choice may hang on a near tie
        one.draft()
        one.verify_tree(toks[b])
        one.synchronize()
        for name, size in (("logits", (N, V)), ("d_logits", (shape.K, V)), ("kv.v.1", (lens[b] + N, d))):
            x, y = many.get_tensor(f"{name}#{b}", size), one.get_tensor(name, size)
            assert float((x - y).norm() / y.norm()) <= 1e-2, (name, b)   # two bf16 layers; sums in another order (2^-8 per rounding)
    many.close()
    one.close()
