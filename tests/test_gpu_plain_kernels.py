"""The CUDA-core projection and tree attention (fp32 models) where their tiles end: features that are not a multiple of a
block's, K below, at and beyond one step, row counts around 4 and 16, both storage types; contexts around multiples of the
64-key tile and of the 128 keys from which the KV axis is split."""
import pytest
import torch

import inputs
from oracle import amphista_oracle as ao

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows", [1, 4, 5, 16, 17, 130])
@pytest.mark.parametrize("n_seg,out,inner", [(1, 1, 8), (3, 9, 256), (8, 130, 264), (2, 1003, 520), (1, 5000, 128)])
def test_projection_against_double(dtype, rows, n_seg, out, inner):
    from paper_2406_13170_b200 import project
    g = torch.Generator(device="cuda").manual_seed(rows + out)
    x = torch.randn(rows, inner, device="cuda", generator=g).to(dtype)
    ws = [torch.randn(out, inner, device="cuda", generator=g).to(dtype) for _ in range(n_seg)]
    y = project(x, ws, rows, False).double()
    want = torch.cat([x.double() @ w.double().T for w in ws], 1)
    # every product and every addition rounds once: at most (inner + 1) * 2^-24 of the sum of magnitudes
    bound = torch.cat([x.double().abs() @ w.double().abs().T for w in ws], 1) * (inner + 1) * 2.0 ** -24
    assert bool(((y - want).abs() <= bound).all())


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows", [6, 8, 9])
@pytest.mark.parametrize("n_seg,out,inner", [(3, 9, 256), (8, 296, 264), (8, 297, 520), (1, 2369, 128)])
def test_blocks_of_eight_rows(dtype, rows, n_seg, out, inner):
    """Five to eight rows; 296 and 297 blocks of one feature per warp are the two sides of two features per warp."""
    test_projection_against_double(dtype, rows, n_seg, out, inner)


@pytest.mark.parametrize("heads,dh", [(4, 64), (2, 128)])
@pytest.mark.parametrize("n", [1, 15, 48, 63, 64, 65, 111, 113, 200, 400])
def test_tree_attention_inside_a_step(heads, dh, n):
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("tiny").with_(n_heads=heads, head_dim=dh, prompt_len=n, n_nodes=19, topk=(6, 4, 2, 1))
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    t = ao.tree_tables(topo.parent, topo.depth, topo.rank)
    w = inputs.make_weights(shape, seed=0, init="fan_in")
    m = Amphista(shape, topo, {k: v.to("cuda:0") for k, v in w.items()}, max_ctx=512)
    orc = ao.Oracle(shape, w, dtype=torch.float64)
    prompt = inputs.make_prompt(shape).tolist()
    st = orc.prefill(prompt)
    m.prefill(prompt)
    m.draft()
    m.verify_tree()
    m.synchronize()
    toks = m.get_tensor("tree_tokens", (t.n_nodes,), torch.int32).tolist()
    _, logits, _ = orc.verify(st, toks, t)
    got = m.get_tensor("logits", (t.n_nodes, shape.vocab)).cpu().double()
    assert float((got - logits).abs().max()) <= 1e-5 * max(1.0, float(logits.abs().max()))      # the parity tests' fp32 bound
    m.close()
