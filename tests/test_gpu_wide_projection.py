"""The CTA-pair projection (many activation rows) at the edges of its tiles: rows around multiples of 32 and of the 256 rows of
one MMA, weight counts that cut tiles over several pairs, K that is not a whole number of work units; and the fused gate / up
and q / k / v forms inside a prefill against the separate kernels."""
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [65, 96, 97, 128, 200, 256, 257, 300, 511, 512])
# stages of two K blocks up to 128 rows or K = 2816 (64, 192, 2816 and 2880: whole and half last stages), of one beyond
@pytest.mark.parametrize("n_seg,out,inner", [(1, 256, 64), (3, 512, 192), (2, 768, 1408), (1, 6656, 512), (1, 768, 2816), (1, 768, 2880),
                                             (2, 512, 4096)])
def test_plain_form_against_double(rows, n_seg, out, inner):
    from paper_2406_13170_b200 import project
    g = torch.Generator(device="cuda").manual_seed(rows * 7 + out)
    x = torch.randn(rows, inner, device="cuda", generator=g).to(torch.bfloat16)
    x = torch.cat([x, torch.zeros((-rows) % 128, inner, dtype=x.dtype, device="cuda")])
    ws = [(torch.randn(out, inner, device="cuda", generator=g) * inner ** -0.5).to(torch.bfloat16) for _ in range(n_seg)]
    y = project(x, ws, rows, True).double()
    x = x[:rows].double()
    want = torch.cat([x @ w.double().T for w in ws], 1)
    # products are exact in fp32; a sum of `inner` of them, in any order and even truncated at every addition, is off by at most
    # inner * 2^-23 times the sum of magnitudes
    bound = torch.cat([x.abs() @ w.double().abs().T for w in ws], 1) * inner * 2.0 ** -23
    assert bool(((y - want).abs() <= bound).all())


# head_dim 64 and 128; odd numbers of tiles; prompts whose passes carry one ragged group, several groups, and two passes
# (24 x 128: K above 2816, stages of one K block from 129 rows on)
@pytest.mark.parametrize("heads,dh,ffn", [(8, 64, 1408), (4, 128, 1408), (10, 128, 3456), (6, 128, 896), (24, 128, 3456)])
@pytest.mark.parametrize("n", [70, 128, 300, 513])
def test_fused_forms_against_the_separate_kernels(heads, dh, ffn, n):
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16").with_(d_model=heads * dh, n_heads=heads, head_dim=dh, d_ffn=ffn, prompt_len=n)
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompt = inputs.make_prompt(shape, seed=2).tolist()
    outs = []
    for flags in (0, 4 | 16, 1):                  # 1: the plain kernels, the residual update apart
        m = Amphista(shape, topo, w, max_ctx=1024, flags=flags)
        m.prefill(prompt)
        m.prefill(prompt)                         # the flags of cut tiles are lowered again after every launch
        last = shape.n_layers - 1
        outs.append([m.get_tensor("hidden", ((n - 1) % 512 + 1, shape.d_model))] +
                    [m.get_tensor(f"kv.{c}.{i}", (n, shape.d_model)) for c in "kv" for i in (0, last)])
        m.close()
    for a, b in list(zip(outs[0], outs[1])) + list(zip(outs[0], outs[2])):
        assert bool(torch.isfinite(a).all())
        # the two forms round the same fp32 sums to bf16 at the same places; a last-bit difference (2^-8) propagates through
        # three layers of unit gain, as in the parity tests' bound
        assert float((a - b).abs().max()) <= 2e-2 * max(1.0, float(b.abs().max()))
        assert float((a - b).norm() / b.norm()) <= 1e-2


# 384 = 3 * 128: the q / k / v and the residual form decline (they own 256 columns at a time), gate / up does not
@pytest.mark.parametrize("heads,dh,ffn", [(8, 64, 1408), (4, 128, 1408), (3, 128, 1408), (10, 128, 3456), (24, 128, 3456)])
@pytest.mark.parametrize("n", [70, 128, 300, 513])
def test_pair_projections_against_the_kernels_of_fewer_rows(heads, dh, ffn, n):
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16").with_(d_model=heads * dh, n_heads=heads, head_dim=dh, d_ffn=ffn, prompt_len=n, n_nodes=100,
                                                 topk=(16, 16, 16, 16))
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompt = inputs.make_prompt(shape, seed=2).tolist()
    toks = torch.randint(0, shape.vocab, (shape.n_nodes,), dtype=torch.int32, generator=torch.Generator().manual_seed(n)).cuda()
    outs = []
    for flags in (0, 512):                        # 512: no pair projection, and with it no residual update in an epilogue
        m = Amphista(shape, topo, w, max_ctx=1024, flags=flags)
        m.prefill(prompt)
        m.set_tensor("root", toks[:1])
        m.draft()
        m.verify_tree(toks)
        m.synchronize()
        outs.append([m.get_tensor("hidden", (shape.n_nodes, shape.d_model)), m.get_tensor("logits", (shape.n_nodes, shape.vocab))] +
                    [m.get_tensor(f"kv.{c}.{shape.n_layers - 1}", (n + shape.n_nodes, shape.d_model)) for c in "kv"])
        m.close()
    for a, b in zip(*outs):
        assert bool(torch.isfinite(a).all())
        assert float((a - b).norm() / b.norm()) <= 1e-2       # sums in another order, roundings to bf16 in the same places (see above)


@pytest.mark.parametrize("n", [70, 97, 128])
def test_residual_update_behind_the_same_sums(n):
    """At widths of 256 nothing is split along K, so both routes have the same sums, and with SwiGLU and the rotary embedding as
    kernels of their own on both sides what differs is the residual update: in the output and down projections' epilogues, or as a
    kernel of its own.  Both add 128 columns' squares in a warp, then the two parts: bit for bit the same."""
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16").with_(d_model=256, n_heads=4, head_dim=64, d_ffn=256, n_layers=4, prompt_len=n)
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompt = inputs.make_prompt(shape, seed=2).tolist()
    outs = []
    for flags in (4 | 16, 4 | 16 | 512):
        m = Amphista(shape, topo, w, max_ctx=512, flags=flags)
        m.prefill(prompt)
        outs.append(m.get_tensor("hidden", (n, shape.d_model)))
        m.close()
    assert torch.equal(outs[0], outs[1])
