"""The projections that finish their rows themselves in passes of up to 64 rows (gate / up with SwiGLU, q / k / v with rotary embedding
and cache write, output and down projection with the residual update) against the separate kernels, at the edges of their tiles:
rows around multiples of 16, a last tile that is not whole, one tile height per head dimension; bf16 and fp32."""
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu


def _outputs(shape, w, prompts, flags):
    from paper_2406_13170_b200 import Amphista
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    m = Amphista(shape, topo, w, max_ctx=max(256, max(map(len, prompts)) + shape.n_nodes + 8), max_batch=len(prompts), flags=flags)
    toks = torch.randint(0, shape.vocab, (len(prompts), shape.n_nodes), dtype=torch.int32, generator=torch.Generator().manual_seed(3)).cuda()
    out = []
    for b, p in enumerate(prompts):
        m.prefill(p, seq=b)
        out.append(m.get_tensor("hidden", (len(p), shape.d_model)))
    for b in range(len(prompts)):
        m.set_tensor("root" if b == 0 else f"root#{b}", toks[b, :1].contiguous())
    m.draft()
    m.verify_tree(toks if len(prompts) > 1 else toks[0])
    m.synchronize()
    last = shape.n_layers - 1
    for b, p in enumerate(prompts):
        out.append(m.get_tensor(f"hidden#{b}", (shape.n_nodes, shape.d_model)))
        out.append(m.get_tensor(f"sal_h#{b}", (2, shape.d_model)))
        out += [m.get_tensor(f"kv.{c}.{i}#{b}", (len(p) + shape.n_nodes, shape.d_model)) for c in "kv" for i in (0, last)]
    m.close()
    return out


def _compare(a, b, rel):
    for x, y in zip(a, b):
        assert bool(torch.isfinite(x).all())
        assert float((x - y).norm() / y.norm()) <= rel
        # a tile that went wrong may be a fraction of a per cent of a tensor's norm: twice the bound for every element, in units of the
        # largest one (the pair projection's tests)
        assert float((x - y).abs().max()) <= 2 * rel * max(1.0, float(y.abs().max()))


# 11008 = 137 tiles of 80 and one of 48 (rows above 16), 2432 = 101 of 24 and one of 8; width 2176: no residual form; widths 576 and 320:
# an odd number of K blocks, the last stage of two has one that does not exist
@pytest.mark.parametrize("heads,dh,ffn", [(8, 64, 1408), (4, 128, 2432), (10, 128, 3456), (4, 128, 11008), (17, 128, 1408), (9, 64, 1152),
                                          (5, 64, 1408)])
@pytest.mark.parametrize("n,nodes", [(1, 5), (16, 16), (17, 33), (48, 43), (63, 50), (64, 64)])
def test_bf16_forms_against_the_separate_kernels(heads, dh, ffn, n, nodes):
    shape = inputs.get_shape("small_bf16").with_(d_model=heads * dh, n_heads=heads, head_dim=dh, d_ffn=ffn, n_nodes=nodes, topk=(16, 16, 16, 16))
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompts = [inputs.make_prompt(shape.with_(prompt_len=n), seed=2).tolist()]
    # 512: no residual update in an epilogue.  Sums in another order, roundings to bf16 (2^-8) in the same places; three layers of
    # unit gain, as in the tests of the projection of many rows
    _compare(_outputs(shape, w, prompts, 0), _outputs(shape, w, prompts, 4 | 16 | 512), 1e-2)


@pytest.mark.parametrize("n_nodes", [16, 43, 64, 100])
def test_up_matrix_below_the_gate_matrix(n_nodes):
    """Gate and up come through one tensor map that begins at the lower of the two: the same bits whichever that is."""
    shape = inputs.get_shape("small_bf16").with_(n_nodes=n_nodes, topk=(16, 16, 16, 16))
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompts = [inputs.make_prompt(shape, seed=2).tolist()]
    outs = []
    for first, second in (("w_gate", "w_up"), ("w_up", "w_gate")):
        v = dict(w)
        for name in [k for k in w if k.endswith("w_gate")]:
            pre = name[: -len("w_gate")]
            both = torch.empty(2, *w[name].shape, dtype=w[name].dtype, device="cuda:0")
            both[0].copy_(w[pre + first])
            both[1].copy_(w[pre + second])
            v[pre + first], v[pre + second] = both[0], both[1]
        outs.append(_outputs(shape, v, prompts, 0))
    assert all(torch.equal(a, b) for a, b in zip(*outs))


# two accumulators (the sums of two K ranges, 512 and 1280 wide), and shapes that decline (more K ranges, an odd number of K blocks)
@pytest.mark.parametrize("heads,dh,ffn", [(8, 64, 1408), (4, 128, 11008), (10, 128, 3456), (17, 128, 1408), (9, 64, 1152)])
@pytest.mark.parametrize("nodes", [65, 80, 113, 128])
def test_one_order_of_sums_above_64_rows(heads, dh, ffn, nodes):
    shape = inputs.get_shape("small_bf16").with_(d_model=heads * dh, n_heads=heads, head_dim=dh, d_ffn=ffn, n_nodes=nodes, topk=(16, 16, 16, 16),
                                                 lm_rank=24)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompts = [inputs.make_prompt(shape.with_(prompt_len=100), seed=2).tolist()]
    # the same sums in the same order, the same exponential and division: bit for bit (the adaptation layers' pass of 16 rows, which
    # feeds output 2 only, has the fast exponential in one of them)
    for i, (a, b) in enumerate(zip(_outputs(shape, w, prompts, 0), _outputs(shape, w, prompts, 4 | 16))):
        assert i == 2 or torch.equal(a, b)


# the residual form's rule is 296 blocks of 8 features x 16 rows: at width 256 up to 144 rows of a pass take it, at width 1024 32
@pytest.mark.parametrize("heads,dh,ffn", [(4, 64, 688), (3, 128, 1000), (1, 64, 8), (8, 128, 2824)])
@pytest.mark.parametrize("lens,nodes", [((1,), 5), ((17,), 16), ((33,), 24), ((40, 7, 21), 19), ((144, 160, 5), 40), ((300, 3, 150, 9), 40)])
def test_fp32_forms_against_the_separate_kernels(heads, dh, ffn, lens, nodes):
    shape = inputs.get_shape("tiny").with_(d_model=heads * dh, n_heads=heads, head_dim=dh, d_ffn=ffn, n_nodes=nodes, topk=(8, 8, 8, 8))
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    prompts = [inputs.make_prompt(shape.with_(prompt_len=n), seed=b).tolist() for b, n in enumerate(lens)]
    # 512: the residual update too is a kernel of its own.  The same fp32 sums; squares are added in another order and the last operations
    # may be contracted differently (a few ulps of 2^-24 per layer)
    _compare(_outputs(shape, w, prompts, 0), _outputs(shape, w, prompts, 4 | 16 | 512), 4e-6)
