"""Contexts with low-rank drafting heads (Appendix A.2.4).  The candidates of such a head lie within a rounding of one another,
so the tree, and with it how a text is cut into steps, changes with the order of any sum in the passes before: their results are
pinned bit for bit (tokens, counts, tree tokens; CRC-32 of logits and caches), for passes below and above 64 rows, prompts of
several chunks and passes, several key ranges, batches.  The last tests compare such contexts with the oracle."""
import os
import zlib

import pytest
import torch

import inputs
from oracle import amphista_oracle as ao
from tests.parity import run_parity

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "low_rank_outputs.txt")

# name: (shape, changes to it, prompt lengths, steps)
CASES = {
    "tree128": ("small_bf16", dict(lm_rank=64, n_nodes=128, topk=(16, 16, 16, 16)), [300], 5),
    "dh64_three_passes": ("small_bf16", dict(n_heads=8, head_dim=64, lm_rank=24, n_nodes=100, topk=(16, 16, 16, 16)), [1300], 4),
    "batch": ("small_bf16", dict(lm_rank=32, n_nodes=48, topk=(10, 10, 10, 10)), [530, 70, 200], 4),
    "below_64_rows": ("small_bf16", dict(lm_rank=64, n_nodes=43), [60], 4),
    "tree128_7b_widths": ("7b_l2", dict(lm_rank=256, n_nodes=128), [700], 3),
}


def outputs(case):
    """One line of integers: everything that a context's user reads back."""
    from paper_2406_13170_b200 import Amphista
    name, change, lens, steps = CASES[case]
    shape = inputs.get_shape(name).with_(**change)
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    B, K, V, d = len(lens), shape.K, shape.vocab, shape.d_model
    m = Amphista(shape, topo, w, max_batch=B, max_ctx=max(lens) + steps * (K + 1) + shape.n_nodes + 8)
    out = [m.prefill(inputs.make_prompt(shape.with_(prompt_len=n), seed=n).tolist(), seq=b) for b, n in enumerate(lens)]
    tok = torch.zeros(B, K + 1, dtype=torch.int32, device="cuda:0")
    cnt = torch.zeros(B, dtype=torch.int32, device="cuda:0")
    crc = lambda t: zlib.crc32(t.cpu().numpy().tobytes())
    for _ in range(steps):
        m.step(tok, cnt)
        m.synchronize()
        out += tok.flatten().tolist() + cnt.tolist()
        for b in range(B):
            out.append(crc(m.get_tensor(f"tree_tokens#{b}", (shape.n_nodes,), torch.int32)))
            out.append(crc(m.get_tensor(f"d_logits#{b}", (K, V))))
            out.append(crc(m.get_tensor(f"logits#{b}", (shape.n_nodes, V))))
    for b in range(B):
        C = m.get_state(b)[0]
        out += [C, crc(m.get_tensor(f"kv.k.{shape.n_layers - 1}#{b}", (C, d))), crc(m.get_tensor(f"sal2.v#{b}", (lens[b] - 1, d)))]
    m.close()
    return out


@pytest.mark.parametrize("case", list(CASES))
def test_outputs_are_pinned(case):
    with open(GOLDEN) as f:
        want = dict(line.split(":") for line in f if ":" in line)
    assert outputs(case) == [int(v) for v in want[case].split()]


@pytest.mark.parametrize("rank", [24, 64])
def test_128_nodes_against_the_oracle(rank):
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape("small_bf16").with_(lm_rank=rank, n_nodes=128, topk=(16, 16, 16, 16), prompt_len=150)
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0)
    m = Amphista(shape, topo, {k: v.to("cuda:0") for k, v in w.items()}, max_ctx=512)
    rep = run_parity(m, ao.Oracle(shape, w, dtype=torch.float64), shape, topo, inputs.make_prompt(shape).tolist(), 4, 2e-2, 1e-3, True)
    m.close()
    assert rep.steps == 4
