"""Selection, acceptance and sampling at the sizes where their kernels' splits can go wrong: vocabularies that are not a multiple
of four or smaller than the number of slices, as many candidates as a head may keep, batches, and accepted paths of every
length.  All of it is integer logic on values read back from the GPU, so it is compared exactly (sampling: up to the stated
margin around a decision boundary)."""
import pytest
import torch

import inputs
from oracle import amphista_oracle as ao
from oracle import amphista_sampling as sm
from tests.test_gpu_sampling import _check_choices

pytestmark = pytest.mark.gpu


def _model(shape, batch=1, temperature=0.0):
    from paper_2406_13170_b200 import Amphista
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    m = Amphista(shape, topo, w, max_batch=batch, temperature=temperature, seed=9)
    for b in range(batch):
        m.prefill(inputs.make_prompt(shape.with_(prompt_len=20 + 7 * b), seed=3 + b).tolist(), seq=b)
    return m, ao.tree_tables(topo.parent, topo.depth, topo.rank)


@pytest.mark.parametrize("batch", [1, 3])
@pytest.mark.parametrize("name,vocab,topk", [("tiny", 20, (16, 16, 1, 5)), ("tiny", 33, (4, 2, 2, 1)), ("tiny", 1003, (16, 9, 3, 1)),
                                             ("small_bf16", 2176, (16, 5, 4, 3))])
def test_candidates_are_the_exact_top_k(name, vocab, topk, batch):
    shape = inputs.get_shape(name).with_(vocab=vocab, topk=topk)
    m, t = _model(shape, batch)
    K = shape.K
    ids = torch.zeros(batch, K, 16, dtype=torch.int32, device="cuda:0")
    vals = torch.zeros(batch, K, 16, device="cuda:0")
    m.draft(ids, vals)
    m.synchronize()
    for b in range(batch):
        logits = m.get_tensor(f"d_logits#{b}", (K, vocab)).cpu()
        toks = m.get_tensor(f"tree_tokens#{b}", (t.n_nodes,), torch.int32).tolist()
        for k in range(K):
            want = torch.sort(logits[k], descending=True, stable=True)       # equal values by ascending id
            assert ids[b, k, :topk[k]].tolist() == want.indices[:topk[k]].tolist()
            assert torch.equal(vals[b, k, :topk[k]].cpu(), want.values[:topk[k]])
        for n in range(1, t.n_nodes):
            assert toks[n] == int(ids[b, t.depth[n] - 1, t.rank[n]])
    m.close()


@pytest.mark.parametrize("name", ["tiny", "small_bf16"])
def test_a_nan_logit_is_nobodys_candidate(name):
    """Ids whose logit is not a number (either sign) are passed over; a head without any number has no candidates (id 2^31 - 1)."""
    from paper_2406_13170_b200 import Amphista
    shape = inputs.get_shape(name).with_(topk=(16, 5, 2, 3))
    topo = inputs.make_tree(shape.n_nodes, shape.topk)
    w = inputs.make_weights(shape, seed=0, device="cuda:0", init="fan_in")
    bad = torch.arange(0, shape.vocab, 3, device="cuda:0")
    w["draft.lm_head.0"][bad] = float("nan")
    w["draft.lm_head.1"][bad] = -float("nan")
    w["draft.lm_head.3"][:] = float("nan")
    m = Amphista(shape, topo, w)
    m.prefill(inputs.make_prompt(shape).tolist())
    ids = torch.zeros(shape.K, 16, dtype=torch.int32, device="cuda:0")
    m.draft(ids)
    m.synchronize()
    logits = m.get_tensor("d_logits", (shape.K, shape.vocab)).cpu()
    for k in range(3):
        assert bool(torch.isnan(logits[k]).any()) == (k < 2)
        want = torch.sort(logits[k].nan_to_num(nan=-float("inf")), descending=True, stable=True).indices
        assert ids[k, :shape.topk[k]].tolist() == want[:shape.topk[k]].tolist()
    assert ids[3, :3].tolist() == [2 ** 31 - 1] * 3
    m.close()


@pytest.mark.parametrize("name", ["tiny", "small_bf16"])
def test_accepted_rows_move_in_every_layer(name):
    shape = inputs.get_shape(name)
    B = 3
    m, t = _model(shape, B)
    N, K, d = t.n_nodes, shape.K, shape.d_model
    kinds = [f"kv.{c}.{i}" for c in "kv" for i in range(shape.n_layers)]
    for leaf in sorted(range(N), key=lambda n: (-t.depth[n], -n))[::5]:
        m.draft()
        m.verify_tree()
        tok = torch.zeros(B, K + 1, dtype=torch.int32, device="cuda:0")
        path, cnt, nxt = tok.clone(), torch.zeros(B, dtype=torch.int32, device="cuda:0"), torch.zeros(B, dtype=torch.int32, device="cuda:0")
        C = [m.get_state(b)[0] for b in range(B)]
        want, before = [], []
        for b in range(B):
            toks = m.get_tensor(f"tree_tokens#{b}", (N,), torch.int32).tolist()
            choice = [(shape.vocab - 1 - n) for n in range(N)]
            n = (leaf + b) % N
            while n > 0:                                             # the tokens of the path to `leaf` are the choices on it
                choice[t.parent[n]] = toks[n]
                n = t.parent[n]
            m.set_tensor(f"argmax#{b}", torch.tensor(choice, dtype=torch.int32, device="cuda:0"))
            want.append(ao.Oracle.accept(toks, choice, t))
            before.append({k: m.get_tensor(f"{k}#{b}@{C[b]}", (N, d)).clone() for k in kinds})
        m.accept(tok, cnt, path, nxt)
        m.synchronize()
        for b in range(B):
            L, p, emitted, root = want[b]
            assert (int(cnt[b]), path[b, :L].tolist(), tok[b, :L].tolist(), int(nxt[b])) == (L, list(p), list(emitted), root)
            assert path[b, L:].tolist() == [-1] * (K + 1 - L) == tok[b, L:].tolist()
            assert m.get_state(b) == (C[b] + L, root, L)
            for k in kinds:
                assert torch.equal(m.get_tensor(f"{k}#{b}@{C[b]}", (L, d)), before[b][k][list(p)]), (k, b)
    m.close()


@pytest.mark.parametrize("vocab", [20, 1003, 4100])
def test_sampled_choices_at_ragged_vocabularies(vocab):
    shape = inputs.get_shape("tiny").with_(vocab=vocab, topk=(16, 9, 3, 1), n_nodes=40)
    B = 2
    m, t = _model(shape, B, temperature=0.7)
    N = t.n_nodes
    m.draft()
    m.verify_tree()
    stats = {"near_boundary": 0, "nodes": 0}
    for b in range(B):
        toks = m.get_tensor(f"tree_tokens#{b}", (N,), torch.int32).tolist()
        logits = m.get_tensor(f"logits#{b}", (N, vocab)).cpu().to(torch.float64)
        u = sm.node_uniforms(9, 0, b, N)
        assert m.get_tensor(f"uniforms#{b}", (N,)).cpu().tolist() == u
        _check_choices(m.get_tensor(f"argmax#{b}", (N,), torch.int32).tolist(), toks, logits, t, 0.7, u, stats)
    assert stats["near_boundary"] <= 2
    m.close()
