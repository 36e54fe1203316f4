"""Sizes and arguments at the edge of what a call may be given: models whose vocabulary is wide against
their hidden size, and caller trees and prompts that do not keep to their own bounds."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2408_08146_b200 import KoalaError
from tests.harness import make_pair, tok_list
from tests.parity import assert_close, check_argmax
from workloads import T7_EAGLE, TINY_EAGLE, reduced
from workloads.generate import prompts

pytestmark = pytest.mark.gpu


def _to(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to("cuda:0")


# (N - 1) rows of logits take more floats than the partial sums of any multiply of these models
WIDE = {"fp32": TINY_EAGLE.with_(N=15, V=40000, S_max=64, prompt_len=20, seed=41),
        "bf16": reduced(T7_EAGLE, 1, K=1, H=512, n_heads=4, F=1376, V=50000, N=64, S_max=256, prompt_len=100, seed=42)}


@pytest.mark.parametrize("model", WIDE)
@pytest.mark.parametrize("B", [1, 2])
def test_short_trees_and_prompts_under_a_wide_vocabulary(model, B):
    cfg = WIDE[model].with_(B=B)
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float64 if model == "fp32" else np.float32, cache_host=model == "fp32")
    N, n_max = cfg.N, cfg.N - 1
    pr = prompts(cfg)
    eng.prefill(pr, n_max)                       # the last parts are shorter than N
    orc.prefill(pr, n_max)

    def check(n, what):
        bufs = eng.buffers()
        for b in range(B):
            assert_close(bufs["verify_logits"][b * N:b * N + n].cpu().numpy(), orc.verify_logits[b][:n], cfg.dtype, f"{what} {b}")
            check_argmax(bufs["verify_tgt"][b * N:b * N + n].cpu().numpy(), orc.verify_logits[b], f"{what} {b}")

    check(len(np.array_split(pr[0], -(-len(pr[0]) // n_max))[-1]), "prompt")
    rng = np.random.default_rng(n_max)
    tok = rng.integers(0, cfg.V, (B, n_max))
    par = np.asarray([[-1] + [int(rng.integers(0, u)) for u in range(1, n_max)] for _ in range(B)])
    eng.koala_verify((_to(tok), _to(par), _to(np.full(B, n_max)), n_max))
    orc.verify([(list(map(int, tok[b])), list(map(int, par[b]))) for b in range(B)])
    check(n_max, "tree")
    assert eng.device_status() == 0
    assert eng.check_guards()[1] == 0
    eng.close()


@pytest.mark.parametrize("N,n_max", [(15, 4), (15, 14), (15, 15)])
def test_a_tree_larger_than_its_bound_is_reported_and_cut(N, n_max):
    """n_nodes[b] = n_max + 1 where the arrays hold that node: the forward has no row for it, so the sequence's
    tree ends at n_max nodes (as if the caller had said so) and the status says that it was cut."""
    cfg = TINY_EAGLE.with_(B=2, N=N, prompt_len=30, S_max=128, seed=43)
    eng, orc, _ = make_pair(cfg)
    pr = prompts(cfg)
    eng.prefill(pr, cfg.N)
    orc.prefill(pr, cfg.N)
    rng = np.random.default_rng(n_max)
    tok = rng.integers(0, cfg.V, (2, n_max + 1))
    par = np.asarray([[-1] + list(range(n_max))] * 2)                     # chains
    eng.koala_verify((_to(tok), _to(par), _to([n_max, n_max + 1]), n_max))
    orc.verify([(list(map(int, tok[b, :n_max])), list(map(int, par[b, :n_max]))) for b in range(2)])
    forced = _to([n_max + 1, n_max + 1])                                   # as far as the tree goes
    got, n = eng.koala_accept(forced)
    assert n.cpu().tolist() == [n_max, n_max]
    assert eng.seq_len.cpu().tolist() == [30 + n_max, 30 + n_max]
    for b in range(2):
        logits = eng.buffers()["verify_logits"][b * N:b * N + n_max].cpu().numpy()
        assert_close(logits, orc.verify_logits[b], cfg.dtype, f"logits {b}")
        check_argmax(got[b, n_max - 1:n_max].cpu().numpy(), orc.verify_logits[b][n_max - 1:], f"bonus {b}")
    assert eng.device_status() == 1
    assert eng.check_guards()[1] == 0
    eng.close()


def test_a_prompt_shorter_than_its_number_of_parts_is_refused():
    """Five tokens cannot be six parts: refused before anything is enqueued, nothing of the batch has moved."""
    cfg = TINY_EAGLE.with_(B=2, prompt_len=60, S_max=128, seed=44)
    eng, orc, _ = make_pair(cfg)
    rng = np.random.default_rng(44)
    long, short = rng.integers(0, cfg.V, 60), rng.integers(0, cfg.V, 5)
    launches = eng.launch_count()
    with pytest.raises(KoalaError) as e:
        eng.prefill([long, short], 10)
    assert e.value.code == 1 and eng.launch_count() == launches
    assert eng.seq_len.cpu().tolist() == [0, 0]
    eng.prefill([long, short], 15)               # four parts: 2 + 1 + 1 + 1 tokens
    orc.prefill([long, short], 15)
    for _ in range(2):
        tk, ln = tok_list(*eng.step())
        rt, rl = orc.step()
        assert [list(x) for x in tk] == [list(x) for x in rt] and list(ln) == list(rl)
    assert eng.device_status() == 0
    eng.close()


def test_a_part_of_more_than_n_tokens_is_refused():
    """2 N + 1 tokens in two parts: the first would have N + 1, a chain that no tree holds."""
    cfg = TINY_EAGLE.with_(prompt_len=31, S_max=128, seed=45)
    eng, orc, _ = make_pair(cfg)
    pr = prompts(cfg)
    tok = _to([pr[0]])
    ingest = lambda parts: eng.lib.koala_ingest(eng._ctx, tok.data_ptr(), 31, (C.c_int32 * 1)(31), parts)
    assert cfg.N == 15 and ingest(2) == 1
    assert eng.seq_len.cpu().tolist() == [0] and eng.koala_accept_stats(20) == ([0] * 20, [0] * 20)
    assert ingest(3) == 0
    eng.koala_accept(eng.buffers()["tree_n"])
    orc.prefill(pr, 15)
    assert eng.seq_len.cpu().tolist() == orc.seq_len
    rt, rl = orc.step()
    tk, ln = tok_list(*eng.step())
    assert [list(x) for x in tk] == [list(x) for x in rt] and list(ln) == list(rl)
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
def test_rows_wider_than_the_vectorised_kernels_take(dtype):
    """A hidden size above 8192 goes by the row-wise kernels of any width: prompt, draft pass and verification."""
    cfg = reduced(T7_EAGLE, 1, dtype=dtype, K=1, H=8320, n_heads=65, F=256, V=512, D=1, topk=2, N=3, S_max=128, prompt_len=6, seed=46)
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    pr = prompts(cfg)
    eng.prefill(pr, 3)
    orc.prefill(pr, 3)
    eng.koala_draft(0)
    orc.draft(0)
    assert_close(eng.buffers()["draft_logits"][:1].cpu().numpy(), orc.draft_logits[0][:1], dtype, "draft logits")
    eng.koala_expand_tree(0)
    eng.koala_verify(None)
    b = eng.buffers()
    n = int(b["tree_n"][0])
    orc.verify([(b["tree_tok"][0, :n].cpu().numpy(), b["tree_parent"][0, :n].cpu().numpy())])
    assert_close(b["verify_logits"][:n].cpu().numpy(), orc.verify_logits[0], dtype, "logits")
    assert eng.device_status() == 0 and eng.check_guards()[1] == 0
    eng.close()
