"""Edge cases of the CUDA path against the oracle: degenerate trees, maximum tree size, a head
without layers, long contexts that span many key tiles and several key chunks, capacity and
malformed-input reporting, and the call-order rules."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle.koala_oracle import KoalaOracle, round_to_bf16
from paper_2408_08146_b200 import Koala, KoalaError
from tests.harness import kv_to_oracle, make_pair, tok_list
from tests.helpers import HostWeights
from tests.parity import assert_close, check_argmax
from workloads import T7_EAGLE, TINY_EAGLE, reduced
from workloads.generate import prompts, random_kv, uniform_ints

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _tree_arrays(eng, toks, parents):
    cfg = eng.cfg
    n = len(toks[0])
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)
    return to(toks), to(parents), to(np.full(cfg.B, n)), n


def test_single_node_tree_is_plain_autoregressive_decoding():
    cfg = TINY_EAGLE.with_(N=1, D=1, S_max=128)
    eng, orc, _ = make_pair(cfg)
    pr = prompts(cfg)
    # one token per call: 64 single-node chains, forced acceptance of 1 = the node itself
    for t in range(cfg.prompt_len):
        tree = _tree_arrays(eng, [[int(pr[0][t])]], [[-1]])
        eng.koala_verify(tree)
        eng.koala_accept(tree[2])
    orc.prefill(pr, 1)
    out = []
    for _ in range(6):
        root = eng.buffers()["root_tok"].cpu().numpy().reshape(1, 1)
        eng.koala_verify(_tree_arrays(eng, root, [[-1]]))
        tk, ln = tok_list(*eng.koala_accept(None))
        assert ln == [1]
        out += tk[0]
    assert out == orc.ar_greedy(6)[0]
    assert eng.device_status() == 0
    eng.close()


def test_maximum_tree_of_128_nodes_chain_and_bushy():
    cfg = TINY_EAGLE.with_(N=128, D=4, topk=2, S_max=400, prompt_len=128)
    eng, orc, _ = make_pair(cfg)
    pr = prompts(cfg)
    eng.prefill(pr, 128)                     # one chain of 128 nodes: every mask bit in use
    orc.prefill(pr, 128)
    assert eng.seq_len.cpu().tolist() == orc.seq_len == [128]
    for l in range(cfg.L):
        assert_close(kv_to_oracle(eng.target_k, l, 0, np.float64)[:128], orc.target_k[l][0][:128], cfg.dtype, "K")
    # a bushy 128-node caller tree on top of it
    n = 128
    par = [-1] + [int(p) for p in (uniform_ints(5, "edge.par", n - 1, 0, 1 << 20) % np.arange(1, n))]
    par = [-1 if u == 0 else min(par[u], u - 1) for u in range(n)]
    tok = uniform_ints(5, "edge.tok", n, 0, cfg.V)
    tok[0] = orc.root_tok[0]
    eng.koala_verify(_tree_arrays(eng, [tok], [par]))
    orc.verify([(tok, np.asarray(par))])
    b = eng.buffers()
    assert_close(b["verify_logits"][:n].cpu().numpy(), orc.verify_logits[0], cfg.dtype, "128-node tree logits")
    check_argmax(b["verify_tgt"][:n].cpu().numpy(), orc.verify_logits[0], "128-node tree arg-max")
    got = tok_list(*eng.koala_accept(None))
    ref = orc.accept()
    assert list(got[0]) == list(ref[0]) and list(got[1]) == list(ref[1])
    assert eng.device_status() == 0
    eng.close()


def test_eagle_head_without_layers():
    cfg = TINY_EAGLE.with_(K=0, S_max=160)
    eng, orc, _ = make_pair(cfg)
    pr = prompts(cfg)
    eng.prefill(pr, 15)
    orc.prefill(pr, 15)
    for _ in range(2):
        got = tok_list(*eng.step())
        ref = orc.step()
        assert list(got[0]) == ref[0] and list(got[1]) == ref[1]
        n = len(orc.tree_tok[0])
        assert eng.buffers()["tree_tok"][0, :n].cpu().tolist() == list(orc.tree_tok[0])
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("context", [1000, 3900])
def test_long_context_many_key_tiles_and_chunks(context):
    """bf16, head_dim 128, one 7B-shaped layer: the attention kernel walks dozens of key tiles and,
    at the longer context, several key chunks merged inside a cluster."""
    cfg = reduced(T7_EAGLE, 1, K=1, N=60, S_max=4096, prompt_len=context)
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    eng.target_k.copy_(random_kv(cfg, "target_k", cfg.L, DEV))
    eng.target_v.copy_(random_kv(cfg, "target_v", cfg.L, DEV))
    orc.target_k[0][0][...] = kv_to_oracle(eng.target_k, 0, 0, np.float32)
    orc.target_v[0][0][...] = kv_to_oracle(eng.target_v, 0, 0, np.float32)
    eng.seq_len.fill_(context)
    orc.seq_len[0] = context
    n = cfg.N
    par = [-1] + [max(0, u - 1 - (u * 7) % min(u, 5)) for u in range(1, n)]
    tok = uniform_ints(9, "edge.long", n, 0, cfg.V)
    eng.koala_verify(_tree_arrays(eng, [tok], [par]))
    orc.verify([(tok, np.asarray(par))])
    b = eng.buffers()
    assert_close(b["verify_hid"][:n].cpu().numpy(), orc.verify_hid[0], cfg.dtype, f"hidden at context {context}")
    assert_close(b["verify_logits"][:n].cpu().numpy(), orc.verify_logits[0], cfg.dtype, f"logits at context {context}")
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("N,B,n_heads,context,S_max", [
    (128, 1, 32, 1000, 4096),    # more than 64 rows: every row warp owns its rows; 4 key chunks
    (100, 2, 32, 700, 1024),     # ragged row count above 64, 2 chunks, two sequences
    (20, 1, 32, 300, 512),       # fewer than 32 rows: one row group, duplicated
    (40, 8, 32, 200, 512),       # more CTAs than SMs: a single chunk, no cluster
    (60, 1, 8, 3000, 4096),      # few heads: 8 key chunks per head
    (33, 1, 32, 64, 256),        # a short context: one tile per chunk
    (33, 1, 32, 20, 1024),       # one key tile, four key chunks: three CTAs of a cluster have no tile and still merge and store their dims
    (60, 1, 8, 10, 4096),        # two key tiles, eight key chunks
])
def test_tensor_core_attention_shapes(N, B, n_heads, context, S_max):
    """One bf16 layer with head_dim 128 at row counts, batch sizes and chunk counts that select
    every variant of the tcgen05 attention kernel; the tree sits on top of a random cache."""
    _attention_case(N, B, n_heads, context, S_max)


@pytest.mark.parametrize("N,B,n_heads,context,S_max", [
    (60, 1, 32, 500, 1024),      # tcgen05 kernel, duplicated rows; the last key tile is partial
    (100, 2, 32, 700, 1024),     # tcgen05 kernel, more than 64 rows
    (8, 1, 32, 300, 512),        # fewer than 16 rows: the mma.sync kernel
])
def test_unwritten_cache_slots_may_hold_nan(N, B, n_heads, context, S_max):
    """Only the slots below seq_len (and the tree's own) ever hold data the caller or the library
    wrote; everything beyond may be uninitialised memory.  The slots from S + N on are filled with
    NaN bit patterns here (plain data, nothing faults) and the result must not change."""
    _attention_case(N, B, n_heads, context, S_max, poison=True)


@pytest.mark.parametrize("N,B,n_heads,context,S_max", [
    (60, 1, 32, 1000, 2048),     # duplicated rows, 4 key chunks of several tiles each
    (128, 1, 32, 1500, 4096),    # every row warp owns its rows
])
def test_scores_that_grow_along_the_context(N, B, n_heads, context, S_max):
    """Keys whose magnitude grows eightfold from the first to the last cached position: the row
    maxima rise by far more than 2^8 from tile to tile, so the running output, which the tcgen05
    kernel keeps in tensor memory relative to a lazily raised reference maximum, is rescaled in place
    several times."""
    _attention_case(N, B, n_heads, context, S_max, growing=True)


@pytest.mark.parametrize("N,context,S_max", [
    (128, 30, 1024),             # more than 64 rows: three tiles for eight chunks, most of which have none
    (128, 1500, 2048),
    (65, 700, 1024),
    (60, 20, 1024),              # duplicated rows
    (64, 1900, 2048),
])
@pytest.mark.parametrize("growing", [False, True])
def test_eight_key_chunks(N, context, S_max, growing):
    """Eight heads leave room for eight chunks per head: merged over the whole cluster, with references that differ from chunk
    to chunk where the scores grow."""
    _attention_case(N, 1, 8, context, S_max, growing=growing)


def _attention_case(N, B, n_heads, context, S_max, poison=False, growing=False):
    H = n_heads * 128
    cfg = reduced(T7_EAGLE, 1, K=1, N=N, B=B, H=H, n_heads=n_heads, F=2 * H, V=2048, D=min(5, N - 1),
                  S_max=S_max, prompt_len=context)
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    eng.target_k.copy_(random_kv(cfg, "target_k", cfg.L, DEV))
    eng.target_v.copy_(random_kv(cfg, "target_v", cfg.L, DEV))
    if growing:
        ramp = 1.0 + 7.0 * torch.arange(S_max, device=DEV, dtype=torch.float32) / context
        eng.target_k.copy_((eng.target_k.float() * ramp.view(1, 1, 1, S_max, 1)).to(eng.target_k.dtype))
    lens = [context - 13 * b for b in range(B)]
    for b in range(B):
        orc.target_k[0][b][...] = kv_to_oracle(eng.target_k, 0, b, np.float32)
        orc.target_v[0][b][...] = kv_to_oracle(eng.target_v, 0, b, np.float32)
        orc.seq_len[b] = lens[b]
    eng.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    if poison:
        for b in range(B):
            eng.target_k[:, b, :, lens[b] + N:, :] = float("nan")
            eng.target_v[:, b, :, lens[b] + N:, :] = float("nan")
    par = [-1] + [max(0, u - 1 - (u * 7) % min(u, 5)) for u in range(1, N)]
    toks = [uniform_ints(11 + b, "edge.shapes", N, 0, cfg.V) for b in range(B)]
    eng.koala_verify(_tree_arrays(eng, toks, [par] * B))
    orc.verify([(toks[b], np.asarray(par)) for b in range(B)])
    bufs = eng.buffers()
    for b in range(B):
        assert_close(bufs["verify_hid"][b * N:(b + 1) * N].cpu().numpy(), orc.verify_hid[b], cfg.dtype,
                     f"hidden, sequence {b}")
    assert eng.device_status() == 0
    eng.close()


def test_capacity_and_malformed_trees_are_reported_not_executed():
    cfg = TINY_EAGLE.with_(S_max=80)                    # the 64-token prompt fits, prompt + tree does not
    eng, orc, _ = make_pair(cfg)
    pr = prompts(cfg)
    eng.prefill(pr, 15)
    assert eng.device_status() == 0
    eng.seq_len.fill_(70)                               # 70 + 15 > 80
    k_before = eng.target_k.clone()
    eng.koala_verify(_tree_arrays(eng, [[1] * 15], [list(range(-1, 14))]))
    assert eng.device_status() == 3                     # KOALA_E_CAPACITY, from the plan kernel
    assert torch.equal(k_before, eng.target_k)          # nothing was written past the capacity
    eng.close()
    eng, _, _ = make_pair(TINY_EAGLE)
    eng.koala_verify(_tree_arrays(eng, [[1, 2, 3]], [[-1, 2, 0]]))     # parent index not below the child
    assert eng.device_status() == 1                     # KOALA_E_INVALID
    eng.close()


def test_call_order_and_argument_errors():
    eng, _, _ = make_pair(TINY_EAGLE)
    with pytest.raises(KoalaError) as e:
        eng.koala_expand_tree(0)                        # nothing drafted
    assert e.value.code == 4
    with pytest.raises(KoalaError) as e:
        eng.koala_draft(1)                              # pass 1 before pass 0
    assert e.value.code == 4
    with pytest.raises(KoalaError) as e:
        eng.koala_draft(99)
    assert e.value.code == 1
    with pytest.raises(KoalaError) as e:
        eng.koala_verify(None)                          # no drafted tree
    assert e.value.code == 4
    with pytest.raises(KoalaError) as e:
        eng.koala_accept(None)                          # nothing verified
    assert e.value.code == 4
    tok = torch.zeros(1, 16, dtype=torch.int32, device=DEV)
    with pytest.raises(KoalaError) as e:
        eng.koala_verify((tok, tok, torch.ones(1, dtype=torch.int32, device=DEV), 16))   # n_max > N
    assert e.value.code == 1
    eng.close()


def test_position_wise_acceptance_counters_match_the_oracle():
    """n-alpha counters (Section 4.1, metrics): chains whose first m tokens are the target's own
    greedy continuation, then free-running iterations with the head's real trees; the device
    counters equal the oracle's and, for the planted part, the tally made here from (m, d)."""
    cfg = TINY_EAGLE.with_(S_max=256)
    eng, orc, store = make_pair(cfg)
    pr = prompts(cfg)
    eng.prefill(pr, 15)
    orc.prefill(pr, 15)
    truth_src = KoalaOracle(cfg, HostWeights(store, np.float64))
    truth_src.prefill(pr, 64)
    truth = truth_src.ar_greedy(80)[0]
    eng.koala_accept_stats(1, reset=True)
    orc.reset_alpha()
    hits, trials = [0] * cfg.N, [0] * cfg.N
    emitted = 0
    for it in range(10):
        d = 1 + (it * 3) % 5
        m = (it * 7) % (d + 1)
        tok = [int(orc.root_tok[0])]
        for i in range(d):
            t = int(truth[emitted + i])
            tok.append(t if i < m else (t + 1 + 13 * it) % cfg.V)
        par = list(range(-1, d))
        eng.koala_verify(_tree_arrays(eng, [tok], [par]))
        orc.verify([(np.asarray(tok), np.asarray(par))])
        got = tok_list(*eng.koala_accept(None))
        ref = orc.accept()
        assert list(got[1]) == list(ref[1]) == [m + 1] and list(got[0][0]) == list(ref[0][0])
        emitted += m + 1
        for n in range(1, d + 1):
            trials[n - 1] += n <= m + 1
            hits[n - 1] += n <= m
    g_hits, g_trials = eng.koala_accept_stats(cfg.N)
    assert g_hits == hits == orc.alpha_hits[:cfg.N] and g_trials == trials == orc.alpha_trials[:cfg.N]
    for _ in range(4):                                   # the head's own trees
        got = tok_list(*eng.step())
        ref = orc.step()
        assert list(got[0]) == ref[0] and list(got[1]) == ref[1]
    g_hits, g_trials = eng.koala_accept_stats(cfg.N, reset=True)
    assert g_hits == orc.alpha_hits[:cfg.N] and g_trials == orc.alpha_trials[:cfg.N]
    assert eng.koala_accept_stats(cfg.N) == ([0] * cfg.N, [0] * cfg.N)
    assert eng.device_status() == 0
    eng.close()


def test_whole_iterations_repeat_bit_for_bit():
    """Two engines on the same weights, prompts ingested in chunks (the first chunks have fewer key
    tiles than key chunks), several forced iterations: trees, target tokens and accepted tokens must
    be identical."""
    from workloads import T7_EAGLE, reduced
    from workloads.generate import WeightStore
    from paper_2408_08146_b200 import Koala
    cfg = reduced(T7_EAGLE, 2, K=1, S_max=768, prompt_len=300)
    store = WeightStore(cfg, DEV)
    forced = torch.tensor([[3], [1], [5], [2]], dtype=torch.int32, device=DEV)
    runs = []
    for _ in range(2):
        eng = Koala(cfg, store.tensors)
        eng.prefill(prompts(cfg), 64)
        rec = [eng.buffers()["root_tok"].cpu().numpy().copy()]
        for i in range(forced.shape[0]):
            toks, lens = eng.step(forced[i])
            torch.cuda.synchronize()
            b = eng.buffers()
            n = int(b["tree_n"][0].item())
            rec += [lens.cpu().numpy().copy(), toks[0, :int(lens[0].item())].cpu().numpy().copy(),
                    b["tree_tok"][0, :n].cpu().numpy().copy(), b["verify_tgt"][:n].cpu().numpy().copy()]
        assert eng.device_status() == 0
        eng.close()
        runs.append(rec)
    for a, c in zip(*runs):
        assert np.array_equal(a, c)


@pytest.mark.parametrize("base,B,N,n_max", [("tiny", 3, 15, 1), ("tiny", 2, 15, 4), ("7b", 4, 64, 1), ("7b", 3, 40, 17),
                                            ("7b", 4, 64, 40)])
def test_short_caller_trees_of_a_batch_run_only_their_rows(base, B, N, n_max):
    """Several sequences with caller trees of at most n_max < N nodes: node u of sequence b is row b * N + u
    of the outputs, whatever rows the forward itself used; ragged node counts, then an accepted path."""
    from tests.parity import assert_close
    if base == "tiny":
        cfg = TINY_EAGLE.with_(B=B, N=N, prompt_len=30, prompt_len_min=21, S_max=128, seed=21)
    else:
        cfg = reduced(T7_EAGLE, 1, B=B, N=N, prompt_len=70, prompt_len_min=33, S_max=256, K=1, seed=22)
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float64 if base == "tiny" else np.float32, cache_host=base == "tiny")
    pr = prompts(cfg)
    eng.prefill(pr, cfg.N)
    orc.prefill(pr, cfg.N)
    rng = np.random.default_rng(n_max)
    counts = [max(1, n_max - b) for b in range(B)]
    tok = rng.integers(0, cfg.V, (B, n_max)).astype(np.int32)
    par = np.asarray([[-1] + [int(rng.integers(0, u)) for u in range(1, n_max)] for _ in range(B)], np.int32)
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to("cuda:0")
    eng.koala_verify((to(tok), to(par), to(np.asarray(counts)), n_max))
    orc.verify([(list(map(int, tok[b, :counts[b]])), list(map(int, par[b, :counts[b]]))) for b in range(B)])
    bufs = eng.buffers()
    for b in range(B):
        n = counts[b]
        assert_close(bufs["verify_hid"][b * N:b * N + n].cpu().numpy(), orc.verify_hid[b][:n], cfg.dtype, f"hidden {b}")
        assert_close(bufs["verify_logits"][b * N:b * N + n].cpu().numpy(), orc.verify_logits[b][:n], cfg.dtype, f"logits {b}")
        got = bufs["verify_logits"][b * N:b * N + n].argmax(1).cpu().tolist()
        assert bufs["verify_tgt"][b * N:b * N + n].cpu().tolist() == got
    eng.koala_accept(None)
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("N,B,n_heads,context,S_max", [
    (2, 1, 32, 1, 128),          # less than one tile
    (2, 1, 32, 63, 256),         # the tree crosses a tile boundary; fewer tiles than CTAs
    (3, 1, 8, 3000, 4096),       # few heads: every head is cut into many parts
    (4, 2, 32, 700, 1024),
    (4, 9, 8, 200, 512),         # more (sequence, head) pairs than parts
    (2, 1, 1, 2000, 2048),       # a single head
    (3, 5, 16, 130, 256),
    (5, 1, 32, 777, 1024),       # three to fifteen rows: mma.sync
    (8, 3, 8, 500, 1024),
    (7, 1, 2, 1900, 2048),
    (9, 1, 32, 1000, 1024),
    (15, 2, 8, 600, 2048),
])
@pytest.mark.parametrize("kind", ["plain", "poison", "growing"])
def test_attention_of_few_rows(N, B, n_heads, context, S_max, kind):
    """Up to fifteen rows per sequence: the CUDA-core kernel (one or two rows) and mma.sync, key chunks as a cluster."""
    _attention_case(N, B, n_heads, context, S_max, poison=kind == "poison", growing=kind == "growing")


@pytest.mark.parametrize("N,lens,n_heads,S_max", [
    (1, [63], 32, 256),              # the new row is the last of a tile / the first of one / alone in the cache
    (1, [64], 32, 1024),
    (1, [1], 8, 128),
    (2, [63], 32, 256),              # two new rows in different tiles, and so in different chunks
    (2, [127, 62, 5], 16, 512),
    (2, [500, 191], 32, 1024),
    (1, [900, 64, 130], 32, 1152),
])
def test_few_rows_take_the_sums_of_the_multiply(N, lens, n_heads, S_max):
    """One or two rows per sequence, where the attention rotates the queries and writes the cache itself: two layers, so
    that the second layer's context reads lie before its dependency wait; hidden states and the rows written."""
    B = len(lens)
    cfg = reduced(T7_EAGLE, 2, K=1, N=N, D=1, topk=1, B=B, H=128 * n_heads, n_heads=n_heads, F=2048, V=2048, S_max=S_max, prompt_len=max(lens))
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    eng.target_k.copy_(random_kv(cfg, "target_k", cfg.L, DEV))
    eng.target_v.copy_(random_kv(cfg, "target_v", cfg.L, DEV))
    for b in range(B):
        for l in range(cfg.L):
            orc.target_k[l][b][...] = kv_to_oracle(eng.target_k, l, b, np.float32)
            orc.target_v[l][b][...] = kv_to_oracle(eng.target_v, l, b, np.float32)
        orc.seq_len[b] = lens[b]
    eng.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    toks, pars = [[5 + b, 9][:N] for b in range(B)], [[-1, 0][:N]] * B
    eng.koala_verify(_tree_arrays(eng, toks, pars))
    orc.verify(list(zip(toks, pars)))
    hid = eng.buffers()["verify_hid"]
    for b in range(B):
        assert_close(hid[b * N:(b + 1) * N].cpu().numpy(), orc.verify_hid[b][:N], cfg.dtype, f"hidden {b}")
        for l in range(cfg.L):
            for name, got, want in (("K", eng.target_k, orc.target_k), ("V", eng.target_v, orc.target_v)):
                assert_close(kv_to_oracle(got, l, b, np.float32)[:lens[b] + N], want[l][b][:lens[b] + N], cfg.dtype, f"{name} {l} {b}")
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("N,lens,n_heads,S_max", [
    (1, [63], 32, 256),
    (1, [1], 8, 128),
    (2, [63], 32, 256),
    (2, [127, 62, 5], 16, 512),
    (2, [500, 191], 32, 1024),
    (1, [800, 64, 130], 32, 896),    # long and ragged: up to seven tiles per chunk
])
@pytest.mark.parametrize("short", [False, True], ids=["all", "last_tree_of_one_node"])
def test_rotary_step_inside_the_attention_runs_and_leaves_other_slots_alone(N, lens, n_heads, S_max, short):
    """The same where the launches say that the fused path ran (a launch less per layer than with more capacity); a row that
    no node uses writes nothing, nor does any row write past its sequence's end."""
    if short and N == 1:
        pytest.skip("every row is in use")
    B = len(lens)
    cfg = reduced(T7_EAGLE, 2, K=1, N=N, D=1, topk=1, B=B, H=128 * n_heads, n_heads=n_heads, F=2048, V=2048, S_max=S_max, prompt_len=max(lens))
    eng, orc, store = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    eng.target_k.copy_(random_kv(cfg, "target_k", cfg.L, DEV))
    eng.target_v.copy_(random_kv(cfg, "target_v", cfg.L, DEV))
    before = (eng.target_k.clone(), eng.target_v.clone())
    for b in range(B):
        for l in range(cfg.L):
            orc.target_k[l][b][...] = kv_to_oracle(eng.target_k, l, b, np.float32)
            orc.target_v[l][b][...] = kv_to_oracle(eng.target_v, l, b, np.float32)
        orc.seq_len[b] = lens[b]
    eng.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    counts = [1 if short and b == B - 1 else N for b in range(B)]
    toks, pars = [[5 + b, 9][:N] for b in range(B)], [[-1, 0][:N]] * B
    tok, par, _, n = _tree_arrays(eng, toks, pars)
    tree = (tok, par, torch.tensor(counts, dtype=torch.int32, device=DEV), n)

    def launches(e):
        first = e.launch_count()
        e.koala_verify(tree)
        return e.launch_count() - first

    fused = launches(eng)
    orc.verify([(toks[b][:counts[b]], pars[b][:counts[b]]) for b in range(B)])
    hid = eng.buffers()["verify_hid"]
    for b in range(B):
        end = lens[b] + counts[b]
        assert_close(hid[b * N:b * N + counts[b]].cpu().numpy(), orc.verify_hid[b][:counts[b]], cfg.dtype, f"hidden {b}")
        for l in range(cfg.L):
            for name, got, want, old in (("K", eng.target_k, orc.target_k, before[0]), ("V", eng.target_v, orc.target_v, before[1])):
                assert_close(kv_to_oracle(got, l, b, np.float32)[:end], want[l][b][:end], cfg.dtype, f"{name} {l} {b}")
                assert torch.equal(got[l, b, :, end:], old[l, b, :, end:])
    assert eng.device_status() == 0
    eng.close()
    # the same with more capacity than the sums are taken for: a rotary launch per layer
    eng = Koala(cfg.with_(S_max=5248), store.tensors)
    eng.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    assert launches(eng) == fused + cfg.L
    assert eng.device_status() == 0
    eng.close()


def test_attention_of_one_row_ragged_batch():
    """One-node trees of a ragged batch, twice on the same engine."""
    cfg = reduced(T7_EAGLE, 1, K=1, N=1, D=1, topk=1, B=4, H=1024, n_heads=8, F=2048, V=2048, S_max=1536, prompt_len=1400)
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    eng.target_k.copy_(random_kv(cfg, "target_k", cfg.L, DEV))
    eng.target_v.copy_(random_kv(cfg, "target_v", cfg.L, DEV))
    lens = [1400, 3, 700, 64]
    for b in range(4):
        orc.target_k[0][b][...] = kv_to_oracle(eng.target_k, 0, b, np.float32)
        orc.target_v[0][b][...] = kv_to_oracle(eng.target_v, 0, b, np.float32)
        orc.seq_len[b] = lens[b]
    eng.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    toks = [[5], [6], [7], [8]]
    first = None
    orc.verify([(t, [-1]) for t in toks])
    for _ in range(2):
        eng.koala_verify(_tree_arrays(eng, toks, [[-1]] * 4))
        hid = eng.buffers()["verify_hid"].clone()
        for b in range(4):
            assert_close(hid[b:b + 1].cpu().numpy(), orc.verify_hid[b][:1], cfg.dtype, f"hidden {b}")
        assert first is None or torch.equal(first, hid)
        first = hid
    assert eng.device_status() == 0 and eng.check_guards()[1] == 0
    eng.close()


@pytest.mark.parametrize("V,k", [(5, 5), (300, 16), (1024, 2), (4096, 10), (4097, 10), (9000, 1), (32000, 16), (32768, 3), (40000, 4)])
def test_topk_of_rows_with_ties_and_extremes(V, k):
    """Top-k over one CTA, a cluster of eight and the wide-row kernel: equal values (the smaller id wins, across
    warps and parts), +-0, infinities, a row whose best are all in one warp; log-probabilities in float64."""
    cfg = TINY_EAGLE.with_(V=V, topk=k, D=2, N=min(8, 1 + k), B=4, prompt_len=8, S_max=64)
    eng, _, _ = make_pair(cfg)
    eng.prefill(prompts(cfg), cfg.N)
    eng.koala_draft(0)
    rng = np.random.default_rng(V * 31 + k)
    x = np.round(rng.normal(size=(4, V)) * 4).astype(np.float32) / 4          # many equal values
    x[1] = 0.0
    x[1, ::2] = -0.0                                                       # all equal
    x[2, : min(V, 40)] = 9.0                                               # ids 0..39: neighbouring lanes
    x[3, V // 2:] = -np.inf
    eng.buffers()["draft_logits"].copy_(torch.from_numpy(x))
    eng.set_expand_mode(1)
    eng.koala_expand_tree(0)
    bufs = eng.buffers()
    tok, lp = bufs["topk_tok"].cpu().numpy(), bufs["topk_logp"].cpu().numpy()
    for r in range(4):
        want = np.argsort(-x[r], kind="stable")[:k]
        if np.isfinite(x[r][want]).all():
            assert tok[r].tolist() == want.tolist(), (r, tok[r], want)
            d = x[r].astype(np.float64)
            ref = d[want] - (d.max() + np.log(np.exp(d - d.max()).sum()))
            assert np.abs(lp[r] - ref).max() <= 2e-6 * (1 + np.abs(ref).max())     # fp32 sum of V terms, log of it
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("N,B,n_heads,context,S_max", [
    (3, 1, 32, 900, 1024), (4, 4, 32, 500, 640),      # just past the rows that the CUDA cores take
    (2, 5, 32, 700, 1024),                            # two rows, more (sequence, head) pairs than SMs
    (5, 5, 32, 1900, 2048), (5, 5, 32, 900, 1024),    # mma.sync a tenth past two CTAs per SM: two chunks from 2048 keys
    (6, 10, 32, 1000, 4096),                          # beyond that from 4096
    (33, 5, 32, 600, 1024), (32, 5, 32, 600, 1024),   # tcgen05: two chunks there with more than 32 rows
])
def test_attention_chunks_beyond_one_round_of_ctas(N, B, n_heads, context, S_max):
    _attention_case(N, B, n_heads, context, S_max)


def test_one_row_of_more_pairs_than_sms_in_two_key_chunks():
    cfg = reduced(T7_EAGLE, 1, K=1, N=1, D=1, topk=1, B=5, H=4096, n_heads=32, F=2048, V=2048, S_max=2048, prompt_len=1900)
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    eng.target_k.copy_(random_kv(cfg, "target_k", cfg.L, DEV))
    eng.target_v.copy_(random_kv(cfg, "target_v", cfg.L, DEV))
    lens = [1900, 1, 64, 700, 1023]
    for b in range(cfg.B):
        orc.target_k[0][b][...] = kv_to_oracle(eng.target_k, 0, b, np.float32)
        orc.target_v[0][b][...] = kv_to_oracle(eng.target_v, 0, b, np.float32)
        orc.seq_len[b] = lens[b]
    eng.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    toks = [[3 + b] for b in range(cfg.B)]
    eng.koala_verify(_tree_arrays(eng, toks, [[-1]] * cfg.B))
    orc.verify([(t, [-1]) for t in toks])
    for b in range(cfg.B):
        assert_close(eng.buffers()["verify_hid"][b:b + 1].cpu().numpy(), orc.verify_hid[b][:1], cfg.dtype, f"hidden {b}")
    assert eng.device_status() == 0 and eng.check_guards()[1] == 0
    eng.close()
