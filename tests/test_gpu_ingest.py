"""Prompt ingestion in wide forwards (koala_ingest, behind Koala.prefill) against the oracle's chunk by
chunk ingestion: caches of the target and of the head, lengths, the pending state the first iteration
starts from, and the acceptance counters."""
import numpy as np
import pytest
import torch

from tests.harness import kv_to_oracle, make_pair, tok_list
from tests.parity import assert_close
from workloads import T7_EAGLE, T7_MEDUSA, TINY_EAGLE, TINY_MEDUSA, reduced
from workloads.generate import prompts

pytestmark = pytest.mark.gpu

TINY = [  # config, prompt lengths, chunk
    (TINY_EAGLE, [64], 15), (TINY_EAGLE, [2], 1), (TINY_EAGLE, [33], 32), (TINY_EAGLE.with_(K=1), [130], 7),
    (TINY_EAGLE.with_(K=0), [40], 9), (TINY_MEDUSA, [50], 12), (TINY_EAGLE.with_(S_max=320), [300], 15),
    (TINY_EAGLE.with_(B=3), [60, 17, 41], 15), (TINY_EAGLE.with_(B=2, S_max=256), [190, 100], 14)]


def _check(eng, orc, cfg, n, dt):
    assert eng.seq_len.cpu().tolist() == orc.seq_len == n
    for b in range(cfg.B):
        for l in range(cfg.L):
            assert_close(kv_to_oracle(eng.target_k, l, b, dt)[:n[b]], orc.target_k[l][b][:n[b]], cfg.dtype, f"K {l}.{b}")
            assert_close(kv_to_oracle(eng.target_v, l, b, dt)[:n[b]], orc.target_v[l][b][:n[b]], cfg.dtype, f"V {l}.{b}")
        if cfg.head_kind == 0:
            held = n[b] - int(eng.buffers()["n_pend"][b])        # the last part's entries come with the first draft
            for j in range(cfg.K):
                assert_close(kv_to_oracle(eng.draft_k, j, b, dt)[:held], orc.draft_k[j][b][:held], cfg.dtype, f"head K {j}.{b}")
                assert_close(kv_to_oracle(eng.draft_v, j, b, dt)[:held], orc.draft_v[j][b][:held], cfg.dtype, f"head V {j}.{b}")


@pytest.mark.parametrize("case", TINY, ids=[f"{c.head_kind}-{n}-{k}" for c, n, k in TINY])
def test_tiny_prompts_free_running(case):
    cfg, n, chunk = case
    cfg = cfg.with_(prompt_len=max(n), seed=31)
    eng, orc, _ = make_pair(cfg)
    rng = np.random.default_rng(sum(n))
    pr = [rng.integers(0, cfg.V, m) for m in n]
    eng.prefill(pr, chunk)
    orc.prefill(pr, min(chunk, cfg.N))          # the library cuts chunks to at most N tokens
    _check(eng, orc, cfg, n, np.float64)
    got = eng.koala_accept_stats(cfg.N)
    pad = lambda a: (list(a) + [0] * cfg.N)[:cfg.N]
    assert got == (pad(orc.alpha_hits), pad(orc.alpha_trials))
    for _ in range(2):
        tk, ln = tok_list(*eng.step())
        rt, rl = orc.step()
        assert [list(x) for x in tk] == [list(x) for x in rt] and list(ln) == list(rl)
    assert eng.device_status() == 0
    assert eng.check_guards()[1] == 0
    eng.close()


@pytest.mark.parametrize("kind,n,chunk", [("eagle", [20], 16), ("eagle", [200], 60), ("eagle", [333, 150], 64),
                                          ("eagle", [600, 450, 70], 64), ("medusa", [150], 64)])
def test_7b_shaped_prompts(kind, n, chunk):
    """bf16, tensor-core attention and CTA-pair multiplies over blocks of several sequences (one or two
    forwards, ragged last blocks)."""
    base = T7_EAGLE if kind == "eagle" else T7_MEDUSA
    cfg = reduced(base, 2, B=len(n), S_max=768, prompt_len=max(n), seed=32, **({"K": 1} if kind == "eagle" else {}))
    eng, orc, _ = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    rng = np.random.default_rng(sum(n))
    pr = [rng.integers(0, cfg.V, m) for m in n]
    eng.prefill(pr, chunk)
    orc.prefill(pr, min(chunk, cfg.N))          # the library cuts chunks to at most N tokens
    _check(eng, orc, cfg, n, np.float32)
    bufs = eng.buffers()
    for b in range(cfg.B):
        k = int(bufs["n_pend"][b])
        assert_close(bufs["pend_hid"][b, :k].cpu().numpy(), orc.pend_hid[b][:k], cfg.dtype, f"pending hidden {b}")
    assert eng.device_status() == 0
    assert eng.check_guards()[1] == 0
    eng.close()


@pytest.mark.parametrize("n", [[261], [270], [258, 100]])
def test_prompts_whose_rows_are_not_whole_groups_of_a_thread(n):
    """261 rows (three blocks of 87), 270, and 360 with rows of a second sequence."""
    test_7b_shaped_prompts("eagle", n, 64)


@pytest.mark.parametrize("n", [[429], [381, 102]])
def test_prompts_whose_last_row_is_alone_in_its_thread(n):
    """From about 370 rows on a thread of the rotary kernel takes two: 429 rows, 483 with rows of a second sequence."""
    test_7b_shaped_prompts("eagle", n, 64)


def test_a_prompt_beyond_the_capacity_is_reported():
    cfg = TINY_EAGLE.with_(S_max=100)
    eng, _, _ = make_pair(cfg)
    eng.prefill([np.arange(140) % cfg.V], 15)
    assert eng.device_status() == 3
    assert eng.check_guards()[1] == 0
    eng.close()


def test_prompts_of_an_engine_on_another_stream():
    """The engine's stream is busy when prefill returns, and the caller's stream takes up freed memory at once: the
    prompt's tokens stay until the engine has read them."""
    cfg = TINY_EAGLE.with_(S_max=256, prompt_len=200, seed=33)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        eng, orc, _ = make_pair(cfg)
    side.synchronize()
    pr = prompts(cfg)
    eng.prefill([pr[0][::-1]], 15)                          # kernels loaded: the next call does not wait for the device
    torch.cuda.synchronize()
    eng.seq_len.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)                      # about 0.1 s
    eng.prefill(pr, 15)                                     # the current stream is the default one
    other = [torch.full((1, 200), 7, dtype=torch.int32, device="cuda:0") for _ in range(8)]
    torch.cuda.synchronize()
    assert all(int(t.sum()) == 1400 for t in other)
    orc.prefill(pr, 15)
    _check(eng, orc, cfg, [200], np.float64)
    assert eng.device_status() == 0
    eng.close()
