"""How exact the sums inside the tensor core are: it adds by truncation, so the error of a product grows with
the number of MMAs that one accumulator takes.  Forms are compared with each other on the same inputs and
with float64."""
import math

import numpy as np
import pytest
import torch

from paper_2408_08146_b200 import binding, koala_gemm_bf16
from tests.harness import make_pair
from workloads import T7_EAGLE, reduced
from workloads.generate import normal_tensor, random_kv, uniform_ints

pytestmark = pytest.mark.gpu


def _pair(M, N, K):
    x = normal_tensor(51, f"x{M}.{N}.{K}", (M, K), 1.0, 0.0, torch.float32, "cuda:0")
    w = normal_tensor(52, f"w{M}.{N}.{K}", (N, K), 0.02, 0.0, torch.bfloat16, "cuda:0")
    hi = x.to(torch.bfloat16)
    lo = (x - hi.float()).to(torch.bfloat16)
    return hi, lo, w, (hi.double() + lo.double()) @ w.double().T


def _rel(y, ref):
    return float((y.double() - ref).norm() / ref.norm())


@pytest.fixture
def short_sums():
    lib = binding.load_library()
    lib.koala_set_tuning(23, 1)
    yield
    lib.koala_set_tuning(23, 0)


@pytest.mark.parametrize("M,N,K", [(65, 512, 1024), (80, 256, 64), (100, 200, 4096), (112, 4096, 1024), (129, 1000, 704),
                                   (200, 11000, 1024), (256, 3072, 4096), (257, 512, 128), (300, 1500, 1088),
                                   (512, 768, 11008), (1000, 384, 2048), (1024, 130, 4096)])
def test_short_chains_against_float64(short_sums, M, N, K):
    """Ragged weight tiles and token tiles, runs that end inside a chain; 32 MMAs per accumulator."""
    hi, lo, w, ref = _pair(M, N, K)
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    y = koala_gemm_bf16(hi, w, True, 0, status, lo)
    assert int(status.item()) == 0
    # a truncated step is off by at most 2^-23 of its running sum (half of that on average): 32 steps per chain,
    # one rounding of 2^-24 per chain (K / 256 of them) and per partial sum (at most 12)
    steps = 2 * 32 + K / 256 + 12
    assert float((y.double() - ref).abs().max()) <= steps * 2.0 ** -24 * float(ref.abs().max())
    assert _rel(y, ref) <= 32 * 2.0 ** -24
    assert torch.equal(y, koala_gemm_bf16(hi, w, True, 0, status, lo))


@pytest.mark.parametrize("M,N,K,split", [(257, 27648, 5120, 2), (300, 27648, 5120, 2), (300, 1024, 2816, 1), (512, 22016, 4096, 1)])
def test_several_token_tiles_sum_no_more_than_with_one_cta_per_tile(M, N, K, split):
    """split: the factor of the form with one CTA per tile at this size."""
    hi, lo, w, ref = _pair(M, N, K)
    auto, one = koala_gemm_bf16(hi, w, True, 0, None, lo), koala_gemm_bf16(hi, w, True, split, None, lo)
    assert _rel(auto, ref) <= 1.02 * _rel(one, ref)


@pytest.mark.parametrize("n", [100, 200, 509])
def test_prompt_forwards_are_as_exact_as_their_parts(n):
    """The first layer's values are one product of exactly known inputs, rounded to bf16: the share that differs
    from the rounded float64 product measures the product's error.  A wide forward may have no more of it
    than the same prompt verified and accepted part by part."""
    cfg = reduced(T7_EAGLE, 1, K=1, N=64, V=4096, S_max=640, prompt_len=n, seed=53)
    eng, _, store = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    tok = uniform_ints(54, "tokens", n, 0, cfg.V)
    x = store["embed"][torch.from_numpy(tok.astype(np.int64)).cuda()].double()
    x = x * torch.rsqrt((x * x).mean(-1, keepdim=True) + cfg.rms_eps) * store["layers.0.attn_norm"].double()
    want = (x @ store["layers.0.wv"].double().T).to(torch.bfloat16).view(n, cfg.n_heads, cfg.head_dim)

    def differing():
        got = eng.target_v[0, 0, :, :n].permute(1, 0, 2)
        return float((got != want).float().mean())

    for part in np.array_split(tok, -(-n // 64)):
        tree = eng.chain_tree([part])
        eng.koala_verify(tree)
        eng.koala_accept(tree[2])
    parts = differing()
    eng.seq_len.zero_()
    eng.target_v.zero_()
    eng.prefill([tok], 64)
    assert differing() <= parts
    assert eng.device_status() == 0
    eng.close()


def test_tcgen05_attention_is_about_as_exact_as_mma_sync():
    """One layer over 64 chained rows on a context of 2000, against float64 on the keys and values as stored; the same rows
    by either kernel (tuning key 9).  P V is added in one truncating accumulator per chunk in the one and in several in the
    other; a probability is a value rounded to bf16 and a rounded residual in both.  Cutting the value part off instead makes the
    residual, and its rounding error, up to twice as large: 1.24 times the whole layer's error; rounded it is 1.02 times."""
    n, ctx, dev = 64, 2000, "cuda:0"
    cfg = reduced(T7_EAGLE, 1, K=1, N=n, H=1024, n_heads=8, F=2048, V=2048, S_max=2176, prompt_len=ctx, seed=55)
    eng, _, store = make_pair(cfg, oracle_dtype=np.float32, cache_host=False)
    eng.target_k.copy_(random_kv(cfg, "target_k", 1, dev))
    eng.target_v.copy_(random_kv(cfg, "target_v", 1, dev))
    tok = uniform_ints(56, "tokens", n, 0, cfg.V)
    tree = eng.chain_tree([tok])
    lib, hid = binding.load_library(), []
    try:
        for min_rows in (16, 129):
            lib.koala_set_tuning(9, min_rows)
            eng.seq_len.fill_(ctx)
            eng.koala_verify(tree)
            hid.append(eng.buffers()["verify_hid"][:n].double())
    finally:
        lib.koala_set_tuning(9, 16)
    w = lambda name: store[name].double()
    rms = lambda x, gain: x * torch.rsqrt((x * x).mean(-1, keepdim=True) + cfg.rms_eps) * w(gain)
    x = w("embed")[torch.from_numpy(tok.astype(np.int64)).to(dev)]
    q = (rms(x, "layers.0.attn_norm") @ w("layers.0.wq").T).view(n, cfg.n_heads, cfg.head_dim)
    pos = ctx + torch.arange(n, device=dev, dtype=torch.float64)
    ang = pos[:, None, None] * cfg.rope_base ** (-2.0 * torch.arange(64, device=dev, dtype=torch.float64) / 128)
    c, s = torch.cos(ang).float().double(), torch.sin(ang).float().double()
    q = torch.cat([q[..., :64] * c - q[..., 64:] * s, q[..., 64:] * c + q[..., :64] * s], -1)
    score = torch.einsum("rhd,hkd->hrk", q, eng.target_k[0, 0, :, :ctx + n].double()) / math.sqrt(128)
    hidden = torch.arange(ctx + n, device=dev)[None] > pos[:, None]
    p = torch.softmax(score.masked_fill(hidden[None], float("-inf")), -1)
    x = x + torch.einsum("hrk,hkd->rhd", p, eng.target_v[0, 0, :, :ctx + n].double()).reshape(n, cfg.H) @ w("layers.0.wo").T
    h = rms(x, "layers.0.ffn_norm")
    x = x + (torch.nn.functional.silu(h @ w("layers.0.w_gate").T) * (h @ w("layers.0.w_up").T)) @ w("layers.0.w_down").T
    ref = rms(x, "final_norm")
    assert _rel(hid[0], ref) <= 1.12 * _rel(hid[1], ref)      # half way between the two
    assert eng.device_status() == 0
    eng.close()
