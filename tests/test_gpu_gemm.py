"""The library's matrix multiplies (tensor-core and CUDA-core paths) against a float64 product."""
import numpy as np
import pytest
import torch

from paper_2408_08146_b200 import koala_gemm_bf16
from workloads.generate import normal_tensor

pytestmark = pytest.mark.gpu

SHAPES = [  # (tokens, out features, in features)
    (1, 128, 64), (10, 4096, 4096), (16, 256, 128), (17, 200, 192), (60, 1536, 4096),
    (64, 384, 11008), (40, 640, 5120), (256, 256, 1024), (300, 256, 512), (6, 32000, 4096),
    (250, 1280, 2048)]      # 256-row weight tiles (N = 256), several of them, ragged token tile


def _inputs(M, N, K):
    x = normal_tensor(7, f"x{M}.{N}.{K}", (M, K), 1.0, 0.0, torch.bfloat16, "cuda:0")
    w = normal_tensor(8, f"w{M}.{N}.{K}", (N, K), 0.02, 0.0, torch.bfloat16, "cuda:0")
    ref = x.double().cpu().numpy() @ w.double().cpu().numpy().T
    return x, w, ref


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("split", [0, 1, 3])
def test_tensor_core_gemm(shape, split):
    M, N, K = shape
    if split > K // 64:
        pytest.skip("fewer K blocks than splits")
    x, w, ref = _inputs(M, N, K)
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    y = koala_gemm_bf16(x, w, True, split, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0, "a bounded device-side wait ran out"
    err = np.abs(y.cpu().numpy() - ref).max()
    assert err <= 2e-5 * np.sqrt(K) + 1e-6, f"max err {err}"      # fp32 accumulation of K products


@pytest.mark.parametrize("shape", SHAPES[:8])
def test_cuda_core_gemm(shape):
    M, N, K = shape
    x, w, ref = _inputs(M, N, K)
    y = koala_gemm_bf16(x, w, False)
    torch.cuda.synchronize()
    err = np.abs(y.cpu().numpy() - ref).max()
    assert err <= 2e-5 * np.sqrt(K) + 1e-6, f"max err {err}"


@pytest.mark.parametrize("M", [1, 7, 8, 9, 17, 24, 25, 40, 55, 72, 100, 112])
@pytest.mark.parametrize("N,K", [(12288, 4096), (200, 192), (1000, 2816), (22016, 512)])
def test_token_tiles_of_a_pair_in_eights(M, N, K):
    """Tiles that are and are not whole sixteens, with ragged weight tiles and split sums."""
    xf = normal_tensor(9, f"xe{M}.{N}.{K}", (M, K), 1.0, 0.0, torch.float32, "cuda:0")
    w = normal_tensor(8, f"we{M}.{N}.{K}", (N, K), 0.02, 0.0, torch.bfloat16, "cuda:0")
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    y = koala_gemm_bf16(hi, w, True, 0, status, lo)
    assert int(status.item()) == 0
    ref = ((hi.double() + lo.double()) @ w.double().T).cpu().numpy()
    err = np.abs(y.cpu().numpy() - ref).max()
    assert err <= 2e-5 * np.sqrt(K) + 1e-6, f"max err {err}"      # fp32 accumulation of K products


@pytest.mark.parametrize("M", [1, 7, 8, 9, 17, 24, 25, 40, 55, 72, 100, 112])
def test_token_tiles_in_eights_with_shared_sums(M):
    """172 tiles of 64 K blocks, dealt to two CTAs per SM: tiles shared by several, two accumulator buffers."""
    test_token_tiles_of_a_pair_in_eights(M, 22016, 4096)


@pytest.mark.parametrize("shape", [(10, 4096, 4096), (60, 1536, 4096), (100, 256, 11008), (130, 384, 512),
                                   (256, 256, 1024), (128, 512, 4096), (200, 1024, 2048), (120, 768, 1024)])
@pytest.mark.parametrize("tc", [True, False], ids=["tensor_core", "cuda_core"])
def test_gemm_with_activation_pairs(shape, tc):
    """fp32 activations given as a bf16 value + bf16 rounding residual: the product must be that of
    the pair's sum (about 16 significant bits of the activations)."""
    M, N, K = shape
    xf = normal_tensor(9, f"xf{M}.{N}.{K}", (M, K), 1.0, 0.0, torch.float32, "cuda:0")
    w = normal_tensor(8, f"w{M}.{N}.{K}", (N, K), 0.02, 0.0, torch.bfloat16, "cuda:0")
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    y = koala_gemm_bf16(hi, w, tc, 0, status, x_lo=lo)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref_pair = (hi.double() + lo.double()).cpu().numpy() @ w.double().cpu().numpy().T
    ref_full = xf.double().cpu().numpy() @ w.double().cpu().numpy().T
    assert np.abs(y.cpu().numpy() - ref_pair).max() <= 2e-5 * np.sqrt(K) + 1e-6
    # and the pair is a much better stand-in for the fp32 activations than plain bf16
    err_pair = np.abs(y.cpu().numpy() - ref_full).max()
    err_bf16 = np.abs(hi.double().cpu().numpy() @ w.double().cpu().numpy().T - ref_full).max()
    assert err_pair < 0.05 * err_bf16 + 1e-5


@pytest.mark.parametrize("shape", [(113, 1536, 1024), (128, 11008, 512), (129, 1024, 4096), (200, 700 * 16, 256),
                                   (256, 5120, 5120), (256, 512, 13824)])
def test_cta_pair_form_and_one_cta_form_agree(shape):
    """113 to 256 rows as a pair of activations: the CTA-pair kernel (default) and the one-CTA kernel
    (tuning key 17 = 1) both give the product of the pair's sum; ragged last tiles, one or many
    K blocks, one or many tiles per cluster."""
    from paper_2408_08146_b200 import binding
    lib = binding.load_library()
    M, N, K = shape
    xf = normal_tensor(11, f"xf{M}.{N}.{K}", (M, K), 1.0, 0.0, torch.float32, "cuda:0")
    w = normal_tensor(12, f"w{M}.{N}.{K}", (N, K), 0.02, 0.0, torch.bfloat16, "cuda:0")
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16)
    ref = (hi.double() + lo.double()).cpu().numpy() @ w.double().cpu().numpy().T
    outs = []
    try:
        for off in (0, 1):
            lib.koala_set_tuning(17, off)
            status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
            y = koala_gemm_bf16(hi, w, True, 0, status, x_lo=lo)
            torch.cuda.synchronize()
            assert int(status.item()) == 0
            outs.append(y.cpu().numpy())
            assert np.abs(outs[-1] - ref).max() <= 2e-5 * np.sqrt(K) + 1e-6
    finally:
        lib.koala_set_tuning(17, 0)
    assert np.abs(outs[0] - outs[1]).max() <= 4e-5 * np.sqrt(K) + 1e-6


@pytest.mark.parametrize("shape", [(140, 1024, 512), (257, 1536, 512), (300, 700 * 16, 256), (512, 1024, 4096),
                                   (1000, 640, 1024), (600, 512, 11008)])
def test_cta_pairs_with_token_tiles_of_any_width(shape):
    """More than 128 rows: token tiles of a multiple of 32 rows (ragged last tile), several of them sharing
    the deal of K blocks; the consumer's count of partial sums follows the row and the column."""
    M, N, K = shape
    xf = normal_tensor(13, f"xf{M}.{N}.{K}", (M, K), 1.0, 0.0, torch.float32, "cuda:0")
    w = normal_tensor(14, f"w{M}.{N}.{K}", (N, K), 0.02, 0.0, torch.bfloat16, "cuda:0")
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16)
    ref = (hi.double() + lo.double()).cpu().numpy() @ w.double().cpu().numpy().T
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    y = koala_gemm_bf16(hi, w, True, 0, status, x_lo=lo)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert np.abs(y.cpu().numpy() - ref).max() <= 2e-5 * np.sqrt(K) + 1e-6      # fp32 accumulation of K products


@pytest.mark.parametrize("shape", [(1, 9, 4), (2, 8, 128), (3, 250, 68), (4, 17, 772), (9, 64, 1028), (17, 33, 2052),
                                   (31, 2500, 256), (5, 20, 66)])
@pytest.mark.parametrize("pair", [False, True])
def test_cuda_core_gemm_of_few_rows(shape, pair):
    """Rows per warp 2 to 16, K with and without a tail past the pre-read weights, K not a multiple of four
    (the staged kernel), features that leave the last block partly empty."""
    M, N, K = shape
    xf = normal_tensor(15, f"xf{M}.{N}.{K}", (M, K), 1.0, 0.0, torch.float32, "cuda:0")
    w = normal_tensor(16, f"w{M}.{N}.{K}", (N, K), 0.02, 0.0, torch.bfloat16, "cuda:0")
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16) if pair else None
    full = hi.double() + lo.double() if pair else hi.double()
    y = koala_gemm_bf16(hi, w, False, 0, None, x_lo=lo)
    torch.cuda.synchronize()
    ref = full.cpu().numpy() @ w.double().cpu().numpy().T
    assert np.abs(y.cpu().numpy() - ref).max() <= 2e-5 * np.sqrt(K) + 1e-6


@pytest.mark.parametrize("shape", [(16, 4096, 4096), (17, 4096, 4096), (17, 1024, 4096), (24, 1001, 4100), (128, 512, 1024), (128, 1000, 1028)])
def test_cuda_core_gemm_on_both_sides_of_the_small_kernel(shape):
    M, N, K = shape
    x, w, ref = _inputs(M, N, K)
    err = np.abs(koala_gemm_bf16(x, w, False).cpu().numpy() - ref).max()
    assert err <= 2e-5 * np.sqrt(K) + 1e-6, f"max err {err}"      # fp32 accumulation of K products
