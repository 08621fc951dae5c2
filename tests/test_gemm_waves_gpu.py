"""The tensor-core GEMM around one wave of tiles: up to one tile per SM it runs 16 warps a tile, above that four warps a
tile and several tiles an SM."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [0, 1, 200])
@pytest.mark.parametrize("N,K", [(16, 64), (48, 192), (144, 128), (256, 256)])
def test_gemm_on_both_sides_of_a_wave(tiles, N, K):
    import torch
    from paper_1209_6038_gb300 import build, cloak as ck
    build.build()
    M = 128 * (torch.cuda.get_device_properties(0).multi_processor_count + tiles)
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    a = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    b = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16)
    c = torch.full((M, N), float("nan"), device="cuda")
    ck.cloak_mlp_gemm(a, b, c)
    ref = a.float() @ b.float().t()
    # same BF16 inputs, FP32 accumulation: the order of K additions, 2^-24 of the largest partial sums each
    tol = 1e-5 * K ** 0.5 * ref.abs().max().item() + 1e-4
    assert torch.isfinite(c).all()
    assert (c - ref).abs().max().item() <= tol
