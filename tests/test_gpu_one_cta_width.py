"""The layers that one CTA per 128-token tile takes, above 128 tokens instead of the CTA pairs.  GPU only."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,M,N", [(129, 1024, 512),      # half a wave of 128-wide tiles, short K: 64-wide
                                   (300, 200, 4096),      # the same with long K: 128-wide, a part-filled column
                                   (100, 4616, 3584),     # up to 128 tokens: long K, 128-wide though half a wave
                                   (128, 1024, 4096),     # 16 K-steps and few tiles: 64-wide
                                   (385, 4736, 256),      # 37 x 4 tiles of 128: a wave to the last SM
                                   (385, 4744, 256),      # one column more: 192-wide
                                   (1000, 4100, 1024),    # four K-steps, two waves: 128-wide
                                   (2100, 12288, 256),    # one K-step, seven waves: 192-wide
                                   (512, 7104, 6144),     # 24 K-steps, the last with 192-wide tiles
                                   (600, 7168, 1280),     # most of a wave of 256-wide tiles
                                   (600, 10240, 1280),    # two nearly full waves of 192-wide ones
                                   (333, 37888, 1280)])   # three row tiles, three full waves of 256-wide ones
@pytest.mark.parametrize("a8", [False, True], ids=["mxfp4", "mxfp8"])
def test_same_bits_as_the_pairs(batq, S, M, N, a8):
    """Every kernel adds the K-steps of an output in the same order, so the choice changes no bit (rows quantised
    and multiplied in parts, as the host entry points do, give the rows of one call)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(S + M)
    ints = lambda lo, hi, shape: torch.randint(lo, hi, shape, generator=gen, dtype=torch.uint8, device="cuda")
    w = batq.batq_weight_import(ints(0, 256, (M, N // 2)), ints(115, 125, (M, N // 32)))
    codes = ints(0, 0x7F if a8 else 256, (S, N if a8 else N // 2))   # E4M3: no NaN code
    scales = ints(121, 133, (batq.batq_sf_bytes(S, N, batq.SF_MMA),))
    fn = batq.batq_gemm_mxfp8_mxfp4 if a8 else batq.batq_gemm_mxfp4
    y = [torch.full((S + 1, M + 8), float("nan"), device="cuda") for _ in range(2)]
    for out, kernel in zip(y, (0, 2)):
        batq.batq_debug_force_gemm_kernel(kernel)
        try:
            fn(codes, scales, w, S, out[:S, :M])
        finally:
            batq.batq_debug_force_gemm_kernel(0)
    assert batq.batq_last_device_status() == 0
    assert torch.isnan(y[0][S]).all() and torch.isnan(y[0][:, M:]).all(), "wrote outside [S x M]"
    assert torch.isfinite(y[0][:S, :M]).all() and torch.equal(y[0][:S, :M], y[1][:S, :M])
