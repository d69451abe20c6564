"""The slots of tensor memory through which the CTA-pair GEMMs' scale factors go.  GPU only."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_steps", [1, 2, 3, 4, 5, 6, 11])
@pytest.mark.parametrize("kernel,width", [(2, 0), (2, 192), (2, 256), (3, 0), (3, 128), (3, 256), (3, 320), (3, 448)])
@pytest.mark.parametrize("a8", [False, True], ids=["mxfp4", "mxfp8"])
def test_same_bits_as_a_slot_for_every_stage(batq, k_steps, kernel, width, a8):
    """Against one CTA per tile, which has a slot for every ring stage: around the counts of slots (two, three, four) and of
    ring stages (four, five), over several tiles a pair, with a ragged edge.  Scales differ from K-step to K-step by
    up to 2^11, so a step multiplied with another's scales shows; the K-steps are added in the same order, so all bits
    agree."""
    S, M, N = 2300, 8960 + 72, (128 if a8 else 256) * k_steps
    gen = torch.Generator(device="cuda")
    gen.manual_seed(k_steps)
    ints = lambda lo, hi, shape: torch.randint(lo, hi, shape, generator=gen, dtype=torch.uint8, device="cuda")
    w = batq.batq_weight_import(ints(0, 256, (M, N // 2)), ints(115, 127, (M, N // 32)))
    codes = ints(0, 0x7F if a8 else 256, (S, N if a8 else N // 2))   # E4M3: no NaN code
    scales = ints(121, 133, (batq.batq_sf_bytes(S, N, batq.SF_MMA),))
    fn = batq.batq_gemm_mxfp8_mxfp4 if a8 else batq.batq_gemm_mxfp4
    y = [torch.full((S, M), float("nan"), device="cuda") for _ in range(2)]
    for out, (k, bn) in zip(y, ((kernel, width), (1, 128))):
        batq.batq_debug_force_gemm_kernel(k)
        batq.batq_debug_force_tile_width(bn)
        try:
            fn(codes, scales, w, S, out)
        finally:
            batq.batq_debug_force_gemm_kernel(0)
            batq.batq_debug_force_tile_width(0)
    assert batq.batq_last_device_status() == 0
    assert torch.isfinite(y[1]).all() and torch.equal(y[0], y[1])
