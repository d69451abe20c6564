"""The layers that one CTA per 128-token tile takes, above 128 tokens instead of the CTA pairs.  GPU only."""
import pytest
import torch

from test_gemm_choice_cpu import MXFP4_WIDTHS, MXFP8_WIDTHS, ONE_CTA

pytestmark = pytest.mark.gpu

CASES = [(*c, a8) for a8, table in ((False, MXFP4_WIDTHS), (True, MXFP8_WIDTHS)) for c in table]


@pytest.mark.parametrize("S,N,M,width,a8", CASES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
def test_same_bits_as_the_pairs(batq, S, N, M, width, a8, dtype):
    """Every kernel adds the K-steps of an output in the same order, so the choice changes no bit (rows quantised
    and multiplied in parts, as the host entry points do, give the rows of one call)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 148:
        assert batq.batq_debug_gemm_choice(S, M, N, a8, sms) == (ONE_CTA, width)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(S + M)
    ints = lambda lo, hi, shape: torch.randint(lo, hi, shape, generator=gen, dtype=torch.uint8, device="cuda")
    w = batq.batq_weight_import(ints(0, 256, (M, N // 2)), ints(115, 125, (M, N // 32)))
    codes = ints(0, 0x7F if a8 else 256, (S, N if a8 else N // 2))   # E4M3: no NaN code
    scales = ints(121, 133, (batq.batq_sf_bytes(S, N, batq.SF_MMA),))
    fn = batq.batq_gemm_mxfp8_mxfp4 if a8 else batq.batq_gemm_mxfp4
    y = [torch.full((S + 1, (M + 15) // 8 * 8), float("nan"), device="cuda", dtype=dtype) for _ in range(2)]
    for out, kernel in zip(y, (0, 2)):
        batq.batq_debug_force_gemm_kernel(kernel)
        try:
            fn(codes, scales, w, S, out[:S, :M])
        finally:
            batq.batq_debug_force_gemm_kernel(0)
    assert batq.batq_last_device_status() == 0
    assert torch.isnan(y[0][S]).all() and torch.isnan(y[0][:, M:]).all(), "wrote outside [S x M]"
    assert torch.isfinite(y[0][:S, :M]).all() and torch.equal(y[0][:S, :M], y[1][:S, :M])
