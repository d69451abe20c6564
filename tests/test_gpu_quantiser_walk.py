"""The order in which the tensor-core quantiser's CTAs go through an activation tensor.  GPU only."""
import pytest
import torch

from paper_2603_16590_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,N", [(128 * 299 + 1, 128),       # one strip of 4 blocks: every CTA walks it
                                 (128 * 23 + 5, 5 * 128),    # single strips, every unit a CTA of its own
                                 (128 * 120 + 5, 5 * 128),   # walked in step, three CTAs without units
                                 (128 * 20 - 3, 41 * 128),   # walked in step, 25 CTAs on the last two rows
                                 (128 * 70, 6 * 128 - 32),   # pairs of strips, the last one part-filled
                                 (128 * 50, 26 * 128),       # pairs, eight CTAs on the last five rows
                                 (128 * 37 + 1, 64 * 128),   # groups of four
                                 (128 * 3, 145 * 128),       # three units for all CTAs but three
                                 (128 * 3 - 7, 200 * 128),   # more strips than CTAs
                                 (257, 149 * 128 + 32)])
@pytest.mark.parametrize("fp8", [False, True], ids=["mxfp4", "mxfp8"])
def test_every_unit_is_quantised_once(batq, S, N, fp8):
    """Rows are independent: the whole tensor has the codes and scale bytes of its 128-row pieces, each of which
    is one row of units (and checked against the oracle by the parity tests)."""
    t = synth.make_transform(N, 7, "baseline")
    tr = batq.batq_transform_create(N, t.left, t.right, t.clip_lo, t.clip_hi)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(S + N)
    x = torch.randn((S, N), generator=gen, device="cuda").to(torch.bfloat16)
    fn = batq.batq_quantize_act_mxfp8 if fp8 else batq.batq_quantize_act

    def run(rows):
        codes = torch.full((rows.shape[0] + 1, N if fp8 else N // 2), 0xA5, dtype=torch.uint8, device="cuda")
        scales = torch.full((rows.shape[0], N // 32), 0xA5, dtype=torch.uint8, device="cuda")
        fn(tr, rows, codes, scales, batq.SF_ROWMAJOR)
        assert (codes[-1] == 0xA5).all(), "wrote past the codes"
        return codes[:-1], scales

    batq.batq_debug_force_quantizer(2)
    try:
        codes, scales = run(x)
        for r in range(0, S, 128):
            c, s = run(x[r:r + 128])
            assert torch.equal(codes[r:r + 128], c) and torch.equal(scales[r:r + 128], s)
    finally:
        batq.batq_debug_force_quantizer(0)
    assert batq.batq_last_device_status() == 0


@pytest.mark.parametrize("units", [1, 2, 3, 4, 5, 7, 13])
@pytest.mark.parametrize("fp8", [False, True], ids=["mxfp4", "mxfp8"])
def test_buffers_are_reused_in_turn(batq, units, fp8):
    """`units` units for every CTA but the last ones, around the counts of its buffers in tensor memory (two of X, three
    of accumulators), of input stages (three) and of staging tiles (four).  Units differ in magnitude, and
    the reference quantises one unit a CTA, which reuses no buffer: whole numbers, no tolerance."""
    n, sms = 128, torch.cuda.get_device_properties(0).multi_processor_count
    s = 128 * sms * units - 3
    t = synth.make_transform(n, 7, "baseline")
    tr = batq.batq_transform_create(n, t.left, t.right, t.clip_lo, t.clip_hi)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(units)
    x = torch.randn((s, n), generator=gen, device="cuda")
    tile = torch.arange(s, device="cuda") // 128
    x = (x * torch.exp2((tile * 7 % 11 - 5).float())[:, None]).to(torch.bfloat16)
    fn = batq.batq_quantize_act_mxfp8 if fp8 else batq.batq_quantize_act

    def run(rows):
        codes = torch.zeros((rows.shape[0], n if fp8 else n // 2), dtype=torch.uint8, device="cuda")
        scales = torch.zeros((rows.shape[0], n // 32), dtype=torch.uint8, device="cuda")
        fn(tr, rows, codes, scales, batq.SF_ROWMAJOR)
        return codes, scales

    batq.batq_debug_force_quantizer(2)
    try:
        whole = run(x)
        parts = [run(p) for p in x.split(128 * sms)]
    finally:
        batq.batq_debug_force_quantizer(0)
    assert batq.batq_last_device_status() == 0
    for got, want in zip(whole, zip(*parts)):
        assert torch.equal(got, torch.cat(want))
