"""Which kernel a GEMM call takes, checked without a GPU."""
import pytest

from paper_2603_16590_b200 import binding as B

ONE_CTA, PAIRS, WIDE, SWAPPED = 1, 2, 3, 4

# tokens, input channels, features, tile width of the layers that one CTA per 128-token tile takes on 148 SMs
MXFP4_WIDTHS = [(129, 512, 1024, 64),       # half a wave of 128-wide tiles, short K
                (300, 4096, 200, 64),       # 16 K-steps and few tiles, a part-filled column
                (128, 4096, 1024, 64),
                (300, 4352, 200, 128),      # one K-step more
                (100, 3584, 4616, 128),     # up to 128 tokens: long K, though half a wave
                (385, 256, 4736, 128),      # 37 x 4 tiles of 128: a wave to the last SM
                (385, 256, 4744, 128),      # one column more, on short K
                (1000, 1024, 4100, 128),    # four K-steps, two waves
                (2100, 256, 12288, 192),    # one K-step, seven waves
                (512, 6144, 7104, 192),     # 24 K-steps, the last with one wave of 192-wide tiles
                (600, 1280, 7168, 256),     # most of a wave of 256-wide tiles
                (600, 1280, 10240, 192),    # two nearly full waves of 192-wide ones
                (333, 1280, 37888, 256),    # three row tiles, three full waves of 256-wide ones
                (257, 1280, 24328, 256)]    # two waves, the last column part-filled
MXFP8_WIDTHS = [(129, 512, 1024, 128), (300, 4352, 200, 128), (385, 256, 4736, 128),
                (1000, 1024, 2300, 128),    # 18 x 8 tiles
                (333, 1280, 37888, 256), (384, 640, 12296, 256), (257, 384, 24328, 256)]


@pytest.mark.parametrize("s,n,m,kernel", [
    # few K-steps: what the wide kernel's only accumulator waits for is most of a tile.  Layers of 1024 -> 8192, pair / wide:
    # 13.6 / 14.6 us at 640 tokens, 14.1 / 14.7 at 768, 15.4 / 16.7 at 896, 15.4 / 16.8 at 1024; 1024 -> 4096 16.1 / 17.7
    (640, 1024, 8192, PAIRS), (768, 1024, 8192, PAIRS), (896, 1024, 8192, PAIRS), (1024, 1024, 8192, PAIRS),
    (2048, 1024, 4096, PAIRS),
    # 31.6 / 34.1 and 30.2 / 30.5: one wide tile takes as long as two of 192 and 256
    (200, 3584, 37888, PAIRS), (256, 4096, 28672, PAIRS),
    # many tiles a pair on few K-steps: 42.8 / 35.9, 29.9 / 26.9
    (3000, 512, 16384, WIDE), (2048, 512, 16384, WIDE),
    # 188 / 177, 32.5 / 29.0, 28.2 / 27.3
    (3000, 13824, 5120, WIDE), (1024, 5120, 5120, WIDE), (896, 2560, 10240, WIDE)])
def test_w4a8_pair_kernels(s, n, m, kernel):
    assert B.batq_debug_gemm_choice(s, m, n, mxfp8=True)[0] == kernel


@pytest.mark.parametrize("a8,table", [(False, MXFP4_WIDTHS), (True, MXFP8_WIDTHS)], ids=["mxfp4", "mxfp8"])
def test_one_cta_per_tile(a8, table):
    for s, n, m, width in table:
        assert B.batq_debug_gemm_choice(s, m, n, mxfp8=a8) == (ONE_CTA, width), (s, n, m)


@pytest.mark.parametrize("s,n,m,a8,kernel", [
    (512, 6400, 7104, False, PAIRS),     # 25 K-steps
    (333, 1280, 36600, False, WIDE),     # three row tiles, the last wave short of full
    (512, 1280, 37888, False, WIDE),     # four row tiles
    (2048, 4096, 28672, False, WIDE), (2048, 4096, 4096, False, PAIRS), (8192, 3584, 37888, False, WIDE),
    (2048, 4096, 28672, True, WIDE), (257, 4096, 128, True, ONE_CTA),
    (16, 4096, 4096, True, SWAPPED), (128, 4096, 12288, True, ONE_CTA)])
def test_other_kernels(s, n, m, a8, kernel):
    assert B.batq_debug_gemm_choice(s, m, n, mxfp8=a8)[0] == kernel


def test_arguments_out_of_range():
    for args in ((0, 128, 128), (128, 0, 128), (128, 128, 0), (128, 128, 96)):
        with pytest.raises(ValueError):
            B.batq_debug_gemm_choice(*args, mxfp8=True)
    with pytest.raises(ValueError):
        B.batq_debug_gemm_choice(128, 128, 40)
    with pytest.raises(ValueError):
        B.batq_debug_gemm_choice(128, 128, 128, sm_count=1)
