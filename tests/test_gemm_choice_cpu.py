"""Which kernel a GEMM call takes, checked without a GPU."""
import pytest

from paper_2603_16590_b200 import binding as B

ONE_CTA, PAIRS, WIDE, SWAPPED = 1, 2, 3, 4


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


def test_arguments_out_of_range():
    for args in ((0, 128, 128), (128, 0, 128), (128, 128, 0), (128, 128, 96)):
        with pytest.raises(ValueError):
            B.batq_debug_gemm_choice(*args, mxfp8=True)
    with pytest.raises(ValueError):
        B.batq_debug_gemm_choice(128, 128, 40)
    with pytest.raises(ValueError):
        B.batq_debug_gemm_choice(128, 128, 128, sm_count=1)
