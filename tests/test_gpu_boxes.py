"""GPU parity of the persistent layer kernel on tiles that are boxes of pixels, where its epilogue makes the whole 2x2 max-pool:
every box shape, margins behind the last column, row and image, every epilogue."""
import pytest

from paper_1711_04713_b200 import binding as B
from tests.test_gpu_layers import run_pool_case

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _default_overrides():
    B.adaption_debug_set("reset")
    yield
    B.adaption_debug_set("reset")


CASES = [
    # N, H, W, Cin, K, R, pad, stride, nx, nw, n_out, relu
    (2, 48, 32, 64, 64, 3, 1, 1, 16, 16, 16, True),        # 16 x 8 pixels, two accumulator sets
    (17, 40, 40, 64, 64, 3, 1, 1, 8, 8, 8, True),          # 8 x 8 x 2, the last boxes half empty
    (2, 32, 24, 128, 128, 3, 1, 1, 16, 16, 16, True),      # 8 x 16 or 8 x 8 x 2, pair tiles
    (8, 28, 28, 128, 192, 3, 1, 1, 16, 16, 16, True),      # 4 x 4 x 8, two column tiles, the second ragged
    (31, 14, 14, 96, 128, 3, 1, 1, 16, 16, 12, True),      # 2 x 2 x 32, one image missing, partial k-blocks
    (32, 14, 14, 128, 256, 3, 1, 1, 8, 8, 8, True),        # 256-column pair tiles of bytes
    (32, 10, 6, 128, 512, 1, 0, 1, 8, 8, 8, True),         # two of them
    (2, 62, 32, 64, 120, 3, 1, 1, 16, 16, 16, False),      # signed outputs, rows behind the last
    (2, 46, 32, 64, 61, 3, 1, 1, 16, 16, 16, True),        # channel count no multiple of 8: 64-bit epilogue
    (2, 32, 32, 96, 20, 3, 1, 1, 16, 8, 16, True),         # 32-column tiles, mixed widths
    (2, 34, 34, 64, 64, 3, 0, 1, 16, 16, 8, True),         # no padding, bytes from 16-bit operands
    (64, 48, 48, 64, 64, 3, 1, 1, 8, 8, 8, True),          # many tiles per block
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("fast", [0, 1])
def test_whole_windows_pooled_in_the_epilogue(case, fast):
    B.adaption_debug_set("cluster", 0)
    B.adaption_debug_set("fast", fast)
    before = B.adaption_launches()
    run_pool_case(case, False)
    # (three calls that run: the whole layer, its convolution and its pooling; the last has nothing left to do)
    assert B.adaption_launches() - before == 2


def test_an_int16_copy_is_pooled_by_its_own_pass():
    B.adaption_debug_set("cluster", 0)
    before = B.adaption_launches()
    run_pool_case(CASES[0], True)
    assert B.adaption_launches() - before == 4
