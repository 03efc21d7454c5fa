"""GPU parity of the convolutions whose neighbouring output pixels share a row of the GEMM (stride 1, at most 32
input channels) against the CPU oracle, bit-exact: both group sizes, filters that begin before, at and inside a
group, padded channels on both sides, ragged row counts, every epilogue, pooling."""
import numpy as np
import pytest

from paper_1711_04713_b200 import binding as B
from tests import test_gpu_layers as layers
from tests.test_gpu_layers import run_conv_case

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, params=[2, 4], ids=["pairs", "fours"])
def _grouped_whatever_the_number_of_tiles(request):
    B.adaption_debug_set("reset")
    B.adaption_debug_set("cluster", 0)
    B.adaption_debug_set("pixels", request.param)
    yield
    B.adaption_debug_set("reset")


CASES = [
    # N, H, W, Cin, K, R, pad, stride, nx, nw, n_out, relu
    (4, 28, 40, 32, 64, 3, 1, 1, 16, 16, 16, True),       # pairs, three accumulators of 128 columns
    (4, 28, 40, 32, 64, 3, 1, 1, 8, 8, 8, True),          # one accumulator
    (4, 28, 40, 32, 64, 3, 1, 1, 16, 8, 16, False),       # two accumulators, generic epilogue
    (4, 28, 40, 32, 64, 3, 1, 1, 8, 16, 8, True),
    (6, 31, 24, 24, 40, 3, 0, 1, 16, 16, 16, True),       # no padding, 22 wide outputs, padded channels on both sides
    (5, 37, 40, 16, 16, 7, 1, 1, 16, 16, 16, True),       # 36 wide outputs, seven taps (fours do not fit beside the weights)
    (5, 37, 40, 16, 16, 7, 1, 1, 8, 8, 8, True),          # fours
    (5, 37, 38, 16, 24, 5, 2, 1, 16, 16, 12, True),       # ragged rows
    (4, 40, 38, 32, 32, 5, 1, 1, 8, 8, 8, True),          # outputs 36 wide from inputs no multiple of 4
    (6, 33, 64, 20, 128, 3, 1, 1, 8, 8, 8, True),         # 256 columns in pairs, one accumulator
    (6, 33, 64, 20, 64, 5, 2, 1, 8, 8, 8, False),         # 256 columns in fours
    (4, 35, 32, 32, 50, 3, 1, 1, 16, 16, 16, True),       # channels no multiple of 8: generic epilogue
    (6, 40, 42, 30, 32, 2, 0, 1, 16, 16, 16, True),       # two taps (42 wide is not grouped), no tap that all of a four see
    (6, 40, 41, 30, 32, 2, 0, 1, 16, 16, 16, True),       # odd width: not grouped
]


@pytest.mark.parametrize("case", CASES)
def test_conv(case):
    run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_TENSOR, with_q16=False)


@pytest.mark.parametrize("case", CASES[:2] + CASES[4:8])
def test_extremes_int16_copy_and_stochastic_rounding(case):
    run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_TENSOR, extreme=True)
    run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_TENSOR, with_q16=False, with_bias=False)
    run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_TENSOR, with_q16=False, stochastic_seed=77)
    run_conv_case(np.random.default_rng(sum(case)), *case[:-1], False, B.ALGO_TENSOR, with_q16=False, stochastic_seed=78)


@pytest.mark.parametrize("case", [CASES[0], CASES[1], (2, 40, 40, 16, 32, 7, 3, 1, 16, 16, 16, True),
                                  (2, 40, 40, 32, 128, 3, 1, 1, 8, 8, 8, True),
                                  (5, 32, 28, 32, 64, 3, 1, 1, 16, 16, 16, False)])   # signed: pooled ungrouped
def test_pool(case):
    layers.test_conv_with_fused_pool(case, False)


@pytest.mark.parametrize("stall_at", [0, 5])
def test_wait_runs_out_and_the_next_call_is_exact(stall_at):
    """The copy-issuing warps stop before one of their stages (nothing is in flight for it): the kernel reports the
    timeout, drains and returns, and the same layer is exact afterwards."""
    shp = B.conv_shape(4, 40, 40, 32, 64, 3, 3, 1, 1)
    x, w = B.QTensor.empty(4 * 40 * 40, 32, 16, 13, 32), B.QTensor.empty(64 * 9, 32, 16, 15, 32)
    for t in (x, w):
        t.lo.zero_(), t.hi.zero_()
    y, st = B.QTensor.empty(4 * 40 * 40, 64, 16, 5, 64), B.new_stats()
    B.adaption_debug_set("timeout_us", 3000)
    B.adaption_debug_set("stall_at", stall_at)
    B.adaption_lp_conv_fwd(shp, x, w, None, 0, True, B.MODE_REQUANT, B.ALGO_TENSOR, y, st, None)
    assert B.read_stats(st).status == B.ERR_TIMEOUT
    B.adaption_debug_set("stall_at", -1)
    B.adaption_debug_set("timeout_us", 0)
    run_conv_case(np.random.default_rng(5), *CASES[0], B.ALGO_TENSOR, with_q16=False)
