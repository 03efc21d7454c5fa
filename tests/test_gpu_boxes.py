"""GPU parity of the persistent layer kernel on tiles that are boxes of pixels: the whole 2x2 max-pool in its epilogue,
activations copied once for all filter taps, first layers read without packing.  Every box shape, margins behind the last
column, row and image, every epilogue."""
import numpy as np
import pytest
import torch

from oracle import reference as orc
from paper_1711_04713_b200 import binding as B
from tests.test_gpu_layers import _pick_f_out, _rand_q, run_conv_case, run_pool_case
from tests.util import Guards, dev, from_qtensor, stats_tuple, to_qtensor

pytestmark = pytest.mark.gpu
ONE_COPY, UNPACKED = 4, 5          # adaption_debug_get("loop")


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
    (2, 48, 32, 96, 32, 3, 1, 1, 16, 16, 16, True),        # partial blocks, warps that store their own rows
    (17, 40, 40, 160, 64, 3, 1, 1, 16, 8, 16, True),       # ... of boxes with two images
    (64, 48, 48, 64, 64, 3, 1, 1, 8, 8, 8, True),          # many tiles per block
    (5, 64, 64, 64, 64, 3, 1, 1, 16, 16, 16, True),        # with one copy for all taps
    (5, 64, 64, 128, 128, 3, 1, 1, 8, 8, 8, True),
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


# 74 pairs of boxes of 8 x 16 pixels and more: activations copied once for all taps
HALO = [
    # N, H, W, Cin, K, R, pad, nx, nw, n_out, relu
    (5, 64, 64, 64, 64, 3, 1, 16, 16, 16, True),
    (7, 48, 56, 64, 64, 3, 1, 8, 8, 8, True),              # an odd number of boxes
    (5, 64, 62, 64, 128, 3, 1, 16, 16, 16, True),          # two column tiles; columns behind the last
    (5, 63, 64, 64, 100, 3, 1, 16, 16, 16, True),          # the second one ragged; rows behind the last
    (5, 64, 64, 96, 128, 3, 1, 8, 8, 8, True),             # partial k-block
    (5, 64, 64, 160, 72, 3, 1, 8, 8, 8, True),             # two channel blocks, the second partial; a pitch too narrow to stage
    (5, 64, 64, 160, 64, 3, 1, 8, 8, 8, True),             # ... and staged
    (5, 64, 64, 128, 128, 3, 1, 8, 8, 16, False),          # signed outputs of 8-bit operands
    (5, 64, 64, 128, 64, 3, 1, 8, 8, 16, False),           # ... and staged
    (5, 66, 66, 64, 61, 3, 0, 16, 16, 16, True),           # no padding, 64-bit epilogue
    (5, 64, 64, 64, 64, 5, 2, 16, 16, 12, True),
    (5, 65, 65, 64, 64, 2, 0, 16, 16, 16, True),           # even filter
    (3, 112, 112, 64, 64, 3, 1, 16, 16, 16, True),         # several tiles per pair
]
# (no room for the weights beside the staged outputs: the ordinary loop stores this one)
STAGED_ELSEWHERE = [(5, 64, 64, 128, 128, 3, 1, 8, 8, 16, False)]


@pytest.mark.parametrize("case", HALO)
@pytest.mark.parametrize("fast,staged,stochastic", [(1, 1, False), (0, 1, False), (1, 0, False), (1, 1, True)])
def test_one_copy_for_all_taps(case, fast, staged, stochastic):
    N, H, W, Cin, K, R, pad, nx, nw, n_out, relu = case
    B.adaption_debug_set("fast", fast)
    B.adaption_debug_set("staged", staged)
    B.adaption_debug_set("halo", 2)                        # whatever the number of tiles
    run_conv_case(np.random.default_rng(sum(case)), N, H, W, Cin, K, R, pad, 1, nx, nw, n_out, relu, B.ALGO_AUTO,
                  with_q16=False, stochastic_seed=77 if stochastic else None)
    assert (B.adaption_debug_get("loop") == ONE_COPY) == (not staged or case not in STAGED_ELSEWHERE)
    assert B.adaption_debug_get("staged") == (staged if K > 32 and B.pad_to(K, 32) >= (64 if K <= 64 or nx > 8 else 128) else 0)


@pytest.mark.parametrize("pooled", [False, True])
def test_a_16_bit_ring_that_wraps(pooled):
    case = (19, 112, 112, 64, 64, 3, 1, 1, 16, 16, 16, True)
    if pooled:
        run_pool_case(case, False)
    else:
        run_conv_case(np.random.default_rng(3), *case, B.ALGO_AUTO, with_q16=False)
    assert B.adaption_debug_get("loop") == ONE_COPY
    assert B.adaption_debug_get("tiles") >= 74 * 1.5 * B.adaption_debug_get("stages")


# filters whose rows and columns differ, each with its own padding
LONG = [
    # loop, R, S, Cin, K, n_bits
    (ONE_COPY, 3, 5, 64, 64, 16), (ONE_COPY, 5, 3, 64, 64, 8), (ONE_COPY, 1, 9, 128, 128, 8), (ONE_COPY, 3, 2, 96, 48, 16),
    (UNPACKED, 1, 9, 3, 64, 8), (UNPACKED, 9, 1, 3, 64, 16), (UNPACKED, 2, 5, 2, 20, 16), (UNPACKED, 5, 2, 3, 128, 8),
]


@pytest.mark.parametrize("loop,R,S,Cin,K,n_bits", LONG)
def test_filters_that_are_not_square(loop, R, S, Cin, K, n_bits):
    N, cs, pad = 2, 16 if loop == UNPACKED else B.pad_to(Cin, 32), (R // 2, S // 2)
    H, W = 48 + R - 1 - 2 * pad[0], 40 + S - 1 - 2 * pad[1]          # outputs of whole boxes
    rng = np.random.default_rng(10 * R + S)
    xq, wq, bq = _rand_q(rng, (N, H, W, Cin), n_bits, 0.3), _rand_q(rng, (K, R, S, Cin), n_bits), _rand_q(rng, (K,), n_bits)
    fx, fw = n_bits - 3, n_bits - 1
    acc = orc.conv_acc(xq, wq, pad)
    A, f = _pick_f_out(acc, bq, fw, fx + fw, True, n_bits)
    want, cnt = orc.epilogue(acc, bq, fw, fx + fw, True, n_bits, f)
    x, w = to_qtensor(xq.reshape(-1, Cin), n_bits, fx, cs), to_qtensor(wq.reshape(-1, Cin), n_bits, fw, cs)
    guards = Guards()
    y = guards.qtensor(acc.size // K, K, n_bits, f, B.pad_to(K, 32))
    shp = B.adaption_conv_shape(N, H, W, Cin, K, R, S, pad[0], pad[1], 1, 1)
    need = B.adaption_lp_conv_workspace_bytes(shp, x.fmt(), w.fmt(), cs)
    ws = guards.alloc(need) if need else None
    B.adaption_debug_set("halo", 2)
    B.adaption_debug_set("cluster", 0)
    for mode in (B.MODE_RANGE, B.MODE_REQUANT):
        st = B.new_stats()
        B.adaption_lp_conv_fwd(shp, x, w, dev(bq), fw, True, mode, B.ALGO_AUTO, y if mode == B.MODE_REQUANT else None, st, ws)
        assert B.read_stats(st).status == 0 and B.adaption_debug_get("loop") == loop
        if mode == B.MODE_RANGE:
            assert int(B.read_stats(st).max_abs_acc) == A
    assert np.array_equal(from_qtensor(y).reshape(want.shape), want)
    assert stats_tuple(st) == (cnt.zeros, cnt.sat_pos, cnt.sat_neg)
    guards.check()


@pytest.mark.parametrize("Cin,n_bits", [(64, 8), (64, 16), (3, 8), (3, 16)])
@pytest.mark.parametrize("stall_at", [0, 3])
def test_wait_runs_out_and_the_next_call_is_exact(Cin, n_bits, stall_at):
    """The copying warps stop before a stage, with nothing in flight for it: the waits of the issuing warps (two of them at 8
    bits) and of the epilogue run out, the kernel sets the status and returns."""
    case = (8, 112, 112, Cin, 64, 3, 1, 1, n_bits, n_bits, n_bits, True)          # five tiles for every pair or SM
    N, H, W, _, K = case[:5]
    rng, cs = np.random.default_rng(21), 16 if Cin == 3 else Cin
    xq, wq = _rand_q(rng, (N, H, W, Cin), n_bits, 0.4), _rand_q(rng, (K, 3, 3, Cin), n_bits)
    x, w = to_qtensor(xq.reshape(-1, Cin), n_bits, 5, cs), to_qtensor(wq.reshape(-1, Cin), n_bits, 7, cs)
    shp = B.conv_shape(N, H, W, Cin, K, 3, 3, 1, 1)
    y = B.QTensor.empty(N * H * W, K, n_bits, 5, K)
    need = B.adaption_lp_conv_workspace_bytes(shp, x.fmt(), w.fmt(), cs)
    ws = torch.empty(max(need, 16), dtype=torch.uint8, device="cuda")
    B.adaption_debug_set("halo", 2)
    B.adaption_debug_set("timeout_us", 3000)
    B.adaption_debug_set("stall_at", stall_at)
    st = B.new_stats()
    B.adaption_lp_conv_fwd(shp, x, w, None, 0, True, B.MODE_REQUANT, B.ALGO_AUTO, y, st, ws)
    torch.cuda.synchronize()                               # the kernel returned by itself
    assert B.read_stats(st).status == B.ERR_TIMEOUT
    assert B.adaption_debug_get("loop") == (UNPACKED if Cin == 3 else ONE_COPY)
    B.adaption_debug_set("stall_at", -1)
    B.adaption_debug_set("timeout_us", 0)
    run_conv_case(np.random.default_rng(22), 2, *case[1:], B.ALGO_AUTO, with_q16=False, cs=cs)


# 8 bits: two warps issue every other tile's MMAs from one ring, whose slots change hands between them where its depth is no
# multiple of twice a tile's channel blocks.  At least twice as many tiles per pair of SMs as stages.
RINGS = [
    # N, H, W, Cin, K, n_out, pooled, stages when stored
    (16, 112, 112, 128, 128, 8, False, 3),
    (16, 112, 112, 128, 128, 8, True, 5),
    (28, 112, 112, 64, 128, 8, False, 9),
    (22, 112, 112, 128, 64, 8, True, 7),
    (10, 112, 112, 256, 64, 16, False, 3),                  # two channel blocks
    (8, 112, 112, 256, 128, 8, True, 2),
    (8, 112, 112, 512, 64, 8, True, 2),                     # four
]


@pytest.mark.parametrize("N,H,W,Cin,K,n_out,pooled,stages", RINGS)
def test_rings_shared_by_two_issuing_warps(N, H, W, Cin, K, n_out, pooled, stages):
    case = (N, H, W, Cin, K, 3, 1, 1, 8, 8, n_out, True)
    if pooled:
        run_pool_case(case, False)
    else:
        run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_AUTO, with_q16=False)
    assert [B.adaption_debug_get(k) for k in ("loop", "staged", "stages")] == [ONE_COPY, 1, stages]
    assert B.adaption_debug_get("tiles") >= 2 * stages * 74


def test_range_mode_on_a_ring_of_two_stages():
    """Calibration's measuring pass over two channel blocks: nothing is staged, and two stages are left."""
    N, H, W, Cin, K = 8, 112, 112, 256, 128
    rng = np.random.default_rng(5)
    xq, wq, bq = _rand_q(rng, (N, H, W, Cin), 8, 0.4), _rand_q(rng, (K, 3, 3, Cin), 8), _rand_q(rng, (K,), 8)
    x, w = to_qtensor(xq.reshape(-1, Cin), 8, 5, Cin), to_qtensor(wq.reshape(-1, Cin), 8, 7, Cin)
    want = orc.epilogue_range(orc.conv_acc(xq, wq, (1, 1), (1, 1)), bq, 7, 12, True)
    st = B.new_stats()
    B.adaption_lp_conv_fwd(B.conv_shape(N, H, W, Cin, K, 3, 3, 1, 1), x, w, dev(bq), 7, True, B.MODE_RANGE, B.ALGO_AUTO, None,
                           st, None)
    s = B.read_stats(st)
    assert s.status == 0 and int(s.max_abs_acc) == want
    assert [B.adaption_debug_get(k) for k in ("loop", "staged", "stages")] == [ONE_COPY, 0, 2]


# 3x3 over images of 16 columns, 16 rows a tile of a pair: either side of the sizes where one copy for all taps is taken
LINES = [
    # tiles, Cin, K, n_bits, taken
    (74, 64, 64, 16, False), (75, 64, 64, 16, True),
    (74, 128, 128, 8, False), (75, 128, 128, 8, True),
    (148, 64, 64, 8, False), (149, 64, 64, 8, True), (295, 64, 64, 8, True), (296, 64, 64, 8, False),
    (665, 64, 64, 8, False), (666, 64, 64, 8, True),
    (665, 128, 99, 8, False), (666, 128, 99, 8, True),       # 64-bit epilogue, 128 columns
    (295, 64, 72, 12, False), (296, 64, 72, 12, True),       # two column tiles, the output's pitch is narrower than one of 128
    (400, 64, 61, 16, False),
]


@pytest.mark.parametrize("tiles,Cin,K,n_bits,taken", LINES)
def test_one_copy_is_taken_where_it_pays(tiles, Cin, K, n_bits, taken):
    case = (1, 16 * tiles, 16, Cin, K, 3, 1, 1, n_bits, n_bits, n_bits, True)
    run_conv_case(np.random.default_rng(tiles), *case, B.ALGO_AUTO, with_q16=False)
    assert (B.adaption_debug_get("loop") == ONE_COPY) == taken


# first layers over pixels of 16 bytes
TAPS = [
    # N, H, W, Cin, K, R, pad, nx, nw, n_out, relu
    (2, 32, 32, 3, 64, 3, 1, 16, 16, 16, True),
    (2, 32, 32, 3, 64, 3, 1, 8, 8, 8, True),
    (3, 48, 40, 3, 16, 1, 0, 16, 16, 16, True),            # one tap, no margin
    (2, 34, 34, 3, 100, 3, 0, 16, 16, 12, True),           # no padding, 128 columns, ragged
    (1, 65, 63, 1, 32, 2, 0, 16, 16, 16, False),           # even filter, columns and rows behind the last, signed
    (1, 64, 64, 2, 61, 3, 1, 8, 8, 8, True),               # 64-bit epilogue
    (9, 112, 112, 3, 64, 3, 1, 16, 16, 16, True),          # many tiles per block
    (3, 112, 112, 3, 100, 3, 1, 8, 8, 8, True),            # 294 tiles through the 64-bit epilogue: two groups of warps
    (1, 2400, 16, 3, 100, 3, 1, 8, 8, 8, True),            # 300: four
]


@pytest.mark.parametrize("case", TAPS)
@pytest.mark.parametrize("fast,staged,stochastic", [(1, 1, False), (0, 1, False), (1, 0, False), (1, 1, True)])
def test_first_layers_without_packing(case, fast, staged, stochastic):
    N, H, W, Cin, K, R, pad, nx, nw, n_out, relu = case
    B.adaption_debug_set("fast", fast)
    B.adaption_debug_set("staged", staged)
    before = B.adaption_launches()
    run_conv_case(np.random.default_rng(sum(case)), N, H, W, Cin, K, R, pad, 1, nx, nw, n_out, relu, B.ALGO_AUTO,
                  with_q16=False, stochastic_seed=77 if stochastic else None, cs=16)
    assert B.adaption_launches() - before == 2             # (one to measure, one to store)
    assert B.adaption_debug_get("loop") == UNPACKED


@pytest.mark.parametrize("n_bits", [16, 8])
def test_first_layer_with_its_pool(n_bits):
    N, H, W, C, K = 3, 48, 40, 3, 64
    rng = np.random.default_rng(n_bits)
    xq, wq, bq = _rand_q(rng, (N, H, W, C), n_bits, 0.3), _rand_q(rng, (K, 3, 3, C), n_bits), _rand_q(rng, (K,), n_bits)
    fx, fw = n_bits - 3, n_bits - 1
    acc = orc.conv_acc(xq, wq, (1, 1), (1, 1))
    _, f = _pick_f_out(acc, bq, fw, fx + fw, True, n_bits)
    conv_y, cnt = orc.epilogue(acc, bq, fw, fx + fw, True, n_bits, f)
    want = orc.maxpool2x2(conv_y)
    x, w = to_qtensor(xq.reshape(-1, C), n_bits, fx, 16), to_qtensor(wq.reshape(-1, C), n_bits, fw, 16)
    guards = Guards()
    y = guards.qtensor(N * H * W // 4, K, n_bits, f, 64)
    shp = B.conv_shape(N, H, W, C, K, 3, 3, 1, 1)
    need = B.adaption_lp_conv_pool_workspace_bytes(shp, x.fmt(), w.fmt(), y.fmt(), 16, 64, B.ALGO_AUTO)
    ws, st, before = guards.alloc(need), B.new_stats(), B.adaption_launches()
    B.adaption_lp_conv_pool_fwd(shp, x, w, dev(bq), fw, True, B.ALGO_AUTO, y, st, ws)
    assert B.adaption_launches() - before == 1
    assert np.array_equal(from_qtensor(y).reshape(want.shape), want)
    assert stats_tuple(st) == (cnt.zeros, cnt.sat_pos, cnt.sat_neg)
    guards.check()
