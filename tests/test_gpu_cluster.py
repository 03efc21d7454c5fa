"""GPU parity of the layers that run as one thread-block cluster per output tile (few output tiles:
small batches, deep layers, inner products) against the CPU oracle, bit-exact, at the edges of its
tiles: pixel boxes that cross image borders, several images per tile, partial channel blocks, every
cluster size and column width, reductions shorter than the cluster, pitches wider than the tiles."""
import numpy as np
import pytest
import torch

from oracle import reference as orc
from paper_1711_04713_b200 import binding as B
from tests.test_gpu_layers import _pick_f_out, _rand_q, run_conv_case, run_ip_case
from tests.util import Guards, dev, from_qtensor, stats_tuple, to_qtensor

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cluster_kernel_everywhere():
    B.adaption_debug_set("reset")
    B.adaption_debug_set("cluster", 2)
    yield
    B.adaption_debug_set("reset")


CONV = [
    # N, H, W, Cin, K, R, pad, stride, nx, nw, n_out, relu
    (1, 14, 14, 512, 96, 3, 1, 1, 16, 16, 16, True),     # deep layer of one image, four channel blocks per tap
    (3, 12, 12, 20, 50, 5, 0, 1, 16, 16, 16, True),      # two 8 x 8 images per tile, a half-filled last tile
    (5, 7, 9, 96, 40, 3, 1, 1, 12, 12, 12, False),       # pitch 96: the copies' boxes reach past the channels
    (2, 11, 13, 160, 33, 3, 1, 2, 16, 16, 8, True),      # 128 + 32 channels, stride 2, odd sizes, odd N
    (1, 5, 150, 64, 24, 3, 1, 1, 16, 8, 16, True),       # rows wider than a tile
    (2, 9, 9, 32, 17, 1, 0, 1, 8, 16, 12, False),        # 1x1, 32-byte k-blocks, a single k-block
    (1, 23, 17, 64, 130, 4, 2, 3, 8, 8, 8, True),        # stride 3, even filter, single int8 pass
    (4, 4, 4, 256, 16, 3, 0, 1, 4, 4, 4, True),          # 2 x 2 outputs, four images per tile
]


@pytest.mark.parametrize("case", CONV)
@pytest.mark.parametrize("with_q16", [False, True])
def test_conv(case, with_q16):
    run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_AUTO, with_q16=with_q16)


@pytest.mark.parametrize("size", [1, 2, 4, 8])
@pytest.mark.parametrize("bn", [16, 48, 112, 128])
def test_every_cluster_size_and_width(size, bn):
    B.adaption_debug_set("cluster_size", size)
    B.adaption_debug_set("cluster_bn", bn)
    case = (2, 10, 10, 128, 128 if bn == 128 else bn + 8, 3, 1, 1, 16, 16, 16, True)
    run_conv_case(np.random.default_rng(size + bn), *case, B.ALGO_AUTO, with_q16=False)
    run_ip_case(np.random.default_rng(size * bn), bn - 3, 1300, 150, 16, 16, 16, False, B.ALGO_AUTO, with_q16=False)


@pytest.mark.parametrize("case", [(1, 4096, 300, 16, 16, 16, True), (5, 1000, 33, 16, 8, 12, False),
                                  (17, 33, 129, 8, 16, 16, True), (64, 2000, 10, 8, 8, 8, True),
                                  (129, 640, 256, 16, 16, 16, False), (3, 64, 1, 16, 16, 16, True)])
def test_ip(case):
    for with_q16 in (False, True):
        run_ip_case(np.random.default_rng(sum(case)), *case, B.ALGO_AUTO, with_q16=with_q16)
    run_ip_case(np.random.default_rng(sum(case) + 1), *case, B.ALGO_AUTO, stochastic_seed=77 + case[0])


@pytest.mark.parametrize("case", [CONV[0], CONV[3], CONV[6]])
def test_stochastic_rounding_and_extremes(case):
    run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_AUTO, stochastic_seed=0xABCDEF01234 + case[4])
    run_conv_case(np.random.default_rng(sum(case)), *case, B.ALGO_AUTO, extreme=True, with_bias=False)


@pytest.mark.parametrize("case", [
    (1, 14, 14, 512, 96, 3, 1, 1, 16, 16, 16, True), (3, 12, 12, 20, 50, 5, 0, 1, 16, 16, 16, True),
    (2, 6, 134, 64, 24, 3, 1, 1, 16, 16, 12, False), (7, 4, 4, 32, 16, 3, 0, 1, 8, 8, 8, True),
])
def test_conv_with_pool(case):
    N, H, W, Cin, K, R, pad, stride, nx, nw, n_out, relu = case
    rng = np.random.default_rng(sum(case))
    cs = B.pad_to(Cin, 32)
    xq, wq, bq = _rand_q(rng, (N, H, W, Cin), nx, 0.4), _rand_q(rng, (K, R, R, Cin), nw), _rand_q(rng, (K,), nw)
    fx, fw = nx - 3, nw - 1
    acc = orc.conv_acc(xq, wq, (pad, pad), (stride, stride))
    _, f_out = _pick_f_out(acc, bq, fw, fx + fw, relu, n_out)
    conv_y, cnt = orc.epilogue(acc, bq, fw, fx + fw, relu, n_out, f_out)
    want = orc.maxpool2x2(conv_y)
    x, w = to_qtensor(xq.reshape(-1, Cin), nx, fx, cs), to_qtensor(wq.reshape(-1, Cin), nw, fw, cs)
    for with_q16, pitch in ((False, B.pad_to(K, 16)), (True, B.pad_to(K, 16) + 160)):
        guards = Guards()
        y = guards.qtensor(want.size // K, K, n_out, f_out, pitch, with_q16=with_q16)
        shp = B.conv_shape(N, H, W, Cin, K, R, R, pad, stride)
        need = B.adaption_lp_conv_pool_workspace_bytes(shp, x.fmt(), w.fmt(), y.fmt(), cs, pitch)
        st = B.new_stats()
        B.adaption_lp_conv_pool_fwd(shp, x, w, dev(bq), fw, relu, B.ALGO_AUTO, y, st, guards.alloc(need))
        assert np.array_equal(from_qtensor(y).reshape(want.shape), want)
        assert y.padding_is_zero()
        assert stats_tuple(st) == (cnt.zeros, cnt.sat_pos, cnt.sat_neg)
        guards.check()


def test_pitch_beyond_the_last_tile_is_zeroed():
    rng = np.random.default_rng(8)
    xq, wq = _rand_q(rng, (3, 200), 16, 0.4), _rand_q(rng, (20, 200), 16)
    want, _ = orc.epilogue(orc.ip_acc(xq, wq), None, 0, 29, True, 16, 6)
    guards = Guards()
    y = guards.qtensor(3, 20, 16, 6, 304)
    B.adaption_lp_ip_fwd(3, 200, 20, to_qtensor(xq, 16, 14), to_qtensor(wq, 16, 15), None, 0, True, B.MODE_REQUANT,
                         B.ALGO_AUTO, y, B.new_stats(), None)
    assert np.array_equal(from_qtensor(y), want) and y.padding_is_zero()
    guards.check()


def test_output_pitch_beyond_32_bits():
    """Rows 2^31 + 16 elements apart: the outputs are stored where they belong (outputs of 8 bits, two rows)."""
    rng = np.random.default_rng(12)
    xq, wq = _rand_q(rng, (2, 64), 8, 0.4), _rand_q(rng, (8, 64), 8)
    want, _ = orc.epilogue(orc.ip_acc(xq, wq), None, 0, 13, True, 8, 2)
    pitch = (1 << 31) + 16
    y = B.QTensor(2, 8, pitch, 8, 2, torch.full((2 * pitch,), 0x3C, dtype=torch.uint8, device="cuda"))
    B.adaption_lp_ip_fwd(2, 64, 8, to_qtensor(xq, 8, 6), to_qtensor(wq, 8, 7), None, 0, True, B.MODE_REQUANT, B.ALGO_AUTO,
                         y, B.new_stats(), None)
    got = torch.stack([y.lo[:8], y.lo[pitch:pitch + 8]]).cpu().numpy()
    assert np.array_equal(got.view(np.int8), want)


def test_device_side_wait_runs_out():
    """The copying warps stop before their second stage with nothing in flight; the waits of the others
    run out, the kernel says so in the stats word and returns, and the next call is exact."""
    rng = np.random.default_rng(9)
    x, w = to_qtensor(_rand_q(rng, (8, 4096), 16), 16, 13), to_qtensor(_rand_q(rng, (200, 4096), 16), 16, 15)
    y, st = B.QTensor.empty(8, 200, 16, 3), B.new_stats()
    B.adaption_debug_set("timeout_us", 3000)
    B.adaption_debug_set("stall_at", 1)
    ws = torch.empty(8 * 200 * 8, dtype=torch.uint8, device="cuda")
    B.adaption_lp_ip_fwd(8, 4096, 200, x, w, None, 0, True, B.MODE_REQUANT, B.ALGO_AUTO, y, st, ws)
    torch.cuda.synchronize()
    assert B.read_stats(st).status == B.ERR_TIMEOUT
    B.adaption_debug_set("stall_at", -1)
    B.adaption_debug_set("timeout_us", 0)
    run_ip_case(np.random.default_rng(10), 8, 4096, 200, 16, 16, 16, True, B.ALGO_AUTO)
