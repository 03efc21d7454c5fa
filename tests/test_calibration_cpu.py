"""Calibration's bookkeeping of the layers' status words without a GPU: the library calls are replaced by ones that
write the counters a device would have written."""
import pytest
import torch

from paper_1711_04713_b200 import binding as B
from paper_1711_04713_b200 import build
from paper_1711_04713_b200.network import LPNetwork, _Layer


class _Stub(LPNetwork):
    """One inner product whose storing passes leave the given counters, pass by pass."""

    def __init__(self, passes):
        self.n_bits, self.device, self.rounding_seed = 16, "cpu", None
        self._all_stats = torch.zeros((2, B.STATS_BYTES), dtype=torch.uint8)
        self._host_stats = torch.zeros_like(self._all_stats)
        self.xq = B.QTensor(1, 16, 16, 16, 0, torch.zeros(16, dtype=torch.uint8))
        self.x_stats = self._all_stats[0]
        L = _Layer("ip", "fc", w=B.QTensor(16, 16, 16, 16, 12, torch.zeros(256, dtype=torch.uint8)), row=1,
                   y=B.QTensor(1, 16, 16, 16, 0, torch.zeros(16, dtype=torch.uint8)), stats=self._all_stats[1])
        self.layers, self.passes = [L], iter(passes)

    def quantize_params(self, measure=True, threshold=0.0):
        pass

    def input_frac_bits(self, threshold, group):
        return 12

    def _quantize_input(self, x_f32):
        pass

    def _to_host(self, src, dst):
        dst.copy_(src)
        return dst

    def width_histogram(self, i):
        return [0, 100] + [0] * (B.HIST_BINS - 2)      # every value fits one bit: the second format differs from the first

    def _run_layer(self, L, x, mode):
        s = B.adaption_stats.from_buffer(L.stats.numpy())
        if mode == B.MODE_RANGE:
            s.max_abs_acc = 1 << 30
        else:
            zeros, status = next(self.passes)
            s.zeros += zeros
            if status:
                s.status = status
        return L.y


@pytest.fixture(autouse=True)
def _library():
    build.build_library()


def test_counts_of_the_second_storing_pass_replace_the_first_ones():
    rec = _Stub([(7, 0), (3, 0)]).calibrate(None, threshold=0.01)
    assert rec[1]["stats"].zeros == 3 and rec[1]["stats"].status == 0


@pytest.mark.parametrize("passes", [[(7, B.ERR_TIMEOUT), (3, 0)], [(7, 0), (3, B.ERR_TIMEOUT)]])
def test_a_time_out_in_either_storing_pass_is_reported(passes):
    with pytest.raises(B.AdaptionError) as e:
        _Stub(passes).calibrate(None, threshold=0.01)
    assert e.value.status == B.ERR_TIMEOUT and "fc" in str(e.value)
