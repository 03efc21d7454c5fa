"""GPU parity of the quantizer where a tensor is cut into chunks of padded rows or shares a launch with
others: chunk edges inside a block of four elements, rows longer than a chunk, unaligned inputs, special
values at the edges of the range; deterministic and stochastic rounding."""
import numpy as np
import pytest
import torch

from oracle import reference as orc
from oracle import stochastic as orc_st
from paper_1711_04713_b200 import binding as B
from tests.util import Guards, dev, from_qtensor, q16_of, stats_tuple

pytestmark = pytest.mark.gpu

# outer, inner, pitch: one element per row; odd rows whose chunks start anywhere in a block of four;
# exactly one chunk, one row more; a pitch of a whole chunk; rows of several segments
SHAPES = [(700, 1, 16), (513, 3, 16), (1025, 7, 32), (64, 50, 64), (65, 50, 64), (3, 4081, 4096), (2, 4097, 4112),
          (3, 9001, 9008), (5, 17, 12304), (300, 16, 16)]


def _values(rng, shape, n_bits, f):
    x = (rng.standard_normal(shape) * 2.0 ** (n_bits - 1 - f) * 0.6).astype(np.float32)
    grid = (rng.integers(-(1 << n_bits), 1 << n_bits, shape) / 2).astype(np.float32) * np.float32(2.0 ** -f)
    x = np.where(rng.random(shape) < 0.2, grid, x).astype(np.float32)         # grid values and ties
    special = np.array([np.nan, np.inf, -np.inf, -0.0, 1e-45, -1e-45, 3e38, -2.0 ** -60], np.float32)
    k = min(x.size, special.size)
    x.ravel()[rng.choice(x.size, k, replace=False)] = special[:k]
    return x


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n_bits,f", [(16, 12), (8, 5)])
@pytest.mark.parametrize("offset", [0, 3])
@pytest.mark.parametrize("relu", [False, True])
def test_rows(shape, n_bits, f, offset, relu):
    outer, inner, pitch = shape
    rng = np.random.default_rng(outer + inner + offset)
    x = _values(rng, (outer, inner), n_bits, f)
    src = torch.zeros(outer * inner + offset, device="cuda")
    src[offset:] = dev(x.ravel())
    xr = np.where(x > 0, x, 0).astype(np.float32) if relu else x
    for seed in (None, 0x1234567890 + outer):
        guards = Guards()
        y = guards.qtensor(outer, inner, n_bits, f, pitch, with_q16=True)
        st = B.new_stats()
        if seed is None:
            B.adaption_lp_act(src[offset:], None, outer, inner, relu, y, None, B.ROUND_DETERMINISTIC, st)
            want, cnt = orc.quantize(xr, n_bits, f)
            cnt = (cnt.zeros, cnt.sat_pos, cnt.sat_neg)
        else:
            B.adaption_quantize_stochastic(src[offset:], outer, inner, y, seed, relu, None, st)
            want, cnt = orc_st.quantize_stochastic(x, n_bits, f, seed, relu)
        assert np.array_equal(from_qtensor(y), want)
        assert np.array_equal(q16_of(y), want)
        assert y.padding_is_zero()
        assert stats_tuple(st) == tuple(cnt)
        guards.check()


# (the last four: the widest pitch at which the rows of a run are told apart by a multiplication, and the pitches
# from which a run of as many rows has too many vectors for it)
@pytest.mark.parametrize("shape", [(76001, 17, 32), (40003, 50, 64), (20001, 256, 272), (160001, 5, 16),
                                   (1030, 1, 32752), (1030, 1, 33024), (1030, 1, 65520), (230, 5, 74144)])
def test_rows_of_a_large_tensor_stochastic(shape):
    """Tensors large enough for a warp to assemble several rows at a time: odd row lengths, the longest rows,
    a last run of rows that is not full."""
    outer, inner, pitch = shape
    rng = np.random.default_rng(outer)
    x = _values(rng, (outer, inner), 16, 12)
    want, cnt = orc_st.quantize_stochastic(x, 16, 12, 99 + inner, False)
    for offset in (0, 1):
        src = torch.zeros(outer * inner + offset, device="cuda")
        src[offset:] = dev(x.ravel())
        guards = Guards()
        y = guards.qtensor(outer, inner, 16, 12, pitch)
        st = B.new_stats()
        B.adaption_quantize_stochastic(src[offset:], outer, inner, y, 99 + inner, False, None, st)
        assert np.array_equal(from_qtensor(y), want)
        assert y.padding_is_zero()
        assert stats_tuple(st) == tuple(cnt)
        guards.check()


@pytest.mark.parametrize("shape", [(460001, 3, 16), (460001, 9, 16), (230001, 17, 32)])
@pytest.mark.parametrize("relu", [False, True])
def test_blocks_of_several_chunks(shape, relu):
    """Tensors of more chunks than there are blocks, without a generator; the last chunk is not full."""
    outer, inner, pitch = shape
    x = _values(np.random.default_rng(outer), (outer, inner), 16, 12)
    want, cnt = orc.quantize(np.where(x > 0, x, 0).astype(np.float32) if relu else x, 16, 12)
    guards = Guards()
    y = guards.qtensor(outer, inner, 16, 12, pitch)
    st = B.new_stats()
    B.adaption_lp_act(dev(x), None, outer, inner, relu, y, None, B.ROUND_DETERMINISTIC, st)
    assert np.array_equal(from_qtensor(y), want)
    assert y.padding_is_zero()
    assert stats_tuple(st) == (cnt.zeros, cnt.sat_pos, cnt.sat_neg)
    guards.check()


@pytest.mark.parametrize("stochastic", [False, True])
def test_many_tensors_in_one_launch(stochastic):
    """More tensors than one launch takes, dense and padded in turn, small and large, formats on host and device."""
    rng = np.random.default_rng(3)
    shapes = [(1 + (7 * k) % 90, [16, 50, 3, 128, 1][k % 5]) for k in range(45)] + [(3000, 64), (9, 5000)]
    guards, entries, host, seeds = Guards(), [], [], []
    for k, (outer, inner) in enumerate(shapes):
        n = 16 if k % 3 else 8
        f = n - 3
        x = _values(rng, (outer, inner), n, f)
        y = guards.qtensor(outer, inner, n, f if k % 4 else 0, None, with_q16=k % 2 == 0)
        fmt = None if k % 4 else torch.tensor([n, f], dtype=torch.int32, device="cuda")
        entries.append((dev(x), outer, inner, y, fmt))
        host.append((x, n, f))
        seeds.append(0xFFFFFFFF00000000 + 1000 * k)
    items = B.quantize_items(entries)
    if stochastic:
        B.adaption_quantize_batch_stochastic(items, seeds)
    else:
        B.adaption_quantize_batch(items)
    for (x, n, f), (_, _, _, y, _), seed in zip(host, entries, seeds):
        want = orc_st.quantize_stochastic(x, n, f, seed, False)[0] if stochastic else orc.quantize(x, n, f)[0]
        assert np.array_equal(from_qtensor(y), want)
        assert y.padding_is_zero()
    guards.check()


def test_a_batch_without_tensors():
    """No array at all is fine for no tensors, and an invalid argument of the library for any."""
    B.adaption_quantize_batch(None, 0)
    with pytest.raises(B.AdaptionError) as e:
        B.adaption_quantize_batch(None, 1)
    assert e.value.status == B.ERR_INVALID_ARG


@pytest.mark.parametrize("n_bits,f", [(16, 14), (8, 7), (4, 3)])
def test_stochastic_decisions_next_to_the_draw(n_bits, f):
    """Values whose fraction lies on, next to, or a last place of single precision away from the draw that decides them,
    of both signs and all magnitudes down to 2^-40: the rounding in single precision takes no other side than exact arithmetic."""
    n, seed = 1 << 16, 0xABCDEF0123456789
    rng = np.random.default_rng(n_bits)
    r = orc_st.draws(n, seed).astype(np.float64)
    whole = rng.integers(-3, 4, n).astype(np.float64)
    y = (whole + (r + rng.integers(-1, 3, n)) * 2.0 ** -32).astype(np.float32)
    tiny = (rng.choice([-1.0, 1.0], n) * rng.uniform(1, 2, n) * 2.0 ** rng.integers(-40, 0, n)).astype(np.float32)
    y = np.where(rng.random(n) < 0.25, tiny, y).astype(np.float32)
    y = np.nextafter(y, y + rng.integers(-1, 2, n).astype(np.float32)).astype(np.float32)
    x = (y * np.float32(2.0 ** -f)).reshape(-1, 64)                       # (exact: a power of two)
    guards = Guards()
    q, st = guards.qtensor(x.shape[0], 64, n_bits, f, 64), B.new_stats()
    B.adaption_quantize_stochastic(dev(x), x.shape[0], 64, q, seed, False, None, st)
    want, cnt = orc_st.quantize_stochastic(x, n_bits, f, seed, False)
    assert np.array_equal(from_qtensor(q), want)
    assert stats_tuple(st) == tuple(cnt)
    guards.check()
