"""The linear read path where its launches change shape: rasters at every byte
alignment read in place, ragged and single-pixel rows, memory that ends with
the last pixel, and the edges of the split into slices and slabs, against the
CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


def shifted(m: np.ndarray, shift: int, pitch: int, gap: int):
    """Device copy at byte (or word) offset `shift`, rows `pitch` and members pitch * h + gap elements apart, ones between."""
    n, h, w = m.shape
    stride = pitch * h + gap
    span = (n - 1) * stride + (h - 1) * pitch + w
    buf = torch.full((shift + span,), 1, dtype=torch.uint8 if m.dtype == np.uint8 else torch.float32, device="cuda")
    view = buf[shift:].as_strided((n, h, w), (stride, pitch, 1), storage_offset=shift)
    view.copy_(torch.from_numpy(m))
    return view


# members: the edges of a load batch (8, 4), of slices (16, 32, 64) and of a slab (255)
MEMBERS = [1, 4, 7, 9, 15, 16, 33, 64, 255, 256, 300]
LAYOUTS = [(1, 1, 0, 0, 0), (3, 2, 5, 0, 0), (15, 3, 1, 0, 0), (16, 4, 8, 0, 0), (17, 5, 0, 1, 0), (40, 3, 3, 2, 7),
           (64, 2, 0, 0, 16), (100, 37, 13, 0, 0), (1501, 11, 9, 3, 1), (48, 600, 4, 0, 0)]


@pytest.mark.parametrize("count_bits", [16, 32])
@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS)
def test_masks_at_any_alignment(w, h, shift, pad, gap, count_bits):
    with binding.Composite(w, h, count_bits=count_bits) as comp:
        for n in MEMBERS:
            m = synth.scramble_nonzero(synth.random_masks(n, n, h, w), 3)
            dev = shifted(m, shift, w + pad, gap)
            comp.clear()
            comp.add(dev)
            c = oracle.count(m)
            got = comp.render_host()
            np.testing.assert_array_equal(got["counts"].astype(np.int64), c)
            np.testing.assert_array_equal(got["bucket"], oracle.bucket(c, n))
            comp.remove(dev[: n // 2])
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m[n // 2:]))


@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS)
def test_depths_at_any_alignment(w, h, shift, pad, gap):
    with binding.Composite(w, h, mode="mean_depth") as comp:
        for n in (1, 4, 9, 16, 40, 130):
            d = synth.random_depths(n, n, h, w)
            comp.clear()
            comp.add(shifted(d, shift, w + pad, gap))
            err = np.abs(comp.render_host()["mean"].astype(np.float64) - oracle.mean_depth(d)).max()
            # float32 sums of n depths below 4, each addition rounded once: at most n * 2^-24 * 4 n / n per pixel
            assert err <= 4.0 * n * 2.0 ** -24


@pytest.mark.parametrize("w,h,shift", [(64, 8, 0), (61, 9, 3)])
def test_depth_sums_of_many_members_round_seldom(w, h, shift):
    n = 1000
    d = synth.random_depths(5, n, h, w)
    with binding.Composite(w, h, mode="mean_depth") as comp:
        comp.add(shifted(d, shift, w, 0))
        err = np.abs(comp.render_host()["mean"].astype(np.float64) - oracle.mean_depth(d)).max()
    # a value of at most 4 n meets 3 roundings in a tree of 8, 8 in a block, 16 blocks, 3 slices, and the division
    assert err <= 4.0 * (3 + 8 + 16 + 3 + 1) * 2.0 ** -24


@pytest.mark.parametrize("count_bits", [16, 32])
@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS + [(8, 4, 3, 1, 0), (33, 3, 4, 3, 4), (200, 9, 8, 7, 8), (1856, 5, 0, 0, 0)])
def test_bit_rows_at_any_alignment(w, h, shift, pad, gap, count_bits):
    with binding.Composite(w, h, count_bits=count_bits, mask_format="bits") as comp:
        for n in MEMBERS:
            m = synth.random_masks(n, n, h, w)
            packed = synth.pack_masks(m)
            dev = shifted(packed, shift, packed.shape[2] + pad, gap)
            comp.clear()
            comp.add(dev)
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m))
            comp.remove(dev[: n // 2])
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m[n // 2:]))


def test_more_members_than_the_slabs_of_one_launch():
    n, limit = 65535 * 255 + 300, 65535 * 255
    base = torch.zeros((n, 1, 1), dtype=torch.uint8, device="cuda")
    base[::3] = 1
    with binding.Composite(1, 1, count_bits=32) as comp:
        comp.add(base)
        assert int(comp.render_host()["counts"][0, 0]) == (n + 2) // 3
    assert n > limit
