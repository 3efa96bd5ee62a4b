"""The TMA path over runs (unpadded rasters of any width) and device rasters
copied into aligned staging rows first: sizes around a 2 KiB piece and a
16-member box, planes with and without row padding, and a persistent CTA that
takes several tiles, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


def shifted(m: np.ndarray, shift: int, pitch: int, gap: int):
    """Device copy at element offset `shift`, rows `pitch` and members pitch * h + gap elements apart, ones between."""
    n, h, w = m.shape
    stride = pitch * h + gap
    buf = torch.full((shift + (n - 1) * stride + (h - 1) * pitch + w,), 1,
                     dtype=torch.uint8 if m.dtype == np.uint8 else torch.float32, device="cuda")
    view = buf.as_strided((n, h, w), (stride, pitch, 1), storage_offset=shift)
    view.copy_(torch.from_numpy(m))
    return view


# runs: w * h a multiple of 16 (mask bytes) and of 4 (depths); then layouts that are not: shift, pad, gap
LAYOUTS = [(16, 1, 0, 0, 0), (13, 16, 0, 0, 0), (64, 32, 0, 0, 0), (1, 2064, 0, 0, 0), (130, 48, 0, 0, 16), (1501, 16, 0, 0, 0),
           (1024, 400, 0, 0, 0), (13, 7, 0, 0, 0), (33, 16, 1, 0, 0), (100, 36, 0, 3, 0), (48, 20, 5, 0, 1)]


@pytest.mark.parametrize("count_bits", [16, 32])
@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS)
def test_masks(w, h, shift, pad, gap, count_bits):
    with binding.Composite(w, h, read_path="tma", count_bits=count_bits) as comp:
        for n in (1, 15, 16, 40, 300):
            m = synth.scramble_nonzero(synth.random_masks(n, n, h, w), 9)
            dev = shifted(m, shift, w + pad, gap)
            comp.clear()
            comp.add(dev)
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m))
            comp.remove(dev[: n // 2])
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m[n // 2:]))
        # a member that is not there
        comp.clear()
        comp.add(shifted(np.zeros((1, h, w), np.uint8), shift, w + pad, gap))
        comp.remove(shifted(np.ones((1, h, w), np.uint8), shift, w + pad, gap))
        with pytest.raises(binding.CompositeError) as e:
            comp.sync()
        assert e.value.code == binding.CPT_EUNDERFLOW


@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS)
def test_depths(w, h, shift, pad, gap):
    for path in ("tma", "texture"):
        with binding.Composite(w, h, read_path=path, mode="mean_depth") as comp:
            for n in (1, 15, 17, 200):
                d = synth.random_depths(n, n, h, w)
                dev = shifted(d, shift, w + pad, gap)
                comp.clear()
                comp.add(dev)
                comp.add(dev[:1])
                want = oracle.mean_depth(np.concatenate([d, d[:1]]))
                # n + 1 depths below 4, fewer than n + 2 roundings of sums below 4 (n + 1), then a division
                assert np.abs(comp.render_host()["mean"].astype(np.float64) - want).max() <= 4.0 * (n + 3) * 2.0 ** -24
