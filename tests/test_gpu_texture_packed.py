"""The texture path's bit-packed arrays: widths around a texel (64 pixels), a
conversion tile (512 x 8) and its narrow forms, device rasters at any
alignment converted in place, members around a conversion thread's eight
layers, a fold step's 16 and an array's fill, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu

LAYOUTS = [(1, 1, 0, 0, 0), (15, 9, 3, 2, 1), (16, 8, 0, 0, 0), (63, 17, 1, 0, 0), (64, 16, 8, 0, 0), (65, 3, 0, 15, 16),
           (129, 33, 5, 0, 3), (511, 8, 0, 1, 0), (512, 9, 0, 0, 0), (513, 7, 2, 0, 0), (1501, 11, 9, 3, 1)]


def shifted(m: np.ndarray, shift: int, pitch: int, gap: int):
    """Device copy at byte offset `shift`, rows `pitch` and members pitch * h + gap bytes apart, ones between."""
    n, h, w = m.shape
    stride = pitch * h + gap
    buf = torch.full((shift + (n - 1) * stride + (h - 1) * pitch + w,), 1, dtype=torch.uint8, device="cuda")
    view = buf.as_strided((n, h, w), (stride, pitch, 1), storage_offset=shift)
    view.copy_(torch.from_numpy(m))
    return view


@pytest.mark.parametrize("count_bits", [16, 32])
@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS)
def test_device_rasters_at_any_alignment(w, h, shift, pad, gap, count_bits):
    with binding.Composite(w, h, read_path="texture", count_bits=count_bits) as comp:
        for n in (1, 7, 8, 17, 64, 255, 300):
            m = synth.scramble_nonzero(synth.random_masks(n, n, h, w), 9)
            dev = shifted(m, shift, w + pad, gap)
            comp.clear()
            comp.add(dev)
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m))
            comp.remove(dev[: n // 2])
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m[n // 2:]))


@pytest.mark.parametrize("kind", ["device", "pinned"])
@pytest.mark.parametrize("chunk", [1, 3, 16, 255])
def test_chunks_fill_an_array(chunk, kind):
    w, h, n = 200, 21, 40
    m = synth.random_masks(chunk, n, h, w)
    src = torch.from_numpy(m).cuda() if kind == "device" else torch.from_numpy(m).pin_memory()
    for k in (1, 2, 3):
        with binding.Composite(w, h, read_path="texture", staging_buffers=k, chunk_members=chunk) as comp:
            comp.add(src)
            comp.add(src[:5])
            comp.remove(src[20:])
            np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64),
                                          oracle.count(m[:20]) + oracle.count(m[:5]))
