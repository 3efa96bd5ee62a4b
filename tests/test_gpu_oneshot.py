"""The one-shot composite's single kernel: rasters around its 16-pixel groups
and CTAs, members around its slices (16, 32, 64, 128) and its slabs of 255,
memory that ends with the last pixel, outputs that allow no four-pixel stores,
and calls on several streams at once, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (15, 3), (16, 16), (17, 9), (100, 37), (128, 70), (1023, 5), (2048, 64)]
MEMBERS = [1, 2, 9, 16, 33, 64, 130, 255, 256, 600]


def tight(m: np.ndarray):
    n, h, w = m.shape
    pitch = (w + 15) // 16 * 16
    buf = torch.full((n * h * pitch - (pitch - w),), 255, dtype=torch.uint8, device="cuda")
    view = buf.as_strided((n, h, w), (h * pitch, pitch, 1))
    view.copy_(torch.from_numpy(m))
    return view


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("w,h", SHAPES)
def test_shapes_and_members(w, h, off):
    for n in MEMBERS:
        m = synth.scramble_nonzero(synth.random_masks(n, n, h, w), 4)
        dev, px = tight(m), w * h
        counts = torch.full((px + 2,), -1, dtype=torch.int32, device="cuda")
        bucket = torch.full((px + 2,), 7, dtype=torch.uint8, device="cuda")
        rgba = torch.full((4 * (px + 2),), 7, dtype=torch.uint8, device="cuda")
        binding.composite_oneshot_static(dev, counts[off:off + px].view(h, w), bucket[off:off + px].view(h, w),
                                         rgba[4 * off:4 * (off + px)].view(h, w, 4))
        torch.cuda.synchronize()
        c = oracle.count(m)
        b = oracle.bucket(c, n)
        np.testing.assert_array_equal(counts[off:off + px].cpu().numpy().reshape(h, w), c)
        np.testing.assert_array_equal(bucket[off:off + px].cpu().numpy().reshape(h, w), b)
        np.testing.assert_array_equal(rgba[4 * off:4 * (off + px)].cpu().numpy().reshape(h, w, 4), oracle.rgba(b))
        assert int(counts[-1]) == -1 and int(bucket[-1]) == 7 and int(rgba[-1]) == 7


def test_calls_on_several_streams_at_once():
    work = []
    for i in range(6):
        m = synth.random_masks(i, 40 + i, 300, 500)
        work.append((m, tight(m), torch.empty((300, 500), dtype=torch.int32, device="cuda"), torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(5):
        for _m, dev, counts, stream in work:
            binding.composite_oneshot_static(dev, counts, stream=stream.cuda_stream)
    torch.cuda.synchronize()
    for m, _dev, counts, _s in work:
        np.testing.assert_array_equal(counts.cpu().numpy(), oracle.count(m))
