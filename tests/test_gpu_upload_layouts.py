"""Host rasters of every layout through the staging slots: rows that follow one
another (uploaded as one run of bytes), small and large row padding, gaps
between members, odd base addresses; pinned memory and pageable batches
registered for the call, on every read path, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


def host(m: np.ndarray, shift: int, pitch: int, gap: int, pinned: bool):
    n, h, w = m.shape
    stride = pitch * h + gap
    size = shift + (n - 1) * stride + (h - 1) * pitch + w
    buf = torch.ones(size, dtype=torch.uint8 if m.dtype == np.uint8 else torch.float32)
    buf = buf.pin_memory() if pinned else buf
    view = buf.as_strided((n, h, w), (stride, pitch, 1), storage_offset=shift)
    view.copy_(torch.from_numpy(m))
    return view


LAYOUTS = [(64, 9, 0, 0, 0), (61, 16, 0, 0, 0), (61, 9, 3, 0, 0), (50, 7, 1, 2, 0), (506, 40, 0, 0, 5), (100, 13, 2, 412, 0),
           (1501, 3, 0, 11, 0), (33, 5, 7, 90, 64), (1, 1, 0, 0, 0)]


@pytest.mark.parametrize("memory", ["pinned", "registered"])
@pytest.mark.parametrize("path,fmt", [("linear", "bytes"), ("linear", "bits"), ("texture", "bytes"), ("tma", "bytes")])
@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS)
def test_masks(w, h, shift, pad, gap, path, fmt, memory):
    ingest = "register" if memory == "registered" else "auto"
    for chunk in (0, 7):
        with binding.Composite(w, h, read_path=path, mask_format=fmt, chunk_members=chunk, pageable_ingest=ingest) as comp:
            for n in (1, 20, 41):
                m = synth.random_masks(n, n, h, w)
                data = synth.pack_masks(m) if fmt == "bits" else synth.scramble_nonzero(m, 6)
                src = host(data, shift, data.shape[2] + pad, gap, memory == "pinned")
                comp.clear()
                comp.add(src if memory == "pinned" else src.numpy())
                comp.remove(src[: n // 2])
                np.testing.assert_array_equal(comp.render_host()["counts"].astype(np.int64), oracle.count(m[n // 2:]))


@pytest.mark.parametrize("path", ["linear", "texture", "tma"])
@pytest.mark.parametrize("w,h,shift,pad,gap", LAYOUTS)
def test_depths(w, h, shift, pad, gap, path):
    with binding.Composite(w, h, read_path=path, mode="mean_depth", chunk_members=6) as comp:
        n = 20
        d = synth.random_depths(8, n, h, w)
        comp.add(host(d, shift, w + pad, gap, True))
        # sums of 20 depths below 4, no more roundings than additions, and the division
        err = np.abs(comp.render_host()["mean"].astype(np.float64) - oracle.mean_depth(d)).max()
        assert err <= 4.0 * (n + 1) * 2.0 ** -24
