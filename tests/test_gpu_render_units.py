"""The render's units of four pixels: rasters whose size is around a warp
item (512 pixels) and a CTA's, dense rows, rows of fours and ragged rows, and
outputs that are not aligned to four elements, on the plain and the engine
render, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (3, 1), (4, 1), (16, 32), (20, 7), (511, 1), (73, 7), (512, 8), (1, 4097), (4100, 1), (1000, 13), (1501, 3)]


def outputs(w, h, count_bits, off):
    """counts, classes, colours and histogram on the device, the first three `off` elements past an aligned address."""
    px = w * h
    counts = torch.full((px + off + 1,), -1, dtype=torch.int16 if count_bits == 16 else torch.int32, device="cuda")
    bucket = torch.full((px + off + 1,), 7, dtype=torch.uint8, device="cuda")
    rgba = torch.full((4 * (px + off + 1),), 7, dtype=torch.uint8, device="cuda")
    return (counts[off:off + px].view(h, w), bucket[off:off + px].view(h, w), rgba[4 * off:4 * (off + px)].view(h, w, 4),
            torch.empty(256, dtype=torch.int64, device="cuda")), (counts, bucket, rgba)


def check(outs, whole, c, n, off):
    b = oracle.bucket(c, n)
    got = outs[0].cpu().numpy()
    np.testing.assert_array_equal((got.view(np.uint16) if got.dtype == np.int16 else got).astype(np.int64), c)
    np.testing.assert_array_equal(outs[1].cpu().numpy(), b)
    np.testing.assert_array_equal(outs[2].cpu().numpy(), oracle.rgba(b))
    np.testing.assert_array_equal(outs[3].cpu().numpy(), oracle.histogram(b).astype(np.int64))
    # nothing written before or after
    assert int(whole[0][-1]) == -1 and int(whole[1][-1]) == 7 and int(whole[2][-1]) == 7
    if off:
        assert int(whole[0][0]) == -1 and int(whole[1][0]) == 7 and int(whole[2][3]) == 7


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("count_bits", [16, 32])
def test_plain_and_engine_render(count_bits, off):
    with binding.Engine() as eng:
        rops, checks = [], []
        for i, (w, h) in enumerate(SHAPES):
            n = 1 + 40 * i
            m = synth.random_masks(7 + i, n, h, w, density=0.4)
            c = oracle.count(m)
            dev = torch.zeros((n, h, (w + 15) // 16 * 16), dtype=torch.uint8, device="cuda")
            dev[:, :, :w] = torch.from_numpy(m).cuda()
            with binding.Composite(w, h, count_bits=count_bits) as comp:
                comp.add(dev[:, :, :w])
                outs, whole = outputs(w, h, count_bits, off)
                comp.render_histogram(outs[3], *outs[:3])
                comp.sync()
                check(outs, whole, c, n, off)
                outs, whole = outputs(w, h, count_bits, off)
                comp.render(*outs[:3])
                comp.render_histogram(outs[3])   # by itself
                comp.sync()
                check(outs, whole, c, n, off)
            plane = eng.add_plane(w, h, count_bits)
            eng.submit([eng.op(plane, dev[:, :, :w])])
            outs, whole = outputs(w, h, count_bits, off)
            rops.append(eng.render_op(plane, *outs[:3], histogram_out=outs[3]))
            checks.append((outs, whole, c, n, off))
            eng.sync()
        eng.render(rops)
        eng.sync()
        for args in checks:
            check(*args)


@pytest.mark.parametrize("off", [0, 1])
def test_means(off):
    for i, (w, h) in enumerate(SHAPES):
        d = synth.random_depths(i, 3, h, w)
        with binding.Composite(w, h, mode="mean_depth") as comp:
            comp.add(torch.from_numpy(d).cuda())
            whole = torch.full((w * h + off + 1,), -1.0, device="cuda")
            mean = whole[off:off + w * h].view(h, w)
            comp.render(mean_out=mean)
            comp.sync()
            # three float32 additions of depths below 4 and a division, each rounded once
            assert np.abs(mean.cpu().numpy().astype(np.float64) - oracle.mean_depth(d)).max() <= 4 * 4.0 * 2.0 ** -24
            assert float(whole[-1]) == -1.0 and (not off or float(whole[0]) == -1.0)
