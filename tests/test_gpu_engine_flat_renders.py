"""Engine renders of the classes alone from dense planes of 16-bit counts: items
of 512 pixels and what is left of them, outputs on and off 16-byte boundaries,
beside renders of other kinds, with few members and the most that fit."""
import pytest

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 4, 16])
@pytest.mark.parametrize("kinds", ["flat", "mixed", "histogram"])
def test_classes_alone(off, kinds):
    histogram = kinds == "histogram"
    shapes = [(16, 1), (16, 31), (16, 32), (16, 33), (512, 1), (512, 5), (528, 7), (1024, 600)] + ([] if kinds == "flat" else [(100, 20)])
    eng = binding.Engine()
    work = []
    for w, h in shapes:
        for bits in (16,) if kinds == "flat" else (16, 32):
            p = eng.add_plane(w, h, count_bits=bits)
            pitch = (w + 15) // 16 * 16
            m = torch.randint(0, 2, (5, h, pitch), dtype=torch.uint8, device="cuda")[:, :, :w]
            out = torch.full((w * h + 32,), 7, dtype=torch.uint8, device="cuda")
            hist = torch.full((256,), -1, dtype=torch.int64, device="cuda")
            work.append((p, m, out, hist, w, h))
    eng.submit([eng.op(p, m) for p, m, *_ in work])
    rops = [eng.render_op(p, bucket_out=out[off:off + w * h].view(h, w), histogram_out=hist if histogram else None)
            for p, _m, out, hist, w, h in work]
    eng.render(rops)
    eng.sync()
    for _p, m, out, hist, w, h in work:
        want = (m.sum(0, dtype=torch.int32) * 255 // 5).to(torch.uint8).reshape(-1)
        assert torch.equal(out[off:off + w * h], want)
        assert bool((out[:off] == 7).all()) and bool((out[off + w * h:] == 7).all())
        if histogram:
            assert torch.equal(hist, torch.bincount(want.int(), minlength=256))
    eng.close()


def test_the_most_members_of_16_bit_counts():
    w, h = 64, 32
    eng = binding.Engine()
    p = eng.add_plane(w, h, count_bits=16)
    m = torch.zeros((1, h, w), dtype=torch.uint8, device="cuda").expand(1, h, w).contiguous()
    m[:, ::2] = 1
    index = torch.zeros(65535, dtype=torch.int32, device="cuda")
    eng.submit([eng.op(p, m, index=index)])
    out = torch.empty((h, w), dtype=torch.uint8, device="cuda")
    eng.render([eng.render_op(p, bucket_out=out)])
    eng.sync()
    assert torch.equal(out, m[0] * 255)
    eng.close()
