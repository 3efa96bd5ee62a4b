"""The classes or the 16-bit counts alone of rasters on both sides of the size
from which a lane renders eight units at a time: rows that are dense in the
plane, of whole units, and ragged, and outputs that allow no vector stores."""
import pytest

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("w,h", [(4096, 4095), (4096, 4096), (4100, 4100), (4099, 4101), (16, 1048577)])
def test_classes_and_counts_alone(w, h, off):
    m = torch.randint(0, 2, (3, h, w), dtype=torch.uint8, device="cuda")
    with binding.Composite(w, h, count_bits=16) as comp:
        comp.add(m)
        bucket = torch.full((w * h + 2,), 7, dtype=torch.uint8, device="cuda")
        counts = torch.full((w * h + 2,), -1, dtype=torch.int16, device="cuda")
        comp.render(bucket_out=bucket[off:off + w * h])
        comp.render(counts_out=counts[off:off + w * h])
        comp.sync()
        want = m.sum(0, dtype=torch.int16).reshape(-1)
        assert torch.equal(counts[off:off + w * h], want)
        assert torch.equal(bucket[off:off + w * h], (want.int() * 85).to(torch.uint8))   # floor(255 c / 3)
        assert int(counts[-1]) == -1 and int(bucket[-1]) == 7
