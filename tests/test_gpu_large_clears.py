"""Clears of planes of a size from which memsets take over from the kernel, and
just below it: counts, sums and the underflow state start again from zero."""
import pytest

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,count_bits,w,h", [("count", 32, 6144, 6143), ("count", 32, 6144, 6144), ("count", 16, 9001, 8417),
                                                 ("mean_depth", 16, 6144, 6144)])
def test_a_cleared_plane_starts_again(mode, count_bits, w, h):
    one = torch.ones((1, h, w), dtype=torch.uint8 if mode == "count" else torch.float32, device="cuda")
    with binding.Composite(w, h, mode=mode, count_bits=count_bits) as comp:
        for _ in range(2):
            comp.add(one)
            comp.add(one)
            comp.clear()
            comp.add(one)
            if mode == "count":
                out = torch.full((h, w), -1, dtype=torch.int16 if count_bits == 16 else torch.int32, device="cuda")
                comp.render(counts_out=out)
            else:
                out = torch.full((h, w), -1.0, dtype=torch.float32, device="cuda")
                comp.render(mean_out=out)
            comp.sync()
            assert bool((out == 1).all())
        if mode == "count":
            comp.clear()
            comp.add(one * 0)
            comp.remove(one)
            with pytest.raises(binding.CompositeError) as e:
                comp.sync()
            assert e.value.code == binding.CPT_EUNDERFLOW
            comp.clear()
            comp.sync()
