"""Bit-packed engine ops of several slabs, which run as five CTAs per SM where
they are most of a submit's work: slabs and steps of members at their edges, adds
and removes, and submits on both sides of half of the work, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


def device_rows(m: np.ndarray):
    """Bit-packed rows 16 bytes apart."""
    packed = synth.pack_masks(m)
    n, h, row = packed.shape
    buf = torch.zeros((n, h, (row + 15) // 16 * 16), dtype=torch.uint8, device="cuda")
    view = buf[:, :, :row]
    view.copy_(torch.from_numpy(packed))
    return view


@pytest.mark.parametrize("ctas", [4, 5])
@pytest.mark.parametrize("schedule", ["persistent", "grid"])
@pytest.mark.parametrize("count_bits", [16, 32])
def test_deep_and_shallow_ops(count_bits, schedule, ctas):
    w, h = 777, 95
    eng = binding.Engine(schedule=schedule, slab_members=32, ctas_per_sm=ctas)
    planes = [eng.add_plane(w, h, count_bits=count_bits) for _ in range(3)]
    for deep, shallow in ((33, 0), (300, 1), (65, 32), (33, 32), (64, 32)):
        m = synth.random_masks(deep, max(deep, 40), h, w)
        dev = device_rows(m)
        idx = torch.randperm(deep, device="cuda", dtype=torch.int32)
        ops = [eng.op(planes[0], dev[:deep], mask_format="bits"), eng.op(planes[1], dev, index=idx, mask_format="bits")]
        if shallow:
            ops += [eng.op(planes[2], dev[:shallow], mask_format="bits")] * 2
        eng.clear_many(planes)
        eng.submit(ops)
        eng.submit([eng.op(planes[0], dev[:deep - 20], sign=-1, mask_format="bits")])
        outs = [torch.empty((h, w), dtype=torch.int16 if count_bits == 16 else torch.int32, device="cuda") for _ in planes]
        eng.render([eng.render_op(p, counts_out=o) for p, o in zip(planes, outs)])
        eng.sync()
        for o, want in zip(outs, (oracle.count(m[deep - 20:deep]), oracle.count(m[:deep]), 2 * oracle.count(m[:shallow]))):
            np.testing.assert_array_equal(o.cpu().numpy().astype(np.int64), want)
    eng.close()
