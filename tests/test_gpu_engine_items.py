"""How the engine cuts a submit into work items: ops chained on one plane,
slabs split for launches short of items, ragged right edges read by whole
groups (and exactly, at the end of the caller's memory), every mask format and
count width, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (16, 1), (17, 2), (24, 3), (31, 5), (33, 3), (47, 1), (1023, 7), (130, 64)]
MEMBERS = [(1, 0), (7, 1), (8, 8), (9, 3), (33, 17), (130, 100), (256, 40), (300, 0)]


def tight(m: np.ndarray):
    """Device copy whose rows are padded to 16 bytes (with bytes of ones) except the very last, which ends the memory."""
    n, h, w = m.shape
    pitch = (w + 15) // 16 * 16
    buf = torch.full((n * h * pitch - (pitch - w),), 255, dtype=torch.uint8, device="cuda")
    view = buf.as_strided((n, h, w), (h * pitch, pitch, 1))
    view.copy_(torch.from_numpy(m))
    return view


@pytest.mark.parametrize("count_bits", [16, 32])
@pytest.mark.parametrize("fmt", ["bytes", "bits"])
@pytest.mark.parametrize("adds,removes", MEMBERS)
def test_adds_and_removes_of_many_planes(adds, removes, fmt, count_bits):
    with binding.Engine() as eng:
        checks = []
        ops, rops = [], []
        for i, (w, h) in enumerate(SHAPES):
            m = synth.random_masks(90 + i, adds, h, w, density=0.5)
            dev = tight(synth.pack_masks(m) if fmt == "bits" else m)
            order = np.random.RandomState(i).permutation(adds).astype(np.int32)
            gone = order[:removes]
            plane = eng.add_plane(w, h, count_bits)
            counts = torch.empty((h, w), dtype=torch.int32 if count_bits == 32 else torch.int16, device="cuda")
            # in: the first half in place, the second by index; out: some of both, in two ops
            half = adds // 2
            if half:
                ops.append(eng.op(plane, dev[:half], mask_format=fmt))
            ops.append(eng.op(plane, dev, index=torch.arange(half, adds, dtype=torch.int32, device="cuda"), mask_format=fmt))
            for part in (gone[: removes // 2], gone[removes // 2:]):
                if len(part):
                    ops.append(eng.op(plane, dev, sign=-1, index=torch.from_numpy(part.copy()).cuda(), mask_format=fmt))
            rops.append(eng.render_op(plane, counts))
            checks.append((counts, np.delete(m, gone, axis=0)))
        # the planes' ops interleaved, as requests of several users would be
        by_turn = sorted(range(len(ops)), key=lambda k: (sum(ops[j].plane == ops[k].plane for j in range(k)), k))
        eng.submit([ops[k] for k in by_turn])
        eng.render(rops)
        eng.sync()
        for counts, left in checks:
            got = counts.cpu().numpy().astype(np.int64)
            want = oracle.count(left) if len(left) else np.zeros(got.shape, np.int64)
            np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("schedule", ["persistent", "grid"])
@pytest.mark.parametrize("fmt", ["bytes", "bits"])
def test_few_long_ops_are_split_and_replayed(fmt, schedule):
    # too few groups for every CTA: slabs of down to 32 members by atomics; slices of 4 at 32 members and more
    sizes = [(40, 9, 31), (96, 33, 32), (513, 5, 255), (300, 70, 700)]
    with binding.Engine(schedule=schedule) as eng:
        ops, rops, checks = [], [], []
        for i, (w, h, n) in enumerate(sizes):
            m = synth.random_masks(70 + i, n, h, w)
            plane = eng.add_plane(w, h)
            counts = torch.empty((h, w), dtype=torch.int32, device="cuda")
            ops.append(eng.op(plane, tight(synth.pack_masks(m) if fmt == "bits" else m), mask_format=fmt))
            rops.append(eng.render_op(plane, counts))
            checks.append((counts, oracle.count(m)))
        keep = list(eng._keep)
        eng.capture(ops, rops, keep=keep)
        for _ in range(3):   # the item counter starts every replay from zero
            for counts, _c in checks:
                counts.fill_(-1)
            eng.replay()
            eng.sync()
            for counts, c in checks:
                np.testing.assert_array_equal(counts.cpu().numpy(), c)


def test_mixed_formats_and_underflow_on_one_plane():
    w, h = 200, 50
    a, b = synth.random_masks(1, 40, h, w), synth.random_masks(2, 12, h, w)
    full = np.ones((1, h, w), np.uint8)
    with binding.Engine() as eng:
        p, q = eng.add_plane(w, h), eng.add_plane(w, h)
        out = [torch.empty((h, w), dtype=torch.int32, device="cuda") for _ in range(2)]
        bits = tight(synth.pack_masks(b))
        eng.submit([eng.op(p, tight(a)), eng.op(p, bits, mask_format="bits"), eng.op(q, tight(full)),
                    eng.op(q, tight(full), sign=-1)])
        eng.render([eng.render_op(p, out[0]), eng.render_op(q, out[1])])
        eng.sync()   # a member added and taken away in one submit is no underflow
        np.testing.assert_array_equal(out[0].cpu().numpy(), oracle.count(a) + oracle.count(b))
        assert int(out[1].abs().sum()) == 0
        # a member that was never added, taken away between two adds: found on its plane
        dry = np.zeros((2, h, w), np.uint8)
        eng.submit([eng.op(q, tight(dry)), eng.op(q, tight(full), sign=-1), eng.op(q, tight(dry))])
        with pytest.raises(binding.CompositeError) as e:
            eng.sync()
        assert e.value.code == binding.CPT_EUNDERFLOW and e.value.plane == q
