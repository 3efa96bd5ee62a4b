"""Work of one context queued back to back, without a wait of the host in
between: clears, folds and renders launched while their predecessors drain
must still take effect one after another.  Every render of a long sequence has
outputs of its own; they are compared with the CPU oracle once the whole
sequence has run."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu

ROUNDS = 24
# small enough that kernels are over before the next is queued, and large enough that several are queued at once
SIZES = [(96, 64), (1999, 2001), (2048, 2000)]


def place(m: np.ndarray, shift: int):
    """Device copy whose first row starts `shift` elements into its allocation, rows one after another."""
    t = torch.from_numpy(m)
    buf = torch.zeros(m.size + shift, dtype=t.dtype, device="cuda")
    buf[shift:].copy_(t.reshape(-1))
    return buf[shift:].view(m.shape)


class Masks:
    """Byte or bit-packed masks: a render is the classes."""
    members = 12

    def __init__(self, w, h, count_bits, fmt="bytes", path="linear", shift=0):
        self.m = synth.random_masks(w + h, self.members, h, w)
        self.dev = place(synth.pack_masks(self.m) if fmt == "bits" else synth.scramble_nonzero(self.m, 7), shift)
        self.comp = binding.Composite(w, h, count_bits=count_bits, mask_format=fmt, read_path=path)
        self.shape = (h, w)

    def render(self):
        out = torch.full(self.shape, 99, dtype=torch.uint8, device="cuda")
        self.comp.render(bucket_out=out)
        return out

    def want(self, ids):
        c = oracle.count(self.m[ids])
        return oracle.bucket(c, len(ids))


class Depths:
    """Depths of small whole numbers, whose sums are exact in float32 in any order."""
    members = 12

    def __init__(self, w, h, path="linear", shift=0):
        self.d = np.random.default_rng(w).integers(0, 64, (self.members, h, w)).astype(np.float32)
        self.dev = place(self.d, shift)
        self.comp = binding.Composite(w, h, mode="mean_depth", read_path=path)
        self.shape = (h, w)

    def render(self):
        out = torch.full(self.shape, -1.0, dtype=torch.float32, device="cuda")
        self.comp.render(mean_out=out)
        return out

    def want(self, ids):
        return self.d[ids].sum(axis=0, dtype=np.float32) / np.float32(len(ids))


MAKERS = {
    "bytes16": lambda w, h: Masks(w, h, 16),
    "bytes32": lambda w, h: Masks(w, h, 32),
    "bytes16_odd": lambda w, h: Masks(w, h, 16, shift=3),
    "bytes32_odd": lambda w, h: Masks(w, h, 32, shift=3),
    "bits": lambda w, h: Masks(w, h, 16, fmt="bits"),
    "bits_odd": lambda w, h: Masks(w, h, 32, fmt="bits", shift=1),
    "tma": lambda w, h: Masks(w, h, 16, path="tma"),
    "texture": lambda w, h: Masks(w, h, 16, path="texture"),
    "depths": lambda w, h: Depths(w, h),
    "depths_odd": lambda w, h: Depths(w, h, shift=1),
    "depths_tma": lambda w, h: Depths(w, h, path="tma"),
}


@pytest.mark.parametrize("what", list(MAKERS))
@pytest.mark.parametrize("w,h", SIZES)
def test_renders_between_folds_and_clears(w, h, what):
    case = MAKERS[what](w, h)
    everyone, few, one = list(range(12)), list(range(8)), [3]
    got = {"few": [], "all": [], "one": []}
    with case.comp as comp:
        torch.cuda.synchronize()
        for _ in range(ROUNDS):
            comp.clear()
            comp.add(case.dev[:8])
            got["few"].append(case.render())
            comp.add(case.dev[8:])
            got["all"].append(case.render())
            comp.remove(case.dev[8:])
            got["few"].append(case.render())
            comp.clear()
            comp.add(case.dev[3:4])
            got["one"].append(case.render())
        comp.sync()
    for name, ids in (("few", few), ("all", everyone), ("one", one)):
        want = torch.from_numpy(case.want(ids)).cuda()
        for i, out in enumerate(got[name]):
            assert torch.equal(out, want), (name, i)


@pytest.mark.parametrize("what", ["bytes16", "bytes32_odd", "bits"])
@pytest.mark.parametrize("w,h", SIZES)
def test_histograms_around_folds_of_one_member(w, h, what):
    case = MAKERS[what](w, h)
    got = {11: [], 12: []}
    with case.comp as comp:
        torch.cuda.synchronize()
        for i in range(ROUNDS):
            comp.clear()
            comp.add(case.dev[:11])
            for j in range(3):
                for n in (11, 12):
                    hist = torch.full((256,), -1, dtype=torch.int64, device="cuda")
                    bucket = torch.empty(case.shape, dtype=torch.uint8, device="cuda")
                    comp.render_histogram(hist, bucket_out=bucket)
                    got[n].append((hist, bucket))
                    (comp.add if n == 11 else comp.remove)(case.dev[11:])
        comp.sync()
    for n, outs in got.items():
        classes = case.want(list(range(n)))
        want = torch.from_numpy(classes).cuda()
        counts = torch.from_numpy(np.bincount(classes.ravel(), minlength=256)).cuda()
        for hist, bucket in outs:
            assert torch.equal(bucket, want)
            assert torch.equal(hist, counts)
