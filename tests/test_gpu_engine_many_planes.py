"""Engines of many planes: the host's share of a submit follows the planes that
its ops name, not the planes that the engine holds; chains still fold in order."""
import time

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu

PLANES = 30000


def submit_us(eng, ops) -> float:
    best = 1e9
    for _ in range(10):
        start = time.perf_counter()
        for _ in range(30):   # fewer than the uploads that may be in flight
            eng.submit(ops)
        best = min(best, (time.perf_counter() - start) / 30)
        torch.cuda.synchronize()
    return 1e6 * best


def test_a_small_submit_among_many_planes():
    m = synth.random_masks(1, 3, 16, 16)
    dev = torch.from_numpy(m).cuda()
    eng = binding.Engine()
    first = eng.add_plane(16, 16)
    ops = [eng.op(first, dev[:1])]
    few = submit_us(eng, ops)
    last = [eng.add_plane(16, 16) for _ in range(PLANES - 1)][-1]
    many = submit_us(eng, ops)
    # the member counts of the engine's planes are looked through once per
    # submit (8 bytes each: 20 us); tables of 48 bytes a plane more took 90
    assert many - few < 45.0, (few, many)
    # ops on planes far apart, and a chain on one of them
    eng.clear_many([first, last])
    eng.submit([eng.op(last, dev), eng.op(first, dev[:2]), eng.op(last, dev[:1], sign=-1)])
    counts = {p: torch.empty((16, 16), dtype=torch.int32, device="cuda") for p in (first, last)}
    eng.render([eng.render_op(p, counts_out=c) for p, c in counts.items()])
    eng.sync()
    np.testing.assert_array_equal(counts[first].cpu().numpy(), oracle.count(m[:2]))
    np.testing.assert_array_equal(counts[last].cpu().numpy(), oracle.count(m[1:]))
    eng.close()
