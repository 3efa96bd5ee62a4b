"""The work that users of the compositor have it do, as timed cases: each goes
through the public Python entry points (binding.Composite, Engine, Server and
the allocation-free one-shot) the way a program calls them.

A case names a `kind` and plain sizes:

* compose  clear, add every member, render.  `memory` says where the rasters
           are (device, or pinned host memory streamed through the staging
           buffers), `data` what they are (bytes: uint8 masks, bits: bit-packed
           masks, depths: float32), `path` the read path, `out` where the
           render goes (device tensors or host arrays).
* toggle   the interactive list: a resident ensemble, members taken out and
           others put in, the composite rendered with its class histogram.
* oneshot  the call for render callbacks that may not allocate.
* batch    many composites of uneven size in one engine submit and one render,
           or the same work replayed from a captured graph.
* serve    sessions that toggle member subsets of a resident ensemble with a
           pinned overflow part; one request per session, drained.

Rasters come from a synthetic terrain: a member floods the pixels below its
water level, levels chosen so that 10 to 50 % of the pixels are flooded.
"""
import math
import random

import numpy as np
import torch

from paper_2104_14667_gb300 import binding

DEVICE = "cuda"
MAX_SIDE = 4608
MAX_MEMBERS = 1024
DRAW_DEVICE_BYTES = 2 << 30     # rasters of a drawn case, in device memory
DRAW_PINNED_BYTES = 256 << 20   # and in pinned host memory


def listed():
    return [
        # a viewer's per-frame callback over a small region of interest: the smallest call
        {"name": "oneshot_512x512x8", "kind": "oneshot", "width": 512, "height": 512, "members": 8},
        # the plain method, tiny: 16 masks of 1024^2 streamed through two staging buffers
        {"name": "stream_1024x1024x16", "kind": "compose", "width": 1024, "height": 1024, "members": 16,
         "data": "bytes", "memory": "pinned", "path": "linear", "count_bits": 16, "out": "device"},
        # a user of the interactive list swaps four members of a ~2k raster ensemble
        {"name": "toggle_1856x2208x64_4", "kind": "toggle", "width": 1856, "height": 2208, "members": 64, "swap": 4,
         "data": "bytes", "count_bits": 16},
        # a cropped area whose width is no multiple of anything, as tensors come from a slice or a file: 32-bit counts
        {"name": "masks_1501x1103x100", "kind": "compose", "width": 1501, "height": 1103, "members": 100,
         "data": "bytes", "memory": "device", "path": "linear", "count_bits": 32, "out": "device"},
        # mean flood depth over a ~2k raster ensemble
        {"name": "depths_1856x2208x64", "kind": "compose", "width": 1856, "height": 2208, "members": 64,
         "data": "depths", "memory": "device", "path": "linear", "count_bits": 16, "out": "device"},
        # the read-path sweep's tensor-memory-accelerator row, masks
        {"name": "masks_tma_4096x4096x128", "kind": "compose", "width": 4096, "height": 4096, "members": 128,
         "data": "bytes", "memory": "device", "path": "tma", "count_bits": 16, "out": "device"},
        # the read-path sweep's image row, masks
        {"name": "masks_texture_2048x2048x256", "kind": "compose", "width": 2048, "height": 2048, "members": 256,
         "data": "bytes", "memory": "device", "path": "texture", "count_bits": 16, "out": "device"},
        # a compressed ~2k ensemble kept resident: rows of 232 bytes, as packing gives them
        {"name": "bits_1856x2208x1024", "kind": "compose", "width": 1856, "height": 2208, "members": 1024,
         "data": "bits", "memory": "device", "path": "linear", "count_bits": 16, "out": "device"},
        # the batched form: 64 requests of uneven member counts and raster sizes in one captured launch
        {"name": "batch_64", "kind": "batch", "requests": 64, "mix": 4, "side_max": 2048, "members_max": 512,
         "graph": True, "histogram": False, "count_bits": 16},
        # the served form: eight users toggle 8 to 512 members each of a resident ensemble with some overflow
        {"name": "serve_1024x1024_8", "kind": "serve", "width": 1024, "height": 1024, "resident": 1024,
         "overflow": 128, "sessions": 8, "toggle_max": 512, "mix": 5, "data": "bytes"},
        # a ~4k ensemble streamed from pinned memory, the result read back: the paper's own workload
        {"name": "stream_3712x4416x64", "kind": "compose", "width": 3712, "height": 4416, "members": 64,
         "data": "bytes", "memory": "pinned", "path": "linear", "count_bits": 16, "out": "host"},
        # a resident ensemble recomposed in full: the largest
        {"name": "masks_4096x4096x1024", "kind": "compose", "width": 4096, "height": 4096, "members": 1024,
         "data": "bytes", "memory": "device", "path": "linear", "count_bits": 16, "out": "device"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.5)))))))


def _row_bytes(data, width):
    return {"bytes": width, "bits": (width + 7) // 8, "depths": 4 * width}[data]


def _draw_size(rng, data, budget, side_max=MAX_SIDE, side_min=64):
    """Sides and members over their ranges; half the widths are multiples of 64, the others anything."""
    width = _log_int(rng, side_min, side_max)
    height = _log_int(rng, side_min, side_max)
    if rng.random() < 0.5:
        width = max(64, width // 64 * 64)
    most = max(1, min(MAX_MEMBERS, budget // (_row_bytes(data, width) * height)))
    return width, height, _log_int(rng, 1, most)


def draw(rng):
    kind = rng.choices(["compose", "toggle", "oneshot", "batch", "serve"], [6, 2, 1, 1, 1])[0]
    if kind == "compose":
        data = rng.choices(["bytes", "bits", "depths"], [3, 1, 1])[0]
        memory = rng.choices(["device", "pinned"], [3, 1])[0]
        path = "linear" if data == "bits" else rng.choices(["linear", "tma", "texture"], [2, 1, 1])[0]
        w, h, n = _draw_size(rng, data, DRAW_DEVICE_BYTES if memory == "device" else DRAW_PINNED_BYTES)
        return {"kind": kind, "width": w, "height": h, "members": n, "data": data, "memory": memory, "path": path,
                "count_bits": rng.choice([16, 32]), "out": rng.choices(["device", "host"], [3, 1])[0]}
    if kind == "toggle":
        data = rng.choice(["bytes", "bits"])
        w, h, n = _draw_size(rng, data, DRAW_DEVICE_BYTES)
        n = max(2, n)
        return {"kind": kind, "width": w, "height": h, "members": n, "swap": _log_int(rng, 1, n // 2),
                "data": data, "count_bits": rng.choice([16, 32])}
    if kind == "oneshot":
        w, h, n = _draw_size(rng, "bytes", DRAW_DEVICE_BYTES, side_max=2048)
        return {"kind": kind, "width": w, "height": h, "members": n}
    if kind == "batch":
        return {"kind": kind, "requests": _log_int(rng, 2, 64), "mix": rng.randrange(1 << 20), "side_max": 1024,
                "members_max": 256, "graph": rng.random() < 0.5, "histogram": rng.random() < 0.5,
                "count_bits": rng.choice([16, 32])}
    return {"kind": kind, "width": 16 * _log_int(rng, 8, 64), "height": _log_int(rng, 128, 1024),
            "resident": _log_int(rng, 64, 1024), "overflow": _log_int(rng, 16, 128), "sessions": rng.randint(1, 16),
            "toggle_max": _log_int(rng, 16, 64), "mix": rng.randrange(1 << 20), "data": rng.choice(["bytes", "bits"])}


# --- inputs ------------------------------------------------------------------

def _terrain(gen, width, height):
    """float32[height, width]: 12 Gaussian bumps and a little noise."""
    u = torch.rand((12, 4), generator=gen, device=DEVICE)
    xs = torch.arange(width, device=DEVICE, dtype=torch.float32)
    ys = torch.arange(height, device=DEVICE, dtype=torch.float32)
    sigma = 20.0 + 180.0 * u[:, 2:3]
    gx = torch.exp(-((xs[None] - u[:, 0:1] * width) ** 2) / (2.0 * sigma * sigma)) * u[:, 3:4]
    gy = torch.exp(-((ys[None] - u[:, 1:2] * height) ** 2) / (2.0 * sigma * sigma))
    t = torch.zeros((height, width), device=DEVICE)
    for k in range(12):
        t += gy[k][:, None] * gx[k][None]
    return t + 0.01 * torch.randn((height, width), generator=gen, device=DEVICE)


def _levels(gen, terrain, members):
    """One water level per member, flooding 10 to 50 % of the pixels."""
    flat = terrain.reshape(-1)
    sample = flat[torch.randint(flat.numel(), (min(flat.numel(), 1 << 16),), generator=gen, device=DEVICE)].sort()[0]
    f = 0.1 + 0.4 * torch.rand((members,), generator=gen, device=DEVICE)
    return sample[(f * (sample.numel() - 1)).long()]


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _fill(terrain, levels, data, out):
    """Rasters of every level into out[n, height, row], on the device or in host memory, a few at a time."""
    height, width = terrain.shape
    step = max(1, min(len(levels), (256 << 20) // (4 * height * width)))
    weights = (1 << torch.arange(8, device=DEVICE)).to(torch.uint8)
    for m0 in range(0, len(levels), step):
        lv = levels[m0:m0 + step, None, None]
        if data == "depths":
            r = (lv - terrain).clamp_(min=0.0)
        else:
            r = terrain < lv
            if data == "bits":
                r = torch.nn.functional.pad(r, (0, -width % 8)).reshape(len(lv), height, -1, 8)
                r = (r.to(torch.uint8) * weights).sum(-1, dtype=torch.uint8)
            else:
                r = r.view(torch.uint8)
        out[m0:m0 + step].copy_(r)


def _rasters(gen, width, height, members, data, memory, pad_rows_to=1):
    """Contiguous rasters [n, height, row]; pad_rows_to: the rows' storage is a multiple of that many bytes."""
    row = _row_bytes(data, width) if data == "bits" else width
    pitch = -(-row // pad_rows_to) * pad_rows_to
    dtype = torch.float32 if data == "depths" else torch.uint8
    shape = (members, height, pitch)
    out = torch.empty(shape, dtype=dtype, pin_memory=True) if memory == "pinned" else torch.empty(shape, dtype=dtype, device=DEVICE)
    terrain = _terrain(gen, width, height)
    view = out[:, :, :row]
    _fill(terrain, _levels(gen, terrain, members), data, view)
    torch.cuda.synchronize()
    return view


def _images(width, height, count_bits=None, histogram=False, host=False):
    """Output tensors of a render: counts of the given width (None: none), classes, colours, histogram."""
    where = {"pin_memory": True} if host else {"device": DEVICE}
    out = {}
    if count_bits:
        out["counts"] = torch.empty((height, width), dtype=torch.int16 if count_bits == 16 else torch.int32, **where)
    out["bucket"] = torch.empty((height, width), dtype=torch.uint8, **where)
    out["rgba"] = torch.empty((height, width, 4), dtype=torch.uint8, **where)
    if histogram:
        out["histogram"] = torch.empty(256, dtype=torch.int64, **where)
    return out


def _image_set(sizes, counts=False, histogram=False):
    """Outputs of many renders, each kind in one flat buffer: (the buffers, [the views of every render])."""
    kinds = [("counts", torch.int32, 1)] if counts else []
    kinds += [("bucket", torch.uint8, 1), ("rgba", torch.uint8, 4)]
    room = [-(-w * h // 256) * 256 for w, h in sizes]   # every view starts on a 256-byte boundary
    flat = {key: torch.zeros(sum(room) * per, dtype=dtype, device=DEVICE) for key, dtype, per in kinds}
    if histogram:
        flat["histogram"] = torch.zeros((len(sizes), 256), dtype=torch.int64, device=DEVICE)
    views, at = [], 0
    for i, (w, h) in enumerate(sizes):
        v = {key: flat[key][at * per:(at + w * h) * per].view((h, w, 4) if per == 4 else (h, w)) for key, _, per in kinds}
        if histogram:
            v["histogram"] = flat["histogram"][i]
        views.append(v)
        at += room[i]
    return flat, views


def _batch_requests(case):
    """(width, height, members) of every request: sides log-uniform from 64, half of them multiples of 64."""
    rng = random.Random(case["mix"])
    return [(_log_int(rng, 1, case["side_max"] // 64) * 64 if rng.random() < 0.5 else _log_int(rng, 64, case["side_max"]),
             _log_int(rng, 64, case["side_max"]), _log_int(rng, 8, case["members_max"])) for _ in range(case["requests"])]


def _toggles(case):
    """The member ids that each session toggles on every request, and those it holds at the start (half of all)."""
    rng = random.Random(case["mix"])
    total = case["resident"] + case["overflow"]
    toggles = [sorted(rng.sample(range(total), min(total, _log_int(rng, 8, case["toggle_max"])))) for _ in range(case["sessions"])]
    held = [sorted(rng.sample(range(total), total // 2)) for _ in range(case["sessions"])]
    return toggles, held


def _composite(case):
    mode = "mean_depth" if case["data"] == "depths" else "count"
    return binding.Composite(case["width"], case["height"], read_path=case.get("path", "linear"), mode=mode,
                             mask_format="bits" if case["data"] == "bits" else "bytes", count_bits=case["count_bits"])


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, gen)
    if kind == "serve":
        return _prepare_serve(case, gen)
    w, h, n = case["width"], case["height"], case["members"]
    if kind == "oneshot":
        # rows padded to the 16 bytes that the call asks for
        members = _rasters(gen, w, h, n, "bytes", "device", pad_rows_to=16)
        return {"kind": kind, "members": members, "out": _images(w, h, 32)}
    if kind == "toggle":
        members = _rasters(gen, w, h, n, case["data"], "device")
        comp = _composite(case)
        comp.add(members[case["swap"]:])   # all but the first few, which the first pass puts in
        comp.sync()
        return {"kind": kind, "comp": comp, "members": members, "swap": case["swap"], "outside": 0,
                "out": _images(w, h, case["count_bits"], histogram=True)}
    members = _rasters(gen, w, h, n, case["data"], case["memory"])
    host = case["out"] == "host"
    if case["data"] == "depths":
        out = {"mean": torch.empty((h, w), dtype=torch.float32, **({"pin_memory": True} if host else {"device": DEVICE}))}
    else:
        out = _images(w, h, case["count_bits"], host=host)
    return {"kind": kind, "comp": _composite(case), "members": members, "out": out}


def _prepare_batch(case, gen):
    eng = binding.Engine()
    requests = _batch_requests(case)
    flat, views = _image_set([(w, h) for w, h, _ in requests], histogram=case["histogram"])
    state = {"kind": "batch", "engine": eng, "graph": case["graph"], "planes": [], "ops": [], "rops": [], "keep": [], "out": flat}
    for i, (w, h, n) in enumerate(requests):
        # engine rows are multiples of 16 bytes
        members = _rasters(gen, w, h, n, "bytes", "device", pad_rows_to=16)
        plane = eng.add_plane(w, h, case["count_bits"])
        index = None
        if i % 4 == 3:   # every fourth request picks half of its ensemble by index
            index = torch.randperm(n, generator=gen, device=DEVICE)[: max(1, n // 2)].to(torch.int32)
        out = views[i]
        state["planes"].append(plane)
        state["ops"].append(eng.op(plane, members, index=index))
        state["rops"].append(eng.render_op(plane, None, out["bucket"], out["rgba"], out.get("histogram")))
        state["keep"].append((members, index))
    if case["graph"]:
        eng.capture(state["ops"], state["rops"])
    eng.sync()
    return state


def _prepare_serve(case, gen):
    w, h = case["width"], case["height"]
    both = _rasters(gen, w, h, case["resident"] + case["overflow"], case["data"], "device", pad_rows_to=16)
    row, n_res = both.shape[2], case["resident"]
    pitch = both.stride(1)
    base = both.as_strided((both.shape[0], h, pitch), both.stride())
    resident = base[:n_res].clone()
    overflow = torch.empty((case["overflow"], h, pitch), dtype=torch.uint8, pin_memory=True)
    overflow.copy_(base[n_res:])
    del both, base
    bits = case["data"] == "bits"
    server = binding.Server(resident[:, :, :row], overflow[:, :, :row], mask_format=case["data"], width=w if bits else None)
    sessions = [server.open_session() for _ in range(case["sessions"])]
    flat, views = _image_set([(w, h)] * len(sessions), counts=True, histogram=True)
    toggles, held = ([np.asarray(t, dtype=np.int32) for t in sets] for sets in _toggles(case))
    for session, ids in zip(sessions, held):
        server.request(session, ids)
    server.drain()
    return {"kind": "serve", "server": server, "sessions": sessions, "toggles": toggles, "views": views, "out": flat}


# --- one pass ----------------------------------------------------------------

def run(state):
    kind, out = state["kind"], state["out"]
    if kind == "oneshot":
        binding.composite_oneshot_static(state["members"], out["counts"], out["bucket"], out["rgba"])
        return out
    if kind == "compose":
        comp = state["comp"]
        comp.clear()
        comp.add(state["members"])
        if "mean" in out:
            comp.render(mean_out=out["mean"])
        else:
            comp.render(out["counts"], out["bucket"], out["rgba"])
        return out
    if kind == "toggle":
        comp, k, at = state["comp"], state["swap"], state["outside"]
        members = state["members"]
        # the list's first and second k members take turns in the composite
        comp.remove(members[k - at:2 * k - at])
        comp.add(members[at:at + k])
        state["outside"] = k - at
        comp.render_histogram(out["histogram"], out["counts"], out["bucket"], out["rgba"])
        return out
    if kind == "batch":
        eng = state["engine"]
        if state["graph"]:
            eng.replay()
        else:
            eng.clear_many(state["planes"])
            eng.submit(state["ops"])
            eng.render(state["rops"])
        return out
    server = state["server"]
    for session, toggle, o in zip(state["sessions"], state["toggles"], state["views"]):
        server.request(session, toggle, o["counts"], o["bucket"], o["rgba"], o["histogram"])
    server.drain()
    return out


# --- what a pass cannot do without ---------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = 0
        for i, (w, h, n) in enumerate(_batch_requests(case)):
            total += w * h * ((max(1, n // 2) if i % 4 == 3 else n) + 5) + (2048 if case["histogram"] else 0)
        return {"bytes": total, "flops": 0}
    px = case["width"] * case["height"]
    if kind == "serve":
        row = _row_bytes(case["data"], case["width"]) * case["height"]
        toggles, _ = _toggles(case)
        outputs = 9 * px + 2048
        planes = 8 * px   # each session's composite, updated in place
        return {"bytes": sum(len(t) for t in toggles) * row + len(toggles) * (outputs + planes), "flops": 0}
    raster = _row_bytes(case.get("data", "bytes"), case["width"]) * case["height"]
    if kind == "oneshot":
        return {"bytes": case["members"] * raster + 9 * px, "flops": 0}
    if kind == "toggle":
        count = case["count_bits"] // 8
        return {"bytes": 2 * case["swap"] * raster + px * (3 * count + 5) + 2048, "flops": 0}
    if case["data"] == "depths":
        return {"bytes": case["members"] * raster + 4 * px, "flops": px * case["members"]}
    return {"bytes": case["members"] * raster + px * (case["count_bits"] // 8 + 5), "flops": 0}


def exact(case, seed):
    """Mean depths in 64 bits; counts, classes and colours are whole numbers."""
    if case.get("data") != "depths":
        return None
    gen = _generator(seed)
    members = _rasters(gen, case["width"], case["height"], case["members"], "depths", case["memory"])
    total = torch.zeros(members.shape[1:], dtype=torch.float64, device=DEVICE)
    for m in members:
        total += m.to(DEVICE).double()
    return {"mean": total / case["members"]}
