"""Clears, folds and renders captured into graphs.  A graph may be replayed
beside other work of its context, on any stream, so a captured histogram render
keeps nothing in the context: it counts into its own output."""
import os
import re

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
from paper_2104_14667_gb300 import binding  # noqa: E402

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_14667_gb300", "csrc")


def test_captured_histograms_take_no_scratch_of_the_context():
    with open(os.path.join(CSRC, "api.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = text.index("int render(composite_ctx")
    render = text[start:text.index("\n}\n", start)]
    device, host = render.split("if (out_on_device) {")[-1].split("return CPT_OK;", 1)
    assert "capturing(ctx->compute) ? nullptr : ctx->hist_scratch" in device and "hist_out, scratch)" in device
    assert "capturing" not in host   # waits for its copies: never captured


def histogram(classes):
    return torch.from_numpy(np.bincount(classes.ravel(), minlength=256)).cuda()


@pytest.mark.gpu
@pytest.mark.parametrize("count_bits", [16, 32])
@pytest.mark.parametrize("w,h", [(200, 33), (1999, 2001)])
def test_histogram_renders_replayed_beside_one_another(w, h, count_bits):
    m = synth.random_masks(w, 9, h, w)
    dev = torch.from_numpy(m).cuda()
    classes = oracle.bucket(oracle.count(m), 9)
    want = histogram(classes)
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = [(torch.full((256,), -1, dtype=torch.int64, device="cuda"),
             torch.empty((h, w), dtype=torch.uint8, device="cuda")) for _ in streams]
    with binding.Composite(w, h, count_bits=count_bits, stream=streams[0].cuda_stream) as comp:
        torch.cuda.synchronize()
        comp.add(dev)
        comp.sync()
        graphs = []
        for hist, bucket in outs[1:]:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=streams[0]):
                comp.render_histogram(hist, bucket_out=bucket)
            graphs.append(g)
        for _ in range(20):
            for hist, bucket in outs:
                hist.fill_(-1)
                bucket.fill_(7)
            torch.cuda.synchronize()
            for _ in range(5):   # the same values each time
                comp.render_histogram(outs[0][0], bucket_out=outs[0][1])
                for g, s in zip(graphs, streams[1:]):
                    with torch.cuda.stream(s):
                        g.replay()
            torch.cuda.synchronize()
            for hist, bucket in outs:
                assert torch.equal(hist, want)
                assert torch.equal(bucket, torch.from_numpy(classes).cuda())


@pytest.mark.gpu
@pytest.mark.parametrize("fmt", ["bytes", "bits"])
def test_clear_folds_and_renders_in_one_graph(fmt):
    w, h = 1500, 701
    m = synth.random_masks(5, 12, h, w)
    dev = torch.from_numpy(synth.pack_masks(m) if fmt == "bits" else m).cuda()
    s = torch.cuda.Stream()
    hists = torch.full((2, 256), -1, dtype=torch.int64, device="cuda")
    classes = torch.empty((2, h, w), dtype=torch.uint8, device="cuda")
    with binding.Composite(w, h, mask_format=fmt, stream=s.cuda_stream) as comp:
        torch.cuda.synchronize()
        comp.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            comp.clear()
            comp.add(dev)
            comp.render_histogram(hists[0], bucket_out=classes[0])
            comp.remove(dev[:1])
            comp.render_histogram(hists[1], bucket_out=classes[1])
        for _ in range(20):
            hists.fill_(-1)
            classes.fill_(7)
            torch.cuda.synchronize()
            for _ in range(4):
                g.replay()
            torch.cuda.synchronize()
            for i, ids in enumerate((m, m[1:])):
                want = oracle.bucket(oracle.count(ids), len(ids))
                assert torch.equal(classes[i], torch.from_numpy(want).cuda())
                assert torch.equal(hists[i], histogram(want))
