"""Draws of dense process noise on two streams at once: a fused step draws the next frame's block on a side stream,
and letkf_forecast draws its own on the context's stream.  Neither may write what the other reads, so the result
of calls queued back to back is that of the same calls with the device idle in between, bit for bit."""

import pytest
import torch

from paper_1310_5954_gb300 import build as builder

from _gpu_common import gpu_filter, slopes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


def _run(name, prec, idle):
    y, _ = slopes(name, 4)
    ys = [torch.as_tensor(v, dtype=torch.float32, device="cuda") for v in y]
    f = gpu_filter(name, prec, "fused")
    for k in range(4):
        f.step(ys[k % 2])
        idle()
        f.analyze(ys[2])
        f.forecast()
        idle()
        f.step(ys[3])
        idle()
    out = f.get_state()[0].clone()
    assert f.sync() == 0
    f.close()
    return out


@pytest.mark.parametrize("name,prec", [("vlt-40x40", "mixed"), ("vlt-40x40", "fp32"), ("elt-80x80", "mixed"),
                                       ("elt-80x80", "fp32")])
def test_forecast_beside_the_look_ahead(name, prec):
    a = _run(name, prec, lambda: None)
    b = _run(name, prec, torch.cuda.synchronize)
    assert torch.equal(a, b)


@pytest.mark.parametrize("prec", ["mixed", "fp32"])
def test_captured_forecast(prec):
    """letkf_forecast in a CUDA graph of the caller's, launched behind a step's look-ahead, and a step behind it."""
    y, _ = slopes("vlt-40x40", 4)
    ys = [torch.as_tensor(v, dtype=torch.float32, device="cuda") for v in y]
    out = []
    for captured in (False, True):
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            f = gpu_filter("vlt-40x40", prec, "fused")
            f.step(ys[0])
            f.analyze(ys[1])
            if captured:
                s.synchronize()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s):
                    f.forecast()
                g.replay()
            else:
                f.forecast()
            f.step(ys[2])
            out.append(f.get_state()[0].clone())
            assert f.sync() == 0
            f.close()
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("name,prec", [("vlt-40x40", "mixed"), ("elt-80x80", "fp32")])
@pytest.mark.parametrize("back", [1, 2, 5])
def test_another_frame_behind_a_graph_step(name, prec, back):
    """Steps as graphs draw the next frame's block; set_state to another frame has it drawn on the side stream."""
    y, _ = slopes(name, 4)
    ys = [torch.as_tensor(v, dtype=torch.float32, device="cuda") for v in y]
    out = []
    for idle in (lambda: None, torch.cuda.synchronize):
        f = gpu_filter(name, prec, "fused")
        f.set_graph(True)
        x0 = f.get_state()[0].clone()
        for k in range(4):
            f.step(ys[k % 3])
            f.step(ys[k % 3])
            f.set_state(x0, 10 * k + back)
            idle()
            f.step(ys[3])
            f.step(ys[0])
            idle()
        out.append(f.get_state()[0].clone())
        assert f.sync() == 0
        f.close()
    assert torch.equal(out[0], out[1])
