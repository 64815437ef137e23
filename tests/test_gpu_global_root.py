"""The one-kernel inverse square root and weights of the global path at ensemble sizes around its tiles (64
columns, 128 rows, 64 x 64 blocks of the Gram), against the FP64 oracle with the bound of the global path's
own tests (4 sqrt(kappa) 2^-16, at least 1e-4, derived there); and two filters on two streams at once, whose
cooperative launches must not hold each other up, against the same frames one after the other."""

import numpy as np
import pytest
import torch

from paper_1310_5954_gb300 import LETKF, _lib
from paper_1310_5954_gb300 import build as builder

from _gpu_common import rel, slopes
from test_gpu_global import _kappa, _kw, _oracle, _t, _tol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()
    _lib.load()


@pytest.mark.parametrize("m", [2, 33, 63, 64, 65, 127, 128, 129, 193, 385])
def test_sizes_around_the_tiles(m):
    y, _ = slopes("tiny-8x8", 1)
    f = LETKF(**_kw("tiny-8x8", m))
    o = _oracle("tiny-8x8", m)
    tol = _tol(_kappa(o, y[0]))
    f.analyze(_t(y[0]))
    xa = f.get_state()[0].cpu().numpy().astype(np.float64)
    o.analyze(y[0].astype(np.float32).astype(np.float64))
    assert f.sync() == 0
    assert rel(xa.mean(axis=1), o.X.mean(axis=1)) < tol
    assert rel(xa - xa.mean(axis=1, keepdims=True), o.X - o.X.mean(axis=1, keepdims=True)) < tol
    f.close()


def test_two_filters_on_two_streams():
    y, _ = slopes("tiny-8x8", 6)
    ys = [_t(v) for v in y]
    sizes = (300, 700)
    serial = []
    for m in sizes:
        f = LETKF(**_kw("tiny-8x8", m))
        serial.append([f.step(v).clone() for v in ys])
        assert f.sync() == 0
        f.close()
    streams = [torch.cuda.Stream() for _ in sizes]
    fs, outs = [], [[], []]
    for m, s in zip(sizes, streams):
        with torch.cuda.stream(s):
            fs.append(LETKF(**_kw("tiny-8x8", m)))
    torch.cuda.synchronize()
    for v in ys:
        for q, s in enumerate(streams):
            with torch.cuda.stream(s):
                outs[q].append(fs[q].step(v).clone())
    torch.cuda.synchronize()
    for q in range(2):
        assert fs[q].sync() == 0
        for a, b in zip(outs[q], serial[q]):
            assert torch.equal(a, b)
        fs[q].close()


@pytest.mark.parametrize("ar2", [False, True])
def test_step_with_a_rejected_frame(ar2):
    """A step whose frame is rejected keeps both instants, also where an AR(1) step otherwise writes the first
    instant's analysis only, and the next step goes on from there as the split calls do."""
    over = dict(ar1_a=1.2, ar2_a=-0.3) if ar2 else {}
    y, _ = slopes("tiny-8x8", 3)
    a, b = LETKF(**_kw("tiny-8x8", 150, **over)), LETKF(**_kw("tiny-8x8", 150, **over))
    bad = y[1].copy()
    bad[3] = np.inf
    a.step(_t(y[0]))
    s0 = a.get_state()[0].clone()
    p = a.step(_t(bad))
    assert a.sync() == _lib.LETKF_ENONFINITE
    s1 = a.get_state()[0]
    assert torch.equal(s1, s0)
    n_act = s0.shape[0] // 2
    assert rel(p.cpu().numpy(), s0[:n_act].double().mean(dim=1).cpu().numpy()) < 1e-6
    b.step(_t(y[0]))
    b.analyze(_t(bad))
    b.forecast()
    a.step(_t(y[2]))
    b.analyze(_t(y[2]))
    b.forecast()
    assert torch.equal(a.get_state()[0], b.get_state()[0])
    a.close()
    b.close()
