"""The FP32 / FP64 process-noise draw V = L xi at the edges of its tile shapes, against the oracle's normals.

Bound: every element of V sums at most n_act products in working precision; relative to ||V||, 2e-6 (FP32) and
1e-13 (FP64), the bounds stated for this draw.
"""

import numpy as np
import pytest
import torch

from oracle import geometry, philox
from paper_1310_5954_gb300 import LETKF, build as builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


# systems of 9, 69, 437 .. 553 (around 512) and 2117 actuators; ensemble widths around the tile widths
CASES = [(n, m, prec) for n in (2, 8, 22, 24, 50) for m, prec in
         ((2, "fp64"), (24, "fp64"), (25, "fp64"), (65, "fp64"), (20, "fp32"), (33, "fp32"), (97, "fp32"), (113, "fp32"))]
CASES += [(8, 128, "fp32"), (8, 129, "fp32"), (24, 256, "fp32"), (50, 200, "fp32")]


@pytest.mark.parametrize("lower", [True, False])
@pytest.mark.parametrize("n,m,prec", CASES)
def test_draw_matches_normals(n, m, prec, lower):
    g = geometry.make_geometry(n)
    rng = np.random.default_rng(1000 * n + m)
    L = rng.standard_normal((g.n_act, g.n_act)) / np.sqrt(g.n_act)
    if lower:
        L = np.tril(L)
    path = "fused" if m > 128 else "plain"
    f = LETKF(n_sub=n, m=m, ar1_a=0.0, sigma=0.1, dom_sub=4, halo=1, q_sqrt=L, precision=prec, path=path, seed=77)
    f.set_state(torch.zeros((f.info.n, m), dtype=f.dtype, device="cuda"), 5)
    draws = []
    for _ in range(2):
        f.set_state(torch.zeros((f.info.n, m), dtype=f.dtype, device="cuda"), 5)
        f.forecast()
        draws.append(f.get_state()[0][: g.n_act].clone())
    assert f.sync() == 0
    f.close()
    assert torch.equal(draws[0], draws[1])
    ref = L @ philox.normals(77, 1, 5, m, g.n_act)
    err = np.linalg.norm(draws[0].cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= (1e-13 if prec == "fp64" else 2e-6), err
