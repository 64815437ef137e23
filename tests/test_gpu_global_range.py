"""The global path's inverse square root over its whole range of conditioning, s = 1 + |G|_F / (m-1) from 1 (an
ensemble far narrower than the noise) to beyond what FP32 holds, against the FP64 oracle's analysis.

Bound where the arithmetic carries the result, as the global path's tests derive it: 4 sqrt(kappa) 2^-16, at
least 1e-4, kappa = cond(I + G / (m-1))."""

import numpy as np
import pytest
import torch

from oracle import etkf, geometry
from paper_1310_5954_gb300 import LETKF, _lib
from paper_1310_5954_gb300 import build as builder

from _gpu_common import rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()
    _lib.load()


def _analysis(n_sub, m, spread, seed=0):
    """One analysis of a random ensemble with the given spread / sigma: (GPU's, oracle's, kappa, status, steps)."""
    g = geometry.make_geometry(n_sub, 0.3)
    rng = np.random.default_rng(100 * seed + m)
    X = np.vstack([rng.standard_normal((g.n_act, m)), np.cumsum(rng.standard_normal((g.n_act, m)), axis=0) / 4.0])
    X = (0.1 * spread * X).astype(np.float32).astype(np.float64)
    y = (0.3 * rng.standard_normal(g.p)).astype(np.float32).astype(np.float64)
    f = LETKF(n_sub=n_sub, m=m, ar1_a=0.9, sigma=0.1, obstruction=0.3, q_white=0.1, precision="fp32", path="global",
              seed=1)
    f.set_state(torch.as_tensor(X, dtype=torch.float32, device="cuda"), 0)
    f.analyze(torch.as_tensor(y, dtype=torch.float32, device="cuda"))
    xa = f.get_state()[0].cpu().numpy().astype(np.float64)
    status, stats = f.sync(), f.global_stats()
    f.close()
    o = etkf.OracleFilter(g, None, m, 0.9, 0.1, seed=1, q_white=0.1, X0=X)
    Y = o.C @ X
    kappa = 1.0 + np.linalg.norm((Y - Y.mean(axis=1, keepdims=True)) / 0.1, 2) ** 2 / (m - 1)
    o.analyze(y)
    return xa, o.X, kappa, status, stats


def _errors(xa, xo):
    ma, mo = xa.mean(axis=1), xo.mean(axis=1)
    return rel(ma, mo), rel(xa - ma[:, None], xo - mo[:, None])


@pytest.mark.parametrize("n_sub,m", [(32, 100), (16, 64)])
@pytest.mark.parametrize("spread", [1e3, 1e4, 1e5])
def test_a_result_that_is_not_finite_is_reported(n_sub, m, spread):
    # past s ~ 1e7 the iterates of a rank-deficient system overflow the split operands' precision
    xa, _, _, status, _ = _analysis(n_sub, m, spread)
    assert np.isfinite(xa).all() or status == _lib.LETKF_ENOCONV


@pytest.mark.parametrize("n_sub,m", [(32, 197), (40, 300)])
@pytest.mark.parametrize("spread", [30.0, 300.0, 1e3, 1e4])
def test_high_conditioning(n_sub, m, spread):
    # s from 1e5 to 4e10; more slopes than members, so that G has full rank
    xa, xo, kappa, status, _ = _analysis(n_sub, m, spread)
    assert status == 0
    e = _errors(xa, xo)
    assert max(e) <= max(1e-4, 4.0 * np.sqrt(kappa) * 2.0 ** -16), (kappa, e)


# what max |I - P| < 1e-2 on the diagonal leaves of a uniform deviation, 3/8 of its square, and the rounding
# of the iterates: 4 sqrt(kappa) 2^-16 at least 1e-4 covers both at these kappa
@pytest.mark.parametrize("n_sub,m", [(16, 64), (24, 300), (32, 197)])
@pytest.mark.parametrize("spread", [1e-6, 0.01, 0.05, 0.1, 0.126, 0.158, 0.2, 0.25, 0.3, 0.4, 0.5, 0.63])
def test_low_conditioning(n_sub, m, spread):
    for seed in range(3):
        xa, xo, kappa, status, (steps, s) = _analysis(n_sub, m, spread, seed)
        assert status == 0
        e = _errors(xa, xo)
        assert max(e) <= max(1e-4, 4.0 * np.sqrt(kappa) * 2.0 ** -16), (s, steps, kappa, e)
        if spread < 1e-3:
            assert steps == 2, (s, steps)     # G = 0 but for rounding: the first step is exact
