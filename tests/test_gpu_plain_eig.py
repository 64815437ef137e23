"""The plain path's inverse square root (tridiagonal form, quadrature, reflectors) at the edges of its
template and shared-memory ranges, against the FP64 oracle.

Bound of each domain's analysis relative to the oracle's, FP32: the reduction and the Gram it starts
from are backward stable, so T moves by at most kappa times the unit roundoff (kappa = cond((m-1)I + G)),
plus a few roundings of the sums that follow; the oracle is exact beside that.  FP64: both sides carry
such errors; the plain path's FP64 per-domain bound of test_gpu_plain.py, 1e-9.
"""

import numpy as np
import pytest
import torch

from oracle import etkf, geometry
from paper_1310_5954_gb300 import LETKF, build as builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


CASES = [("fp64", m) for m in (2, 3, 31, 32, 33, 64, 65, 115, 116, 118)] + \
        [("fp32", m) for m in (2, 3, 5, 32, 33, 64, 65, 127, 128, 129, 160, 165, 166, 168)]


@pytest.mark.parametrize("spread", [0.05, 2.0])     # well conditioned, and the first frames' kappa
@pytest.mark.parametrize("prec,m", CASES)
def test_analysis_over_ensemble_sizes(prec, m, spread):
    g = geometry.make_geometry(8, 0.2)
    doms = geometry.make_domains(g, 4, 1)
    rng = np.random.default_rng(100 * m + int(10 * spread))
    dt, np_dt = (torch.float64, np.float64) if prec == "fp64" else (torch.float32, np.float32)
    smooth = np.cumsum(rng.standard_normal((g.n_act, m)), axis=0) / 4.0
    X = np.vstack([rng.standard_normal((g.n_act, m)), smooth]) * spread + 3.0
    X = X.astype(np_dt).astype(np.float64)
    y = rng.standard_normal(g.p).astype(np_dt).astype(np.float64)
    f = LETKF(n_sub=8, m=m, ar1_a=0.9, sigma=0.1, dom_sub=4, halo=1, obstruction=0.2, q_white=0.1, precision=prec,
              path="plain", seed=1)
    f.set_state(torch.as_tensor(X, dtype=dt, device="cuda"), 0)
    f.analyze(torch.as_tensor(y, dtype=dt, device="cuda"))
    xa = f.get_state()[0].cpu().numpy().astype(np.float64)
    assert f.sync() == 0
    f.close()
    o = etkf.OracleFilter(g, doms, m, 0.9, 0.1, seed=1, q_white=0.1, X0=X)
    C = o.C
    o.analyze(y)
    Y = C @ X
    Yp = Y - Y.mean(axis=1, keepdims=True)
    for d in doms:
        r = d.rows(g.n_act)
        S = Yp[d.obs_rows(g.n_subv)] / 0.1
        kappa = 1.0 + np.linalg.norm(S, 2) ** 2 / (m - 1) if S.size else 1.0
        err = np.linalg.norm(xa[r] - o.X[r]) / np.linalg.norm(o.X[r])
        assert err <= (1e-9 if prec == "fp64" else (kappa + 30.0) * 2.0 ** -24), (m, kappa, err)
