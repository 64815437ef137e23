"""The plain path's slopes, Gram and transform where the domains fill the SMs (one CTA per domain), at ensemble
sizes for which 16, 8, 4, 2 and 1 lanes share a block of the Gram, the last with more blocks than one pass
takes; odd sizes leave partial blocks.  Against the FP64 oracle with the bounds of the eigensolver's sizes
test: FP32 (kappa + 30) units of roundoff per domain, FP64 1e-9."""

import numpy as np
import pytest
import torch

from oracle import etkf, geometry
from paper_1310_5954_gb300 import LETKF, build as builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


@pytest.mark.parametrize("prec,m", [("fp32", 19), ("fp32", 25), ("fp32", 43), ("fp32", 51), ("fp32", 66),
                                    ("fp32", 101), ("fp64", 18), ("fp64", 45), ("fp64", 67)])
def test_one_cta_per_domain(prec, m):
    g = geometry.make_geometry(48, 0.2)
    doms = geometry.make_domains(g, 4, 1)
    assert len(doms) > 76
    rng = np.random.default_rng(m)
    dt, np_dt = (torch.float64, np.float64) if prec == "fp64" else (torch.float32, np.float32)
    X = (rng.standard_normal((2 * g.n_act, m)) + 3.0).astype(np_dt).astype(np.float64)
    y = rng.standard_normal(g.p).astype(np_dt).astype(np.float64)
    f = LETKF(n_sub=48, m=m, ar1_a=0.9, sigma=0.1, dom_sub=4, halo=1, obstruction=0.2, q_white=0.1, precision=prec,
              path="plain", seed=1)
    f.set_state(torch.as_tensor(X, dtype=dt, device="cuda"), 0)
    f.analyze(torch.as_tensor(y, dtype=dt, device="cuda"))
    xa = f.get_state()[0].cpu().numpy().astype(np.float64)
    assert f.sync() == 0
    f.close()
    o = etkf.OracleFilter(g, doms, m, 0.9, 0.1, seed=1, q_white=0.1, X0=X)
    Y = o.C @ X
    o.analyze(y)
    Yp = Y - Y.mean(axis=1, keepdims=True)
    for d in doms:
        r = d.rows(g.n_act)
        S = Yp[d.obs_rows(g.n_subv)] / 0.1
        kappa = 1.0 + np.linalg.norm(S, 2) ** 2 / (m - 1) if S.size else 1.0
        err = np.linalg.norm(xa[r] - o.X[r]) / np.linalg.norm(o.X[r])
        assert err <= (1e-9 if prec == "fp64" else (kappa + 30.0) * 2.0 ** -24), (m, kappa, err)
