"""The CUDA-core analysis of small domains in its observation-space form (at most 32 slopes, fewer than members) at
high conditioning, against the FP64 oracle domain by domain.

Bound: the factors of T = I - S^T Z (I + Z)^-1 Z S / c are formed by about ten FP32 products of up to 32 terms, each
of which rounds by sqrt(32) u < 6 u (u = 2^-24) of entries up to 1; applied one after another to X'_E S^T, which is
sqrt(c kappa) times X'_E at most, they lose 60 sqrt(kappa) u of the anomalies, and not kappa u.  The iteration's last
step starts from ||I - P|| < 2e-2 and leaves 3/8 of its square, 1.5e-4, in Z.  Kappa u stays well below one."""

import numpy as np
import pytest
import torch

from oracle import etkf, geometry
from paper_1310_5954_gb300 import LETKF
from paper_1310_5954_gb300 import build as builder

from _gpu_common import domain_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


@pytest.mark.parametrize("n_sub", [8, 32])      # one CTA per SM; two (more domains than SMs)
@pytest.mark.parametrize("m", [33, 50, 100])
@pytest.mark.parametrize("prec", ["fp32", "mixed"])
@pytest.mark.parametrize("e", [1, 2, 2.5])
def test_error_grows_with_the_root_of_kappa(n_sub, m, prec, e):
    g = geometry.make_geometry(n_sub, 0.2)
    doms = geometry.make_domains(g, 2, 1)
    rng = np.random.default_rng(m)
    X = np.vstack([rng.standard_normal((g.n_act, m)), np.cumsum(rng.standard_normal((g.n_act, m)), axis=0) / 4.0])
    X = (0.1 * 10.0 ** e * X).astype(np.float32).astype(np.float64)
    y = (0.3 * rng.standard_normal(g.p)).astype(np.float32).astype(np.float64)
    f = LETKF(n_sub=n_sub, m=m, ar1_a=0.9, sigma=0.1, dom_sub=2, halo=1, obstruction=0.2, q_white=0.1, precision=prec,
              path="fused", seed=1)
    assert f.info.n_domains_simt == f.info.n_domains_observing and (f.info.n_domains > 152) == (n_sub == 32)
    f.set_state(torch.as_tensor(X, dtype=torch.float32, device="cuda"), 0)
    f.analyze(torch.as_tensor(y, dtype=torch.float32, device="cuda"))
    xa = f.get_state()[0].cpu().numpy().astype(np.float64)
    f.close()
    o = etkf.OracleFilter(g, doms, m, 0.9, 0.1, seed=1, q_white=0.1, X0=X)
    Y = o.C @ X
    Yp = (Y - Y.mean(axis=1, keepdims=True)) / 0.1
    o.analyze(y)
    for d, (_, anom) in zip(doms, domain_errors(xa, o.X, doms, g.n_act)):
        S = Yp[d.obs_rows(g.n_subv)]
        kappa = 1.0 + (np.linalg.norm(S, 2) ** 2 / (m - 1) if S.size else 0.0)
        assert anom <= 1.5e-4 + 60.0 * np.sqrt(kappa) * 2.0 ** -24, (kappa, anom)
