"""The plain path's analysis over its whole range of conditioning, from ensembles far narrower than the noise to
ones a thousand times wider, against the FP64 oracle domain by domain."""

import numpy as np
import pytest
import torch

from oracle import etkf, geometry
from paper_1310_5954_gb300 import LETKF, _lib
from paper_1310_5954_gb300 import build as builder

from _gpu_common import domain_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


def _analysis(prec, m, spread, seed=0, read_t=False):
    """One analysis of an 8 x 8 system (domains of 24 to 72 slopes) whose ensemble has the given spread / sigma:
    (per-domain errors of mean and anomalies, eigenvalues of I + G / (m-1) of each domain, result, status, oracle's
    result).  read_t: rows of the first instant, which is not observed, have one member that differs each, and the
    innovation is zero (members of the second instant in pairs of either sign, slopes zero)."""
    g = geometry.make_geometry(8, 0.2)
    doms = geometry.make_domains(g, 4, 1)
    rng = np.random.default_rng(1000 * seed + m)
    dt, nd = (torch.float64, np.float64) if prec == "fp64" else (torch.float32, np.float32)
    X = np.vstack([rng.standard_normal((g.n_act, m)), np.cumsum(rng.standard_normal((g.n_act, m)), axis=0) / 4.0])
    if read_t:
        X[:g.n_act] = np.arange(m) == (np.arange(g.n_act) % m)[:, None]
        X[g.n_act:, 1::2] = -X[g.n_act:, ::2]
    X = (0.1 * spread * X).astype(nd).astype(np.float64)
    y = ((0.0 if read_t else 0.3) * rng.standard_normal(g.p)).astype(nd).astype(np.float64)
    f = LETKF(n_sub=8, m=m, ar1_a=0.9, sigma=0.1, dom_sub=4, halo=1, obstruction=0.2, q_white=0.1, precision=prec,
              path="plain", seed=1)
    f.set_state(torch.as_tensor(X, dtype=dt, device="cuda"), 0)
    f.analyze(torch.as_tensor(y, dtype=dt, device="cuda"))
    xa = f.get_state()[0].cpu().numpy().astype(np.float64)
    status = f.sync()
    f.close()
    o = etkf.OracleFilter(g, doms, m, 0.9, 0.1, seed=1, q_white=0.1, X0=X)
    Y = o.C @ X
    Yp = (Y - Y.mean(axis=1, keepdims=True)) / 0.1
    sv = [np.linalg.svd(Yp[d.obs_rows(g.n_subv)], compute_uv=False) for d in doms]
    lam = [1.0 + s * s / (m - 1) for s in sv]
    o.analyze(y)
    return domain_errors(xa, o.X, doms, g.n_act), lam, xa, status, o.X


# An ensemble that narrow is left as it is but for rounding: the reduction and what starts from it move T by a
# few units of roundoff (kappa = 1), as in test_gpu_plain_eig.py; its mean by no more than its anomalies times w_bar.
@pytest.mark.parametrize("prec,m", [("fp32", 20), ("fp32", 50), ("fp32", 100), ("fp64", 20), ("fp64", 100)])
@pytest.mark.parametrize("e", [-12, -11.5, -11, -10.5, -10, -9.5, -9, -8, -6])
def test_narrow_ensembles(prec, m, e):
    if prec == "fp64":
        e *= 7.7          # FP64: squares of 1e-77 are as far out of range as FP32's of 1e-10
    err, _, _, status, _ = _analysis(prec, m, 10.0 ** e)
    assert status == 0
    assert max(max(q) for q in err) <= 31.0 * 2.0 ** (-53 if prec == "fp64" else -24)


# More slopes than members: G has full rank but for the constant direction, which no anomaly has a part in.
# Rounding G moves its smallest eigenvalue by p u |G|, T along its eigenvector by half of that relative to it
# (kappa_eff: the ratio of the largest to the smallest eigenvalue away from the constant direction), and
# rotations that keep small eigenvalues to working accuracy add their own m u; a reduction accurate only beside
# |G| would lose kappa u.
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m", [16, 20])
@pytest.mark.parametrize("e", [1.5, 2.5, 3, 3.5])
def test_wide_ensembles_of_full_rank(prec, m, e):
    u = 2.0 ** (-53 if prec == "fp64" else -24)
    for seed in range(2):
        err, lam, _, status, _ = _analysis(prec, m, 10.0 ** e, seed)
        assert status == 0
        for q, l in zip(err, lam):
            if l.size >= m:                                   # m - 1 eigenvalues away from the constant direction
                assert max(q) <= (72.0 + 30.0) * u * l[0] / l[m - 2], (l[0], l[m - 2], q)


# Fewer slopes than members: the eigenvalue 1 belongs to the anomalies as well, and rounding G loses kappa u of it.
@pytest.mark.parametrize("m", [50, 100])
@pytest.mark.parametrize("e", [2, 2.5, 3])
def test_wide_ensembles_of_low_rank(m, e):
    err, lam, _, status, _ = _analysis("fp32", m, 10.0 ** e)
    assert status == 0
    for q, l in zip(err, lam):
        assert max(q) <= (l[0] + 30.0) * 2.0 ** -24, (l[0], q)


@pytest.mark.parametrize("m", [20, 50, 100])
@pytest.mark.parametrize("e", [3.5, 4, 4.5, 6])
def test_past_the_range_is_finite_or_reported(m, e):
    _, _, xa, status, _ = _analysis("fp32", m, 10.0 ** e)
    assert np.isfinite(xa).all() or status == _lib.LETKF_ENOCONV


# T is the identity to 1e-8 or better and w_bar zero, so that a row whose anomalies are e_j - 1/m reads T's column j:
# one product that counts, and the rounding of T's entry, of the centring and of the sum with the mean, each at most
# u = 2^-24 of the row's one large entry.
@pytest.mark.parametrize("m", [20, 50, 100, 160])
@pytest.mark.parametrize("e", [-9, -7, -6, -5, -4.5])
def test_muted_slopes_leave_the_identity(m, e):
    _, _, xa, status, xo = _analysis("fp32", m, 10.0 ** e, read_t=True)
    assert status == 0
    n = xa.shape[0] // 2
    a, o = xa[:n] - xa[:n].mean(axis=1, keepdims=True), xo[:n] - xo[:n].mean(axis=1, keepdims=True)
    assert (np.linalg.norm(a - o, axis=1) <= 4.0 * 2.0 ** -24 * np.linalg.norm(o, axis=1)).all()
