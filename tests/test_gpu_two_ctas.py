"""The fused kernel with two CTAs per SM gives the bits of the kernel with one.

A launch takes two CTAs per SM when its systems fit and it has more domains than SMs.  Stepped alone, a
60x60 system does; in one batch with an m = 130 system (observation-space form, one CTA per SM) it does not.
The arithmetic is the same, so predictions and ensembles are equal bit for bit, over ensemble sizes around
the operand widths, both forecast models, the SIMT threshold, both noise kinds and the cold start's
conditioning (high/low split Gram, two refinements).
"""

import numpy as np
import pytest
import torch

from paper_1310_5954_gb300 import LETKF, Server, _lib
from paper_1310_5954_gb300 import build as builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


CASES = [  # m, precision, spread of the ensemble / sigma, other parameters
    (2, "mixed", 0.5, {}), (15, "fp32", 0.5, {}), (16, "mixed", 0.5, {"simt_q_max": -1}), (31, "mixed", 5.0, {}),
    (48, "fp32", 5.0, {"simt_q_max": 64}), (63, "mixed", 0.5, {"ar1_a": 1.58, "ar2_a": -0.585}),
    (64, "fp32", 0.5, {"obs_block": 0}), (79, "mixed", 5.0, {"piston": "in_loop"}), (80, "mixed", 0.5, {}),
    (95, "fp32", 20.0, {}), (96, "mixed", 0.5, {}), (100, "mixed", 0.5, {"ar1_a": 1.58, "ar2_a": -0.585}),
    (100, "fp32", 5.0, {"halo": 1, "simt_q_max": -1}), (111, "mixed", 0.5, {"halo": 1}), (100, "mixed", 1e-4, {}),
]


@pytest.mark.parametrize("m,prec,spread,more", CASES)
def test_same_bits_as_one_cta(m, prec, spread, more):
    kw = dict(n_sub=60, m=m, ar1_a=0.99, sigma=0.2, dom_sub=4, halo=2, obstruction=0.2, q_white=0.05, precision=prec,
              seed=3)
    kw.update(more)
    f = LETKF(path="fused", **kw)
    assert f.info.n_domains > 152
    rng = np.random.default_rng(m)
    X = np.cumsum(rng.standard_normal((f.info.n, m)), axis=0) * 0.1 * spread * 0.2
    X = torch.as_tensor((X - X.mean(axis=0)).astype(np.float32), device="cuda")
    ys = (0.3 * rng.standard_normal((3, f.info.p))).astype(np.float32)
    f.set_state(X, 4)
    alone = [f.step(torch.as_tensor(y, device="cuda")).cpu().numpy().copy() for y in ys]
    assert f.sync() == 0
    xa = f.get_state()[0].cpu().numpy()
    f.close()
    assert np.isfinite(xa).all()

    srv = Server(slots=1, max_pending=4)
    sid = srv.admit(**kw)
    wide = srv.admit(n_sub=8, m=130, ar1_a=0.99, sigma=0.2, dom_sub=4, halo=1, q_white=0.05, seed=5)
    _lib.letkf_set_state(_lib.letkf_server_context(srv.srv, sid), X.data_ptr(), 4)
    torch.cuda.synchronize()
    out = srv.set_output(sid, 7)
    for y in ys:
        assert srv.submit(sid, y) == 0
        assert srv.submit(wide, np.zeros(srv.systems[wide].p, dtype=np.float32)) == 0
        srv.drain()
    assert all(r["batch_systems"] == 2 for r in srv.records())
    xs = srv.state(sid)[0].cpu().numpy()
    srv.close()
    for k in range(3):
        assert np.array_equal(out[4 + k], alone[k]), k
    assert np.array_equal(xs, xa)
