"""The grids letkf_autotune chooses from: all SMs, or the fewest CTAs that take as many rounds of domains as all
SMs full of CTAs, two of which fit an SM where there are more domains than SMs (ensembles of at most 127)."""

import pytest
import torch

from paper_1310_5954_gb300 import LETKF
from paper_1310_5954_gb300 import build as builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()


@pytest.mark.parametrize("n_sub,m,two", [(60, 50, True), (80, 100, True), (40, 50, False), (64, 160, False)])
def test_best_is_one_of_the_candidates(n_sub, m, two):
    f = LETKF(n_sub=n_sub, m=m, ar1_a=0.99, sigma=0.2, dom_sub=4, halo=2, obstruction=0.28, q_white=0.05,
              precision="mixed", path="fused", seed=3)
    sms, n = torch.cuda.get_device_properties(0).multi_processor_count, f.info.n_domains
    per = 2 if two else 1
    assert (n > sms) or not two
    rounds = -(-n // (per * sms))
    fewest = -(-(-(-n // rounds)) // per)
    rec = f.autotune(torch.zeros(f.info.p, dtype=torch.float32, device="cuda"), frames=5)
    f.close()
    assert rec["tuning"]["fused_grid"] in (min(sms, n), fewest) and rec["ms_per_frame"] > 0
