"""Pieces and clusters of the tiled tensor-core product (letkf_gemm_selftest): row tiles that leave a
cluster of two with one to spare, widths that take 256, 128 and 64 columns in one row, a last piece with
one column, K below one step, of one step and ragged, more pieces than SMs and columns that are no multiple
of four (scalar stores).  Against an FP64 product; bound per element from the arithmetic: the three-product
split (3 x 2^-17) and the FP32 accumulation (K 2^-24), times sum_k |A_ik| |B_jk|."""

import numpy as np
import pytest
import torch

from paper_1310_5954_gb300 import _lib
from paper_1310_5954_gb300 import build as builder

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    builder.build()
    _lib.load()


@pytest.mark.parametrize("M,N,K", [(129, 65, 16), (257, 448, 64), (384, 193, 130), (640, 321, 1100),
                                   (128, 256, 48), (5000, 1217, 77)])
@pytest.mark.parametrize("bn,b_mn", [(64, 0), (128, 0), (256, 0), (64, 1)])
def test_pieces_match_fp64(M, N, K, bn, b_mn):
    rng = np.random.default_rng(M + 5 * N + 11 * K)
    A = rng.standard_normal((M, K)).astype(np.float32)
    B = rng.standard_normal((N, K)).astype(np.float32)
    a = torch.as_tensor(A, device="cuda")
    b = torch.as_tensor(np.ascontiguousarray(B.T) if b_mn else B, device="cuda")
    # a guard row behind C: nothing may be written past its last element
    c = torch.full((M + 1, N), np.nan, dtype=torch.float32, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert _lib.load().letkf_gemm_selftest(a.data_ptr(), b.data_ptr(), c.data_ptr(), M, N, K, 1, bn, b_mn, st) == 0
    C = c.cpu().numpy().astype(np.float64)
    assert np.isnan(C[M]).all()
    ref = A.astype(np.float64) @ B.astype(np.float64).T
    scale = np.abs(A).astype(np.float64) @ np.abs(B).astype(np.float64).T
    assert (np.abs(C[:M] - ref) <= (3 * 2.0 ** -17 + K * 2.0 ** -24) * scale).all()
