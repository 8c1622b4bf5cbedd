"""Tensor-core FP64 products of few columns: each width takes a tile of its own (16 to 128 columns) and up
to 64 columns accumulators per digit diagonal.  Against extended precision, within 1e-12 of sum |a||b| (the
bound of the 128-column tiles, whose shared accumulator rounds most), and bit for bit for integers."""
import numpy as np
import pytest
import torch

from paper_2410_04204_gb300 import inputs
from tests.test_gpu_dgemm_tc import dgemm_tc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("N", [1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("M,K", [(1, 1), (129, 31), (300, 2049)])
def test_widths(M, N, K):
    g = inputs.rng(1000 * N + K)
    A = g.normal(size=(M, K)) * 10.0 ** g.uniform(-3, 3, (M, 1))
    B = g.normal(size=(N, K)) * 10.0 ** g.uniform(-3, 3, (N, 1))
    C = dgemm_tc(A, B)
    ref = (A.astype(np.longdouble) @ B.astype(np.longdouble).T).astype(np.float64)
    assert (np.abs(C - ref) <= 1e-12 * (np.abs(A) @ np.abs(B).T)).all()
    Ai = g.integers(-2 ** 13, 2 ** 13 + 1, (M, K)).astype(np.float64)
    Bi = g.integers(-2 ** 13, 2 ** 13 + 1, (N, K)).astype(np.float64)
    assert np.array_equal(dgemm_tc(Ai, Bi), (Ai.astype(np.int64) @ Bi.astype(np.int64).T).astype(np.float64))
