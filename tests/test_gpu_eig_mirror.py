"""Eigenvalues through the reflection symmetry (mirror sectors shared, self-mirrored sectors as even and
odd blocks) against the library solver, which takes every sector whole: all combinations of sectors
present, truncations that are and are not closed under the reflection, one block empty."""
import numpy as np
import pytest
import torch

from paper_2410_04204_gb300 import tgba

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("L,h,sectors,mq,cut,cap", [
    (14, 1.0, list(range(14)), 6, -1.0, 0),        # everything
    (14, 0.7, [11, 0, 3, 7, 5], 6, -1.0, 0),       # a pair out of order, both self-mirrored, one alone
    (16, 1.3, [8, 0], 6, -1.0, 0),
    (16, 1.0, [0, 1, 15, 8], 8, -1.0, 101),        # capped: not closed under the reflection in general
    (24, 1.0, [12, 6, 18], 6, 9.5, 0),
    (12, 1.0, [0], 0, -1.0, 0),                    # the two vacua: no odd block
    (10, 1.5, [0, 5], 4, 0.5, 0),                  # one state; an empty sector
    (60, 1.0, [0, 59, 1], 6, 4.6, 0),
])
def test_against_whole_sectors(L, h, sectors, mq, cut, cap):
    fields = [0.0, 0.13, -0.4]
    b = tgba.tgba_build_basis(L, h, sectors, mq, cut, cap)
    try:
        tgba.tgba_compute_x(b)
        n = sum(x + y for x, y in tgba.tgba_sector_sizes(b))
        ev = [torch.full((len(fields) * n,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(3)]
        for m in range(3):
            tgba.tgba_eigvals(b, fields, ev[m], method=m)
        ref = ev[2].cpu().numpy()
        off = np.concatenate([[0], np.cumsum([x + y for x, y in tgba.tgba_sector_sizes(b)] * len(fields))])
        for m in (0, 1):
            got = ev[m].cpu().numpy()
            assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max() * max(1, n) ** 0.5
            for i, j in zip(off[:-1], off[1:]):
                assert np.all(np.diff(got[i:j]) >= -1e-13 * np.abs(ref).max())
    finally:
        tgba.tgba_basis_free(b)


@pytest.mark.parametrize("L,sectors,mq,cut,fields", [
    (14, [3], 6, -1.0, [0.2]),                                  # one matrix, beyond the rows one CTA finishes
    (24, [5], 4, 9.0, [0.1 * i for i in range(1, 7)]),           # 6: one CTA on an SM
    (24, [5], 4, 9.0, [0.1 * i for i in range(1, 8)]),           # 7: two
    (24, [0], 4, 9.0, [1e-160, 1e-146, 1e-140, 1e-130, 1e-60]),   # columns whose squares underflow
    (24, [5], 4, 9.0, [1e-145, 0.0, 1e3]),
])
def test_few_and_many_matrices(L, sectors, mq, cut, fields):
    """Householder steps with the reflector in the column's scale, chunks dealt out (up to six matrices) and
    drawn by ticket, against the library solver; the bound of test_against_whole_sectors."""
    b = tgba.tgba_build_basis(L, 1.0, sectors, mq, cut)
    try:
        tgba.tgba_compute_x(b)
        n = sum(x + y for x, y in tgba.tgba_sector_sizes(b))
        assert n > 130
        ev = [torch.empty(len(fields) * n, dtype=torch.float64, device="cuda") for _ in range(2)]
        tgba.tgba_eigvals(b, fields, ev[0], method=1)
        tgba.tgba_eigvals(b, fields, ev[1], method=2)
        got, ref = (e.cpu().numpy().reshape(len(fields), n) for e in ev)
        assert (np.abs(got - ref).max(axis=1) <= 1e-12 * np.abs(ref).max(axis=1) * n ** 0.5).all()
    finally:
        tgba.tgba_basis_free(b)
