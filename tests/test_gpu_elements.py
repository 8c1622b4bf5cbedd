"""The closed form of the contraction table and the product form of the elements (Schur's Pfaffian
identity) against the general path: the elimination of Eq. S2's matrix (tgba_table_noalloc), Pfaffians
of its rows, and the paper-literal string (tgba_x_direct)."""
import numpy as np
import pytest
import torch

from paper_2410_04204_gb300 import inputs, tgba
from tests.gpu_helpers import GpuSector

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# both phases and the critical point, near and far, every parity of L / 2
@pytest.mark.parametrize("L,h", [(4, 1.0), (4, 2.5), (6, 0.05), (8, 1.4), (22, 1.0), (24, 0.999), (36, 1.7), (20, 8.0),
                                 (64, 0.5), (62, 1.0)])
def test_closed_form_table_equals_the_elimination(L, h):
    """The elimination's own rounding (about 1e-14 of the largest entry at L = 64) sets the bound."""
    b = tgba.tgba_build_basis(L, h, [0], 2)
    try:
        t = torch.empty(4 * L * L, dtype=torch.float64, device="cuda")
        c0 = tgba.tgba_table(b, t)
    finally:
        tgba.tgba_basis_free(b)
    g, gc = torch.empty_like(t), torch.empty(2, dtype=torch.float64, device="cuda")
    tgba.tgba_table_noalloc(L, h, g, gc)
    assert (t - g).abs().max().item() <= 1e-12 * g.abs().max().item()
    assert abs(c0 - complex(*gc.cpu().numpy())) <= 1e-12 * abs(c0)


def pfaffian(A):
    A, v = A.copy(), 1.0
    for k in range(0, len(A), 2):
        p = k + 1 + int(np.argmax(np.abs(A[k + 1:, k])))
        if p != k + 1:
            A[[k + 1, p]] = A[[p, k + 1]]
            A[:, [k + 1, p]] = A[:, [p, k + 1]]
            v = -v
        v *= A[k, k + 1]
        t, r = A[k, k + 2:] / A[k, k + 1], A[k + 1, k + 2:].copy()
        A[k + 2:, k + 2:] += np.outer(r, t) - np.outer(t, r)
    return v


# rows per tile 8, 8, 4, 2 and 1 (L = 14 .. 120), with and without the pair table, ragged last rows
@pytest.mark.parametrize("L,h,mq,cut", [(14, 0.8, 14, -1.0), (24, 1.0, 6, 9.0), (58, 1.0, 6, 5.0), (82, 1.0, 6, 4.0),
                                        (114, 1.0, 4, 3.0), (14, 1.6, 8, -1.0)])
def test_elements_equal_pfaffians_of_the_table(L, h, mq, cut):
    """A Pfaffian of n <= 28 rows of the table by elimination: forward error far below 1e-11 of the
    largest element."""
    b = tgba.tgba_build_basis(L, h, [0, 1], mq, cut)
    try:
        tgba.tgba_compute_x(b)
        t = torch.empty(4 * L * L, dtype=torch.float64, device="cuda")
        c0 = tgba.tgba_table(b, t)
        R = t.cpu().numpy().reshape(2 * L, 2 * L)
        for s in (0, 1):
            g = GpuSector(b, s, mq)
            X = g.x()
            pairs = [tuple(p) for p in inputs.sample_pairs(g.n_ns, g.n_r, 400, tag=L + s)]
            pairs += [(g.n_ns - 1, g.n_r - 1), (0, g.n_r - 1), (g.n_ns - 1, 0)]
            for a, c in pairs:
                ma, mb = g.keys[a][1], g.keys[g.n_ns + c][1]
                sel = [L - 1 - i for i in reversed(ma)] + [L + i for i in mb]
                want = c0 * (-1j) ** (len(sel) // 2) * (pfaffian(R[np.ix_(sel, sel)]) if sel else 1.0)
                assert abs(X[a, c] - want) <= 1e-11 * np.abs(X).max(), (ma, mb)
    finally:
        tgba.tgba_basis_free(b)


@pytest.mark.parametrize("L,h", [(10, 0.6), (12, 1.0), (16, 1.4)])
def test_elements_equal_the_paper_literal_string(L, h):
    b = tgba.tgba_build_basis(L, h, [1], 6)
    try:
        g = GpuSector(b, 0, 6)
        pairs = inputs.sample_pairs(g.n_ns, g.n_r, 500, tag=L).astype(np.int32)
        d = torch.from_numpy(pairs).cuda()
        x, y = (torch.empty(len(pairs), dtype=torch.complex128, device="cuda") for _ in range(2))
        tgba.tgba_x_pairs(b, 0, d, x)
        tgba.tgba_x_direct(b, 0, d, y)
        assert (x - y).abs().max().item() <= 1e-12
    finally:
        tgba.tgba_basis_free(b)
