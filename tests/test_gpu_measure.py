"""S(k, w)'s levels and weights from the spectral measure of the tridiagonalised H_eff (reflectors kept,
divide and conquer carrying three rows) against dense eigenvectors of the assembled H_eff: leaf-sized
and ragged sizes, both kinds of self-mirrored sectors and others, truncations that are not closed
under the reflection, strong and complete deflation (h_x small and zero)."""
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


def heff_blocks(b, hx):
    H = torch.empty(tgba.tgba_basis_totals(b)[2], dtype=torch.complex128, device="cuda")
    tgba.tgba_assemble_heff(b, hx, H)
    out, off = [], 0
    for x, y in tgba.tgba_sector_sizes(b):
        out.append(H[off:off + (x + y) ** 2].view(x + y, x + y).T.contiguous())
        off += (x + y) ** 2
    return out


def level_sums(E, w, tol):
    cuts = np.flatnonzero(np.diff(E) > tol) + 1
    return np.add.reduceat(w, np.concatenate([[0], cuts]))


@pytest.mark.parametrize("L,h,mq,cut,cap", [
    (4, 1.3, 4, -1.0, 0), (8, 1.0, 4, -1.0, 0), (10, 0.6, 6, -1.0, 0), (12, 1.0, 6, -1.0, 0),
    (14, 1.2, 6, -1.0, 0), (16, 1.0, 6, -1.0, 83), (24, 1.0, 6, 9.0, 0), (40, 1.0, 6, 6.6, 0)])
@pytest.mark.parametrize("hx", [0.1, 1e-9, 0.0])
def test_k0_weights(L, h, mq, cut, cap, hx):
    b = tgba.tgba_build_basis(L, h, [0], mq, cut, cap)
    try:
        tgba.tgba_compute_x(b)
        nns, nr = tgba.tgba_sector_sizes(b)[0]
        n = nns + nr
        f = lambda k: torch.full((k,), float("nan"), dtype=torch.float64, device="cuda")  # noqa: E731
        S = torch.empty(300, dtype=torch.float32, device="cuda")
        ev, w, dE = f(n), f(n), f(n)
        tgba.tgba_dsf(b, 0, hx, 0.0, 8.0, 300, 0.05, S, ev, n, w, dE)
        E, U = torch.linalg.eigh(heff_blocks(b, hx)[0])
        X = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
        x = torch.empty(nns * nr, dtype=torch.complex128, device="cuda")
        if nns * nr:
            tgba.tgba_x_export(b, 0, x)
            X[:nns, nns:] = x.view(nns, nr)
            X[nns:, :nns] = X[:nns, nns:].conj().T
        E = E.cpu().numpy()
        scale = np.abs(E).max()
        assert np.abs(ev.cpu().numpy() - E).max() <= 1e-12 * scale
        if E[1] - E[0] <= 1e-8 * scale:
            return                                   # no unique ground state
        wo = (L * (U.conj().T @ (X @ U[:, 0])).abs() ** 2).cpu().numpy()
        got, dg = w.cpu().numpy(), dE.cpu().numpy()
        assert np.abs(dg - (E - E[0])).max() <= 2e-12 * scale
        tol = 1e-7 * scale
        assert np.abs(level_sums(E, got, tol) - level_sums(E, wo, tol)).max() <= 1e-9 * wo.max()
        assert abs(got.sum() - wo.sum()) <= 1e-11 * wo.sum()
    finally:
        tgba.tgba_basis_free(b)


@pytest.mark.parametrize("L,mq,cut,sectors,s", [(12, 6, -1.0, [0, 6], 1), (12, 6, -1.0, [3, 0], 0), (24, 6, 9.0, [0, 12], 1),
                                                (24, 6, 9.5, [0, 5], 1), (10, 4, -1.0, [0, 9, 1], 2)])
def test_weights_at_momentum(L, mq, cut, sectors, s):
    hx, h, s0 = 0.15, 1.0, sectors.index(0)
    b = tgba.tgba_build_basis(L, h, sectors, mq, cut)
    try:
        tgba.tgba_compute_x(b)
        n = sum(tgba.tgba_sector_sizes(b)[s])
        S = torch.empty(64, dtype=torch.float32, device="cuda")
        ev, w, dE = (torch.full((n,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(3))
        tgba.tgba_dsf_k(b, s, s0, hx, 0.0, 8.0, 64, 0.05, S, ev, n, w, dE)
        H = heff_blocks(b, hx)
        E = torch.linalg.eigvalsh(H[s]).cpu().numpy()
        e0 = torch.linalg.eigvalsh(H[s0])[0].item()
        assert np.abs(ev.cpu().numpy() - E).max() <= 1e-12 * np.abs(E).max()
        assert np.abs(dE.cpu().numpy() - (E - e0)).max() <= 2e-12 * np.abs(E).max()
        assert np.isfinite(w.cpu().numpy()).all() and (w >= 0).all()
    finally:
        tgba.tgba_basis_free(b)
