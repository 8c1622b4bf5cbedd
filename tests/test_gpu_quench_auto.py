"""The quench's ways to <sigma^x>(t) against the eigen-decomposition (method 1): the automatic choice, the one
launch of few small variants and the tensor-core steps of many, moments and states, sets that are and are not closed
under the reflection, several and negative fields, the metric of Eq. 11.  Bound: 1e-9, as everywhere for
<sigma^x>(t) (the expansion's own error is about K eps R / (L |h_x|) < 1e-11 here)."""
import numpy as np
import pytest
import torch

from paper_2410_04204_gb300 import tgba

pytestmark = pytest.mark.gpu
L, H0 = 24, 0.5


@pytest.fixture(scope="module")
def basis():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    b = tgba.tgba_build_basis(L, 1.0, [0], 6, 11.0)
    tgba.tgba_compute_x(b)
    yield b
    tgba.tgba_basis_free(b)


def _run(b, hx, trunc, order, t_max, n_t, method, eps):
    nv = len(hx)
    mx = torch.full((nv * n_t,), float("nan"), dtype=torch.float64, device="cuda")
    nrm = torch.full((nv,), float("nan"), dtype=torch.float64, device="cuda")
    ep = torch.full((nv - 1,), float("nan"), dtype=torch.float64, device="cuda") if eps else None
    chi = tgba.tgba_quench_ordered(b, 0, H0, hx, trunc, order, t_max, n_t, mx, nrm, ep, method=method)
    return list(chi), mx.cpu().numpy(), nrm.cpu().numpy(), None if ep is None else ep.cpu().numpy()


ALL = 1e9      # a cutoff beyond every state


@pytest.mark.parametrize("hx,trunc,order,t_max,n_t,method,eps", [
    ([0.3], [ALL], 0, 20.0, 33, 0, False),                                  # one variant
    ([0.3, -0.2, 0.3], [8.0, 9.5, ALL], 0, 20.0, 33, 0, False),
    ([0.25] * 3, [150.0, 301.0, 600.0], 1, 20.0, 33, 0, True),              # the sets may cut a mirror pair
    ([0.25, 0.2], [400.0, 402.0], 1, 20.0, 1, 0, True),                     # one time
    ([0.25] * 5, [17.0, 33.0, 64.0, 65.0, 700.0], 1, 10.0, 300, 2, False),
    ([0.05 * i for i in range(1, 10)], [ALL] * 9, 0, 10.0, 33, 0, False),   # more than one launch takes
    ([0.4], [6.0], 0, 150.0, 65, 2, False),                                 # long: states instead of moments
    ([0.4, 0.1], [4.5, 6.0], 0, 90.0, 65, 2, False),
    ([0.01], [ALL], 0, 20.0, 33, 0, False),                                 # a weak field: not read off the energy
    ([0.3], [ALL], 0, 0.0, 3, 0, False),                                    # no time passes
])
def test_against_eigenvectors(basis, hx, trunc, order, t_max, n_t, method, eps):
    got = _run(basis, hx, trunc, order, t_max, n_t, method, eps)
    ref = _run(basis, hx, trunc, order, t_max, n_t, 1, eps)
    assert got[0] == ref[0]
    assert np.abs(got[1] - ref[1]).max() < 1e-9
    assert np.abs(got[2] - ref[2]).max() < 1e-12
    if eps:
        assert np.abs(got[3] - ref[3]).max() < 1e-9


def test_capped_basis_is_not_closed():
    b = tgba.tgba_build_basis(20, 1.0, [0], 6, -1.0, 351)
    try:
        tgba.tgba_compute_x(b)
        got = _run(b, [0.3, 0.2], [ALL, 8.0], 0, 10.0, 17, 0, False)
        ref = _run(b, [0.3, 0.2], [ALL, 8.0], 0, 10.0, 17, 1, False)
        assert got[0] == ref[0] and np.abs(got[1] - ref[1]).max() < 1e-9
    finally:
        tgba.tgba_basis_free(b)
