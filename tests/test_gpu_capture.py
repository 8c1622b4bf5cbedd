"""tgba_compute_x under stream capture: refused, and the basis stays usable with its stage times."""
import pytest
import torch

from paper_2410_04204_gb300 import tgba

pytestmark = pytest.mark.gpu


def test_compute_x_refuses_capture():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = tgba.tgba_build_basis(10, 1.0, [0], 4)
    try:
        tgba.tgba_compute_x(b)
        torch.cuda.synchronize()
        st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
            with pytest.raises(tgba.TgbaError) as e:
                tgba.tgba_compute_x(b, stream=st.cuda_stream)
        assert e.value.code == tgba.TGBA_ECUDA
        tgba.tgba_profile(b)
        tgba.tgba_compute_x(b)
        tgba.tgba_profile(b)
    finally:
        tgba.tgba_basis_free(b)
