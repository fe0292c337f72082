"""The full cycle's adjoint on grids a few columns wide, where every particle's stencils wrap, and one column
off a warp. Cold electrons in a strong pulse make the intensity gradient come from the field and current
transposes. Gradients against the oracle's FP64 reverse sweep, with the tolerances of the same comparison on
the wider grid (1e-4 for the loss, 2e-3 for the intensity)."""
import pytest

from tests.test_gpu_adjoint import _both_full, gb, rel, small_full  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [3, 5, 31, 33])
def test_intensity_gradient_on_narrow_grids(gb, nx):  # noqa: F811
    w = small_full(T_electron_eV=0.01, I0=1e19, nx=nx)
    (L, gD, gR, gI), (Lo, gDo, gRo, gIo) = _both_full(gb, w, 12, 1e-3)
    assert gIo > 0.0
    assert rel(L, Lo) < 1e-4 and rel(gI, gIo) < 2e-3
