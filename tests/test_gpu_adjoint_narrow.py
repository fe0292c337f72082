"""D and r0 gradients of the full cycle on grids whose stencils wrap (3 and 5 columns) and one column off a warp: the
comparison and the tolerances of the wide grid (test_full_cycle_gradient_matches_oracle)."""
import pytest

from tests.test_gpu_adjoint import _both_full, gb, rel, small_full  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kin", [0.0, 1e-3])
@pytest.mark.parametrize("nx", [3, 5, 31, 33])
def test_pair_force_gradients_on_narrow_grids(gb, nx, kin):  # noqa: F811
    (L, gD, gR, _), (Lo, gDo, gRo, _) = _both_full(gb, small_full(nx=nx), 6, kin)
    assert rel(L, Lo) < 1e-4
    assert rel(gD, gDo) < 3e-4 and rel(gR, gRo) < 2e-4
