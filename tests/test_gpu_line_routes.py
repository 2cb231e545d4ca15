"""Routes of the z and y passes chosen by size, on both sides of their lines:
FP64 2-D grids past the longest single pass."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

D = (2e-9, 3e-9, 2.5e-9)


def _m(n, seed=0):
    m = np.random.default_rng(seed).normal(size=(3,) + n[::-1])
    return m / np.linalg.norm(m, axis=0)


@pytest.mark.parametrize("ny,one", [(128, True), (135, False), (343, False)])
def test_fp64_2d_grids_transform_y_in_its_own_passes_past_256(ny, one):
    """(A CTA of the one-pass kernel holds one column of longer FP64 lines, half a sector
    of each row, and 512x343x1 took 784 us a stage instead of 558.)"""
    from paper_2302_08843_gb300.binding import State
    n = (24, ny, 1)
    s = State(n, D, "fp64")
    s.set_material(Ms=8e5, A=1e-11, alpha=0.1)
    s.demag_setup(1)
    s.set_m(_m(n))
    s.profile_enable(True)
    s.step(1e-15, 0.0, "rk4")
    assert ("p2_y_forward" not in s.profile_read()) == one
    s.profile_enable(False)
    s.close()
