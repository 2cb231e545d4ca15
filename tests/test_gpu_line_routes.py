"""Routes of the z and y passes chosen by size, on both sides of their lines:
FP64 plans of unequal radices, whose idle warps leave passes out, along every
axis and with one, two and four columns per CTA; FP32 lines of 1024 and 2048
points with few and with many columns; z passes that let a short y pass be
placed while they run; and FP64 2-D grids past the longest single pass.
Fields against the oracle where it is quick, else FP32 against FP64 fields with
the FP32 bound of the demag tests; RK4 runs against FP64 ones with that bound
for each step, and bit for bit against themselves."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, rel, to_host

pytestmark = pytest.mark.gpu

D = (2e-9, 3e-9, 2.5e-9)


def _m(n, seed=0):
    m = np.random.default_rng(seed).normal(size=(3,) + n[::-1])
    return m / np.linalg.norm(m, axis=0)


def _field(n, precision, m, p):
    from paper_2302_08843_gb300.binding import State
    s = State(n, D, precision)
    s.set_material(Ms=8e5, A=0.0, alpha=0.1)
    s.demag_setup(p)
    h = to_host(s.heff(m=m))
    s.close()
    return h


# 490, 686 and 882 points (two, three and three idle passes) along z, y and x; 50, 70
# and 98 points with few lines and with enough for four columns per CTA
@pytest.mark.parametrize("n", [(4, 3, 245), (3, 5, 343), (5, 4, 441), (4, 245, 2), (9, 343, 1), (245, 6, 2), (441, 3, 2),
                               (60, 40, 25), (70, 30, 35), (9, 5, 25), (62, 28, 49)])
def test_fp64_plans_of_unequal_radices(n):
    from oracle.demag import demag_fft, magnetization, rounding_sensitivity
    from oracle.newell import demag_tensor
    from paper_2302_08843_gb300.workloads import from_soa
    m = _m(n)
    M = magnetization(from_soa(m), 8e5)
    tol = max(1e-10, rounding_sensitivity(n, D, 5, M))
    assert rel(from_soa(_field(n, "fp64", m, 5)), demag_fft(demag_tensor(n, D, 5), M)) < tol


@pytest.mark.parametrize("n", [(33, 40, 512), (33, 50, 512), (15, 16, 1024), (17, 20, 1024)])
def test_fp32_long_z_lines(n):
    m = _m(n)
    assert rel(_field(n, "fp32", m, 1), _field(n, "fp64", m, 1)) < FP32_TOL


@pytest.mark.parametrize("n", [(256, 8, 2), (256, 16, 4), (60, 16, 16), (400, 32, 4), (70, 32, 20), (256, 16, 8)])
def test_short_y_lines_after_the_z_pass(n):
    from paper_2302_08843_gb300.binding import State
    out = []
    steps = 12
    for precision in ("fp64", "fp32", "fp32"):
        s = State(n, D, precision)
        s.set_material(Ms=8e5, A=1.3e-11, alpha=0.5, Ku1=1e5, ku_axis=(0.0, 0.6, 0.8))
        s.demag_setup(2)
        s.set_m(_m(n, 1))
        t = 0.0
        for _ in range(steps):
            t, _ = s.step(2e-14, t, "rk4")
        out.append(to_host(s.get_m()))
        s.close()
    assert rel(out[1], out[0]) < steps * FP32_TOL
    assert np.array_equal(out[1], out[2])


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
