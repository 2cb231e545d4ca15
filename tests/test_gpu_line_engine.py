"""The line engine's passes (any even 7-smooth length, radix plan at run time)
at the edges of their range, against the oracle's convolution: z lines held in
one thread (up to 16 points), every radix first and last in a plan, y lines of
a 2-D grid up to the longest single pass and just beyond it, a last group of
columns that is nearly empty, lines too long for the engine, and a batch of
grids.  Tolerances are those of the demag tests: FP32 1e-5 of the largest
field, FP64 the oracle's own rounding sensitivity but at least 1e-10."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, rel, to_host

pytestmark = pytest.mark.gpu

D = (2e-9, 3e-9, 2.5e-9)
GRIDS = [(9, 8, 2), (9, 8, 3), (17, 6, 4), (33, 7, 6), (10, 12, 8), (5, 3, 49), (6, 4, 35), (7, 5, 63), (8, 9, 27),
         (3, 245, 1), (20, 257, 1), (5, 512, 1), (6, 525, 1), (2, 3, 1024), (1, 2, 700)]

# FP64 lines whose radix-4 plan would end in a radix 2, enough of them to keep
# whole warps busy: 32, 40, 56, 96, 128, 160, 200, 512, 1536 and 2400 points and the shortest
# (6 and 8, which stay at two passes), and 56 points on both sides of the line
# that parts few lines (radix 2) from many (19456 butterflies of radix 4)
WIDE = [(256, 18, 8), (20, 28, 64), (16, 256, 10), (100, 40, 12), (48, 16, 40), (768, 38, 1), (62, 78, 4), (130, 100, 3),
        (4, 1200, 4), (28, 30, 30), (57, 28, 8), (54, 28, 8)]


@pytest.mark.parametrize("n,precision", [(n, p) for n in GRIDS for p in ("fp64", "fp32")] + [(n, "fp64") for n in WIDE])
def test_lines_match_oracle(n, precision):
    from oracle.demag import demag_fft, magnetization, rounding_sensitivity
    from oracle.newell import demag_tensor
    from paper_2302_08843_gb300.binding import State
    from paper_2302_08843_gb300.workloads import from_soa, to_soa
    rng = np.random.default_rng(sum(n))
    m = rng.normal(size=n + (3,))
    m /= np.linalg.norm(m, axis=-1, keepdims=True)
    s = State(n, D, precision)
    s.set_material(Ms=8e5, A=0.0, alpha=0.1)
    s.demag_setup(20)
    h = from_soa(to_host(s.heff(m=to_soa(m))))
    s.close()
    M = magnetization(m, 8e5)
    tol = FP32_TOL if precision == "fp32" else max(1e-10, rounding_sensitivity(n, D, 20, M))
    assert rel(h, demag_fft(demag_tensor(n, D, 20), M)) < tol


@pytest.mark.parametrize("n", [(11, 9, 1), (6, 7, 8), (5, 30, 3)])
def test_batch_lines_match_single_grids(n):
    """One tiny step of three slots (FP64) against one DP45 step of each alone."""
    from paper_2302_08843_gb300.binding import Batch, State
    from paper_2302_08843_gb300.workloads import to_soa
    rng = np.random.default_rng(5)
    b = Batch(n, D, "fp64", capacity=4)
    states = []
    for slot in (0, 1, 3):
        m = rng.normal(size=n + (3,))
        m /= np.linalg.norm(m, axis=-1, keepdims=True)
        b.set_slot(slot, 7e5 + 1e5 * slot, 1.2e-11, 1.0, to_soa(m), 1e-15)
        s = State(n, D, "fp64")
        s.set_material(Ms=7e5 + 1e5 * slot, A=1.2e-11, alpha=1.0)
        s.demag_setup(20)
        s.set_m(to_soa(m))
        s.step(1e-15, 0.0, "dp45", 1e-5)
        states.append((slot, to_host(s.get_m())))
        s.close()
    b.begin(1, 1e-5, 1e-9, 10)
    st, steps, _ = b.end()
    for slot, m in states:
        assert st[slot] == 1 and steps[slot] == 1
        assert rel(b.get_m(slot), m) < 1e-13
    b.close()


@pytest.mark.parametrize("n", [(25, 25, 1), (24, 9, 2), (32, 16, 3), (50, 7, 1), (18, 1, 5)])
def test_fused_stage_steps_match_fp64(n):
    """FP32 DP45 and RKF45 steps through the fused stage, rows of y paired and the
    last one alone, against the FP64 passes: the step sizes (error norm) to 1e-3,
    the states to 20 times the FP32 field bound."""
    from paper_2302_08843_gb300.binding import State
    from paper_2302_08843_gb300.workloads import to_soa
    rng = np.random.default_rng(3)
    m = rng.normal(size=n + (3,))
    m = to_soa(m / np.linalg.norm(m, axis=-1, keepdims=True))
    for method in ("dp45", "rkf45"):
        out = []
        for precision in ("fp64", "fp32"):
            s = State(n, D, precision)
            s.set_material(Ms=8e5, A=1.3e-11, alpha=0.5, Ku1=1e5, ku_axis=(0.0, 0.6, 0.8))
            s.demag_setup(20)
            s.set_m(m)
            t, dt, dts = 0.0, 2e-14, []
            for _ in range(3):
                t, dt = s.step(dt, t, method, 1e-3)
                dts.append(dt)
            out.append((np.array(dts), to_host(s.get_m())))
            s.close()
        assert np.max(np.abs(out[1][0] / out[0][0] - 1)) < 1e-3
        assert rel(out[1][1], out[0][1]) < 20 * FP32_TOL
