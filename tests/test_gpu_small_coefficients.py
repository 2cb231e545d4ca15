"""FP64 fields of a nearly uniform state: beside the large coefficients of its
spectrum stand the small ones of its ripple, and no pass may carry the rounding
of a large one into a small one.  The reference is the same convolution in
extended precision with the library's own spectrum, so that only the passes'
rounding counts; the yardstick is that of an FP64 library FFT on the host."""
import numpy as np
import pytest

from gpu_util import to_host

pytestmark = pytest.mark.gpu

D = (2e-9, 3e-9, 2.5e-9)


def _convolve(n, T, P, m, real):
    import scipy.fft as sf
    ky, py = np.arange(P[1]), P[1]
    up = 2 * ky > py
    s = np.where(up, -1, 1)[:, None].astype(real)
    xx, xy, _, yy, _, zz = T[:, 0].astype(real)[:, np.where(up, py - ky, ky)]
    M = sf.rfftn(m[:, 0].astype(real) * real(8e5), s=P[1::-1], axes=(1, 2))
    H = np.stack([xx * M[0] + s * xy * M[1], s * xy * M[0] + yy * M[1], zz * M[2]])
    return sf.irfftn(H, s=P[1::-1], axes=(1, 2))[:, :n[1], :n[0]] * real(P[0] * P[1])


# one pass of 2-D lines and two of them; radix-2 and radix-4 plans
@pytest.mark.parametrize("n", [(64, 64, 1), (128, 64, 1), (128, 128, 1), (512, 16, 1)])
def test_small_field_beside_a_large_one(n):
    pytest.importorskip("scipy")
    from paper_2302_08843_gb300.binding import State, demag_spectrum_host, padded_extents
    rng = np.random.default_rng(7)
    m = np.zeros((3, 1, n[1], n[0]))
    m[0] = 1.0
    m[1:] = 1e-3 * rng.normal(size=(2, 1, n[1], n[0]))
    m /= np.linalg.norm(m, axis=0)
    s = State(n, D, "fp64")
    s.set_material(Ms=8e5, A=0.0, alpha=0.1)
    s.demag_setup(2)
    h = to_host(s.heff(m))[:, 0]
    s.close()
    P = padded_extents(n)
    T = demag_spectrum_host(n, D, 2)
    exact = _convolve(n, T, P, m, np.longdouble)
    err = [float(np.linalg.norm((v - exact)[:2])) for v in (h, _convolve(n, T, P, m, np.float64))]
    # radix-8 passes that multiply first, both outputs of a butterfly formed alike,
    # are at 1.08 to 1.15 of the host's; 2 a - x in the butterflies at 1.33 to 1.40
    assert err[0] < 1.2 * err[1]
