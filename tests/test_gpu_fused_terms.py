"""Every term of the fused line stage where it can go wrong: material maps with
cells without magnetisation, a damping map, DMI from a map, unequal layers; a
last row of y on its own, x lines of compiled and run-time plans and one with
more than 256 threads.  FP32 fields with energies and torque, and adaptive
steps, against the FP64 passes; and a batch slot whose DMI is switched off."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, rel, to_host

pytestmark = pytest.mark.gpu

D = (2e-9, 3e-9, 2.5e-9)
LAYERS = [1e-9, 0.6e-9, 2.4e-9]


def _set(s, n, kind, rng):
    import torch
    shape = n[::-1]

    def field(lo, hi):
        return torch.as_tensor(rng.uniform(lo, hi, size=shape), device="cuda")

    more = {}
    if kind in ("maps", "layers"):
        ms = field(4e5, 1.2e6)
        if kind == "maps":
            ms[rng.random(shape) < 0.2] = 0.0
        more = dict(Ms_cell=ms, A_cell=field(0.5e-11, 1.5e-11), Ku1_cell=field(0.0, 3e5))
    if kind == "alpha":
        more = dict(alpha_cell=field(0.05, 1.0))
    s.set_material(Ms=0.0 if "Ms_cell" in more else 8e5, A=0.0 if "A_cell" in more else 1.3e-11, alpha=0.5,
                   Ku1=0.0 if "Ku1_cell" in more else 1e5, ku_axis=(0.0, 0.6, 0.8), **more)
    s.set_zeeman(h=(2e4, -1e4, 3e4))
    if kind == "dmi":
        s.set_dmi("interface", 0.0, field(-2e-3, 3e-3))
    if kind == "layers":
        s.set_layers(LAYERS[:n[2]])
    s.demag_setup(5)


@pytest.mark.parametrize("n", [(25, 7, 3), (24, 10, 2), (600, 5, 2)])
@pytest.mark.parametrize("kind", ["maps", "alpha", "dmi", "layers"])
def test_fused_terms_match_fp64(n, kind):
    from paper_2302_08843_gb300.binding import State
    m = np.random.default_rng(3).normal(size=(3,) + n[::-1])
    m /= np.linalg.norm(m, axis=0)
    fields, states = [], []
    for precision in ("fp64", "fp32"):
        s = State(n, D, precision)
        _set(s, n, kind, np.random.default_rng(4))
        h, e, torque = s.heff(m, energies=True, torque=True)
        fields.append((to_host(h), np.array(e), torque))
        for method in ("dp45", "rkf45"):
            s.set_m(m)
            t, dt, dts = 0.0, 5e-15, []
            for _ in range(3):
                t, dt = s.step(dt, t, method, 1e-3)
                dts.append(dt)
            states.append((np.array(dts), to_host(s.get_m())))
        s.close()
    (h64, e64, t64), (h32, e32, t32) = fields
    assert rel(h32, h64) < FP32_TOL
    # an energy sums cells of either sign: against the largest of them
    assert np.max(np.abs(e32 - e64)) < FP32_TOL * np.max(np.abs(e64))
    assert abs(t32 / t64 - 1) < FP32_TOL
    for (dts, m64), (dts32, m32) in zip(states[:2], states[2:]):
        # step sizes from the error norm, states: bounds of the uniform material's test
        assert np.max(np.abs(dts32 / dts - 1)) < 1e-3
        assert rel(m32, m64) < 20 * FP32_TOL


@pytest.mark.parametrize("ms", [8e5, 0.0])
def test_slot_without_its_dmi_again(ms):
    """Switched on and off, a slot's DMI leaves no trace; a slot without
    magnetisation beside it keeps the general variant whatever its terms say."""
    from paper_2302_08843_gb300.binding import Batch
    n = (20, 9, 2)
    m = np.random.default_rng(5).normal(size=(2, 3) + n[::-1])
    m /= np.linalg.norm(m, axis=1, keepdims=True)
    out = []
    for switched in (False, True):
        b = Batch(n, D, "fp32", 2, 2)
        b.set_slot(0, 8e5, 1.2e-11, 1.0, m[0], 1e-14)
        b.set_slot(1, ms, 1.2e-11, 1.0, m[1], 1e-14)
        if switched:
            for slot in (0, 1):
                b.set_slot_terms(slot, "bulk", 2e-3, True)
                b.set_slot_terms(slot, None, 0.0, True)
        b.begin(4, 1e-5, 1e-12, 100)
        status, steps, _ = b.end()
        out.append((status.copy(), steps.copy(), b.get_m(0), b.get_m(1)))
        b.close()
    for a, c in zip(*out):
        assert np.array_equal(a, c)
    assert np.all(np.isfinite(out[0][2])) and np.all(np.isfinite(out[0][3]))
