"""Grids of more than 2^31 / 3 cells are accepted (mm_state_create refuses 2^31
cells and more), so the distance between a field's components and whatever is
added to it has 64 bits in the kernels that work on cells."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_08843_gb300", "csrc")


# (not among them: batch.cu, as a batch holds fewer than 2^31 / 3 cells, and the
# two fused stages, which refuse larger grids)
@pytest.mark.parametrize("name", ["llg_kernels.cu", "adjoint.cu"])
def test_number_of_cells_is_not_narrowed(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    assert not re.search(r"\bint N =|\(int\)p\.N\b|\bT cb, int N\)", text)


@pytest.mark.parametrize("name", ["demag_passes.cu", "demag_rt.cu"])
def test_fused_stages_refuse_what_they_cannot_index(name):
    with open(os.path.join(CSRC, name)) as f:
        assert "3L * d.nx * d.ny * d.nz" in f.read()


@pytest.mark.gpu
def test_field_past_2_31_values():
    """Exchange and Zeeman field of 734 million cells in the last corner, where
    every component's index passes 2^31, against the same sum in torch."""
    import torch
    from paper_2302_08843_gb300.binding import State
    if torch.cuda.mem_get_info()[0] < 160e9:
        pytest.skip("needs 160 GB of free device memory")
    n, mu0 = (1024, 1024, 700), 4e-7 * 3.14159265358979323846
    g = torch.Generator("cuda").manual_seed(3)
    m = torch.randn((3, n[2], n[1], n[0]), generator=g, device="cuda")
    s = State(n, (1e-9, 1e-9, 1e-9), "fp32")
    s.set_material(Ms=8e5, A=1e-11, alpha=0.1)
    s.set_zeeman(h=(1e4, 2e4, 3e4))
    s.demag_disable()
    h = s.heff(m)[:, -4:, -4:, -4:].double()
    s.close()
    b = m[:, -5:, -5:, -5:].double()
    lap = torch.zeros_like(b)
    for axis in (1, 2, 3):
        k = b.shape[axis]
        lo, hi = [b.narrow(axis, i, k - 1) for i in (0, 1)]
        lap.narrow(axis, 0, k - 1).add_(hi - lo)
        lap.narrow(axis, 1, k - 1).add_(lo - hi)
    want = 2e-11 / (mu0 * 8e5) * 1e18 * lap[:, 1:, 1:, 1:]
    want += torch.tensor([1e4, 2e4, 3e4], dtype=torch.float64, device="cuda")[:, None, None, None]
    # a handful of FP32 roundings of terms of at most 12 |m|
    assert float((h - want).abs().max() / want.abs().max()) < 1e-5
