"""Host threads with a state each on one GPU: their grids share kernels, each
with another amount of shared memory, and no thread's launch may be refused
because another's asked for less.  The states after the same steps alone are
the reference, bit for bit."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# x lines past the compiled lengths, which one kernel of the fused stage serves
# with 55 to 102 KB of shared memory (three or six parked values per x); FP64 y
# lines of one kernel with 42 and 55 KB
CASES = [("fp32", "rkf45", [(700, 9, 1), (900, 9, 1), (1000, 9, 1)], 2000),
         ("fp64", "rk4", [(16, 192, 1), (16, 256, 1)], 1000)]


def _run(n, precision, method, steps, out, key, gate=None):
    import torch
    from paper_2302_08843_gb300.binding import State
    try:
        m = np.random.default_rng(1).normal(size=(3,) + n[::-1])
        s = State(n, (2e-9, 2e-9, 2e-9), precision, stream=torch.cuda.Stream())
        s.set_material(Ms=8e5, A=1.3e-11, alpha=0.5)
        s.demag_setup(1)
        s.set_m(m / np.linalg.norm(m, axis=0))
        if gate:
            gate.wait()
        for _ in range(steps):
            s.step(1e-16, 0.0, method, 1e-3)
        m = s.get_m()
        s.stream.synchronize()
        out[key] = m.cpu().numpy()
        s.close()
    except Exception as e:      # the thread's: reported by the test
        out[key] = e


@pytest.mark.parametrize("precision,method,grids,steps", CASES)
def test_threads_share_kernels(precision, method, grids, steps):
    alone, out = {}, {}
    for n in grids:
        _run(n, precision, method, steps, alone, n)
    keys = [(n, k) for n in grids for k in range(2)]
    gate = threading.Barrier(len(keys), timeout=120)
    threads = [threading.Thread(target=_run, args=(n, precision, method, steps, out, (n, k), gate)) for n, k in keys]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for n, k in keys:
        assert not isinstance(out[n, k], Exception), (n, out[n, k])
        assert np.array_equal(out[n, k], alone[n]), n
