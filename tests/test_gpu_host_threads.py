"""Host threads with grids of their own and rows of different lengths: the
kernels' shared-memory limits belong to the process, so no thread's call may
lower one that another thread's launch relies on."""
import threading

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


def test_coefficients_of_long_rows_from_two_threads():
    """4096 and 3100 points a row need 64 and 48.4 KB in the face kernel: both
    above the 48 KB that a launch has without a raised limit."""
    errors = []
    start = threading.Barrier(2)

    def work(nx, ny):
        try:
            torch.cuda.set_device(0)
            s = torch.cuda.Stream()
            P = synth.problem(nx, ny, 900 + nx)
            co = [torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS]
            torch.cuda.synchronize()
            g = sw.sw_grid_create(nx, ny)
            start.wait(60)
            for _ in range(4000):
                sw.sw_elliptic_set_coeffs(g, *co, stream=s)
            s.synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append((nx, repr(e)))

    t = [threading.Thread(target=work, args=a) for a in ((4096, 2), (3100, 2))]
    for q in t:
        q.start()
    for q in t:
        q.join(300)
    assert not errors, errors
    assert not any(q.is_alive() for q in t)
