"""The FP64 operator where its threads take one, two and four rows, with last
groups of one to three rows, against the oracle."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


# a block covers 512 columns; the rows per thread follow from the number of blocks
@pytest.mark.parametrize("nx,ny", [(8, 2), (520, 9), (2048, 113), (2048, 229), (2048, 457), (2048, 458), (2056, 459)])
def test_operator(nx, ny):
    P = synth.problem(nx, ny, 800 + ny)
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *[torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS])
    x = 100.0 + np.random.default_rng(ny).standard_normal((ny, nx))
    y = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
    sw.sw_operator_apply(g, torch.as_tensor(x, device="cuda"), y)
    ref = O.Problem(P).operator(x)
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
