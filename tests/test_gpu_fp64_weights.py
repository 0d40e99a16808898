"""The FP64 solver's nine-point weights of L against the oracle's flux form, at
the sizes where they can go wrong: the smallest grids (neighbours that
coincide), rows that are no multiple of a warp or of a block's threads, one
row either side of a power of two."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


@pytest.mark.parametrize("nx,ny", [(4, 2), (6, 3), (34, 9), (126, 5), (130, 64), (514, 17), (1026, 7), (4096, 3)])
def test_true_residual_of_a_smooth_field(nx, ny):
    P = synth.problem(nx, ny, 700 + nx)
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *[torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS])
    x = 8000.0 + np.random.default_rng(nx).standard_normal((ny, nx))
    rows = torch.empty(ny, dtype=torch.float64, device="cuda")
    phi = torch.as_tensor(x, device="cuda")
    # a tolerance that any residual meets: the solve stops at the first one
    st = sw.sw_gcr_solve(g, sw.sw_solve_opts_default(tol=1e30, row_residual=rows),
                         torch.as_tensor(P["R"], device="cuda"), phi)
    ref = np.linalg.norm(O.Problem(P).operator(x) - P["R"], axis=1)
    assert st.status == sw.SW_OK and st.iterations == 0
    # both forms round 30 terms of the same size: 1e-12 is 4500 units of 2^-52
    assert np.max(np.abs(rows.cpu().numpy() - ref) / ref) <= 1e-12
    assert abs(st.r0_norm / np.linalg.norm(ref) - 1) <= 1e-12
