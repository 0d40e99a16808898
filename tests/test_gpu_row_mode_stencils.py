"""FP64 row modes form L by the same expressions.  Of a residual that is
rounding noise, L(x) - R with R the oracle's L(x) rounded to nearest, every
row's norm agrees between one warp and one block per row to the rounding of
the norm's own sum: two forms of L would differ by as much as the norm."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


@pytest.mark.parametrize("nx,ny", [(128, 2), (128, 64), (512, 33), (2048, 3)])
def test_row_modes_agree_on_rounding_noise(nx, ny):
    P = synth.problem(nx, ny, 950 + ny)
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *[torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS])
    x = 8000.0 + np.random.default_rng(ny).standard_normal((ny, nx))
    Lx = O.Problem(P).operator(x)
    norms = []
    for mode in (1, 2):
        rows = torch.empty(ny, dtype=torch.float64, device="cuda")
        # a tolerance that any residual meets: the solve stops at the first one
        st = sw.sw_gcr_solve(g, sw.sw_solve_opts_default(tol=1e30, row_residual=rows, row_mode=mode),
                             torch.as_tensor(Lx, device="cuda"), torch.as_tensor(x, device="cuda"))
        assert st.status == sw.SW_OK and st.iterations == 0
        norms.append(rows.cpu().numpy())
    assert np.all(norms[0] > 0.0) and np.max(norms[0]) <= 1e-11 * np.max(np.linalg.norm(Lx, axis=1))
    # a sum of nx squares in another order: nx units of 2^-53 at most
    assert np.max(np.abs(norms[1] / norms[0] - 1.0)) <= nx * 2.0 ** -53
