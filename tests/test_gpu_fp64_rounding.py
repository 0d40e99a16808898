"""Rounding of L in the FP64 solver: the first residual of a solve against L in
extended precision, from the same FP64 face coefficients."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


def extended_operator(P, x):
    """L(x), the flux form in numpy's longdouble; faces in FP64, as the library's"""
    ny, nx = x.shape
    dl, dp = 2.0 * np.pi / nx, np.pi / ny
    zonal = lambda f, s: ((f + np.roll(f, -1, 1)) * s).astype(np.longdouble)  # noqa: E731

    def merid(f, s):
        g = np.zeros_like(f)
        g[:-1] = (f[:-1] + f[1:]) * s
        return g.astype(np.longdouble)

    ax, cx, bx = zonal(P["A11"], 0.5 / (dl * dl)), zonal(P["A12"], 0.5 / (4.0 * dl * dp)), zonal(P["B1"], 0.5 / (2.0 * dl))
    ay, cy, by = merid(P["A22"], 0.5 / (dp * dp)), merid(P["A21"], 0.5 / (4.0 * dl * dp)), merid(P["B2"], 0.5 / (2.0 * dp))
    x = x.astype(np.longdouble)
    n = np.vstack([x[1:], np.roll(x[-1:], nx // 2, 1)])
    s = np.vstack([np.roll(x[:1], nx // 2, 1), x[:-1]])
    e, w = lambda f: np.roll(f, -1, 1), lambda f: np.roll(f, 1, 1)  # noqa: E731
    fe = cx * (n + e(n) - s - e(s)) + bx * (x + e(x)) + ax * (e(x) - x)
    fn = ay * (n - x) + cy * (e(x) + e(n) - w(x) - w(n)) + by * (x + n)
    fs = np.vstack([np.zeros((1, nx), np.longdouble), fn[:-1]])
    return fe - w(fe) + fn - fs - P["C"] * x


@pytest.mark.parametrize("nx,ny", [(128, 64), (360, 181), (2048, 33)])
def test_first_residual_of_a_smooth_field(nx, ny):
    P = synth.problem(nx, ny, 970 + ny)
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *[torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS])
    lam, phi = np.arange(nx) * 2.0 * np.pi / nx, -0.5 * np.pi + (np.arange(ny) + 0.5) * np.pi / ny
    x = 8000.0 + 400.0 * (np.cos(phi)[:, None] * np.cos(lam)[None] + np.sin(2.0 * phi)[:, None])
    Lx = extended_operator(P, x)
    st = sw.sw_gcr_solve(g, sw.sw_solve_opts_default(tol=1e30), torch.as_tensor(Lx.astype(np.float64), device="cuda"),
                         torch.as_tensor(x, device="cuda"))
    # C x is nearly all of L(x).  Three values of its size are rounded: its
    # coefficient, the last sum and R.  A rounding is at most half of 2^-52 of the
    # value, 2^-52 / sqrt(12) in the root mean square; three of them 2^-53.
    assert st.iterations == 0
    assert st.r0_norm <= 2.0 ** -53 * float(np.linalg.norm(Lx.astype(np.float64)))
