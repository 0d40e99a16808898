"""The FP32 copies of the face coefficients are the FP64 ones rounded to
nearest even, over the whole range: ties, results below and above FP32's
normal range, zeros of both signs, infinities and NaN.  With C alone set,
L(1) = -C point by point."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


def test_rounding_of_the_fp32_copies():
    nx, ny = 64, 16
    rng = np.random.default_rng(0)
    c = np.ldexp(rng.uniform(1.0, 2.0, nx * ny), rng.integers(-155, 132, nx * ny)) * rng.choice([-1.0, 1.0], nx * ny)
    one = np.float64(np.float32(1.2345))
    ulp = np.spacing(np.float32(1.2345)).astype(np.float64)
    special = [0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028235677973366e38, 3.4028235e38, 3.5e38, 1e300, 2.0 ** -126,
               2.0 ** -126 - 2.0 ** -160, 2.0 ** -149, 2.0 ** -150, 2.0 ** -151, 5e-324]
    special += [one + 0.5 * ulp, one - 0.5 * ulp, one + 1.5 * ulp, np.nextafter(one + 0.5 * ulp, 2.0),
                np.nextafter(one + 0.5 * ulp, 1.0), 2.0 - 2.0 ** -25, 2.0 - 2.0 ** -24, 2.0 - 2.0 ** -26]
    c[:len(special)] = special
    C = torch.as_tensor(c.reshape(ny, nx), device="cuda")
    z = torch.zeros_like(C)
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, z, z, z, z, z, z, C)
    x = torch.ones((ny, nx), dtype=torch.float32, device="cuda")
    y = torch.empty_like(x)
    sw.sw_operator_apply(g, x, y)
    with np.errstate(over="ignore"):
        ref = c.astype(np.float32)
    got = -y.cpu().numpy().reshape(-1)
    # 0 - C x keeps every value but the sign of a zero
    assert np.array_equal(got, ref, equal_nan=True)
