"""R and phi that start on any 8-byte boundary: the kernels with 16-byte loads
of them (one warp per row, the split initial residual) are not taken."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


def problem(nx, ny, seed):
    P = synth.problem(nx, ny, seed)
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *[torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS])
    return g, torch.as_tensor(P["R"], device="cuda")


def shifted(t):
    """the same field, 8 bytes past a 16-byte boundary"""
    b = torch.zeros(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = b[1:].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 8
    return v


def test_automatic_choice_takes_blocks():
    g, R = problem(512, 512, 71)                   # more rows than blocks: one warp per row if it may
    o = sw.sw_solve_opts_default(prec=sw.SW_PREC_MIXED_FP16, tol=1e-8)
    block = sw.sw_solve_opts_default(prec=sw.SW_PREC_MIXED_FP16, tol=1e-8, row_mode=1)
    ref = torch.zeros_like(R)
    want = sw.sw_gcr_solve(g, block, R, ref)
    for Rv, pv in ((shifted(R), torch.zeros_like(R)), (R, shifted(torch.zeros_like(R)))):
        st = sw.sw_gcr_solve(g, o, Rv, pv)
        assert st.status == sw.SW_OK and abs(st.iterations - want.iterations) <= 3
        # each residual is at most 1e-8 of R, so L of the difference at most 2e-8
        # (and the rounding of applying L to it)
        Ld = torch.empty_like(R)
        sw.sw_operator_apply(g, pv - ref, Ld)
        assert float(torch.linalg.norm(Ld)) <= 2.001e-8 * float(torch.linalg.norm(R))


def test_members_of_an_ensemble():
    gs, Rs = zip(*[problem(128, 64, 72 + q) for q in range(12)])
    o = sw.sw_solve_opts_default(prec=sw.SW_PREC_MIXED_FP16, tol=1e-8)
    phis = [torch.zeros_like(R) for R in Rs[:-1]] + [shifted(torch.zeros_like(Rs[-1]))]
    for st in sw.sw_ensemble_solve(gs, o, Rs, phis):
        assert st.status == sw.SW_OK and st.true_rel_residual <= 1e-8


def test_what_needs_the_boundary_refuses():
    g, R = problem(512, 64, 73)
    phi = torch.zeros_like(R)
    sw.sw_split_refresh(g, phi)
    for kw in (dict(row_mode=2), dict(split_r0=1), dict(row_mode=2, prec=sw.SW_PREC_FP64)):
        o = sw.sw_solve_opts_default(**{"prec": sw.SW_PREC_MIXED_FP16, **kw})
        for Rv, pv in ((shifted(R), phi), (R, shifted(phi))):
            for call in (sw.sw_gcr_solve, sw.sw_gcr_solve_noalloc):
                with pytest.raises(sw.SwError) as ei:
                    call(g, o, Rv, pv)
                assert ei.value.status == sw.SW_ERR_INVALID_ARG
    assert float(phi.abs().max()) == 0.0
