"""The FP64 solver's weights of L: held by grids that solve in FP64 only, and
at hand in every call that FP64 has, first calls under capture and without
allocation among them."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402

MIB = 1 << 20


def problem(nx, ny, seed):
    P = synth.problem(nx, ny, seed)
    return [torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS], torch.as_tensor(P["R"], device="cuda")


def grid(nx, ny, co):
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *co)
    return g


def test_grids_that_solve_in_mixed_precision_do_not_hold_them():
    nx, ny = 2048, 1024
    n = nx * ny
    co, R = problem(nx, ny, 11)
    phi = torch.zeros_like(R)
    fp16 = sw.sw_solve_opts_default(prec=sw.SW_PREC_MIXED_FP16, max_iters=2)
    fp64 = sw.sw_solve_opts_default(prec=sw.SW_PREC_FP64, max_iters=2)
    sw.sw_gcr_solve(grid(nx, ny, co), fp16, R, phi)        # the kernels are loaded
    sw.sw_gcr_solve(grid(nx, ny, co), fp64, R, phi)
    torch.cuda.synchronize()
    free = [torch.cuda.mem_get_info()[0]]
    g = grid(nx, ny, co)
    free.append(torch.cuda.mem_get_info()[0])
    sw.sw_gcr_solve(g, fp16, R, phi)
    free.append(torch.cuda.mem_get_info()[0])
    buf = torch.empty(sw.sw_grid_workspace_bytes(g, fp64), dtype=torch.uint8, device="cuda")
    sw.sw_grid_attach_workspace(g, buf)
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
    sw.sw_gcr_solve(g, fp64, R, phi)
    free.append(torch.cuda.mem_get_info()[0])
    # 19 fields of 8 or 4 bytes, six of them twice; allocations come in 2 MiB pieces
    assert free[0] - free[1] <= 168 * n + 8 * MIB
    assert free[1] - free[2] <= sw.sw_grid_workspace_bytes(g, fp16) + 4 * MIB
    assert 96 * n <= free[3] - free[4] <= 96 * n + 4 * MIB


def test_first_fp64_call_recorded_in_a_graph():
    nx, ny = 256, 128
    co, R = problem(nx, ny, 12)
    ref, phi = torch.zeros_like(R), torch.zeros_like(R)
    o = sw.sw_solve_opts_default(prec=sw.SW_PREC_FP64, tol=1e-8)
    sw.sw_gcr_solve(grid(nx, ny, co), o, R, ref)
    g = grid(nx, ny, co)
    buf = torch.empty(sw.sw_grid_workspace_bytes(g, o), dtype=torch.uint8, device="cuda")
    sw.sw_grid_attach_workspace(g, buf)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):                          # global capture mode
        sw.sw_ensemble_solve_async([g], o, [R], [phi])
    graph.replay()
    assert torch.equal(phi, ref)


def test_solves_without_allocation_on_two_grids_in_turn():
    """Both grids' weights are formed in the one fixed array."""
    nx, ny = 256, 128
    pr = [problem(nx, ny, 13 + q) for q in range(2)]
    o = sw.sw_solve_opts_default(prec=sw.SW_PREC_FP64, tol=1e-8)
    ref = []
    for co, R in pr:
        ref.append(torch.zeros_like(R))
        sw.sw_gcr_solve(grid(nx, ny, co), o, R, ref[-1])
    gs = [grid(nx, ny, co) for co, _ in pr]
    for _ in range(2):
        for g, (_, R), want in zip(gs, pr, ref):
            phi = torch.zeros_like(R)
            sw.sw_gcr_solve_noalloc(g, o, R, phi)
            assert torch.equal(phi, want)
    # a grid that has its own, and new coefficients for them
    own = gs[0]
    sw.sw_gcr_solve(own, o, pr[0][1], torch.zeros_like(ref[0]))
    sw.sw_elliptic_set_coeffs(own, *pr[1][0])
    phi = torch.zeros_like(ref[1])
    sw.sw_gcr_solve_noalloc(own, o, pr[1][1], phi)
    assert torch.equal(phi, ref[1])


def test_weights_follow_a_workspace_that_changes():
    """They lie behind the grid's own workspace: one that grows, a lent one in
    its place and back."""
    nx, ny = 256, 128
    co, R = problem(nx, ny, 15)
    o = {k: sw.sw_solve_opts_default(prec=sw.SW_PREC_FP64, tol=1e-8, k=k) for k in (2, 4, 8)}
    ref = {}
    for k in o:
        ref[k] = torch.zeros_like(R)
        sw.sw_gcr_solve(grid(nx, ny, co), o[k], R, ref[k])
    g = grid(nx, ny, co)
    buf = torch.empty(sw.sw_grid_workspace_bytes(g, o[8]), dtype=torch.uint8, device="cuda")
    fp16 = sw.sw_solve_opts_default(prec=sw.SW_PREC_MIXED_FP16, tol=1e-8)
    for k, lent in ((2, None), (4, None), (4, buf), (8, buf), (8, None), (2, None)):
        if lent is not None or k == 8:
            sw.sw_grid_attach_workspace(g, lent)
        phi = torch.zeros_like(R)
        sw.sw_gcr_solve(g, fp16, R, phi)
        phi.zero_()
        sw.sw_gcr_solve(g, o[k], R, phi)
        assert torch.equal(phi, ref[k])
