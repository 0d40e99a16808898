"""Coefficients that a replayed CUDA graph sets: an FP64 solve and an FP64
preconditioner outside the graph use the new ones."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


def test_fp64_calls_after_a_replay():
    nx, ny = 128, 64
    P = [synth.problem(nx, ny, 40 + q) for q in range(3)]
    co = [torch.as_tensor(P[0][k], device="cuda") for k in sw.COEFF_KEYS]
    R, phi = torch.as_tensor(P[0]["R"], device="cuda"), torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
    g = sw.sw_grid_create(nx, ny)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sw.sw_elliptic_set_coeffs(g, *co)
    o = sw.sw_solve_opts_default(tol=1e-8)
    q, r = torch.empty_like(R), torch.ones_like(R)
    for p in P:
        for t, k in zip(co, sw.COEFF_KEYS):
            t.copy_(torch.as_tensor(p[k]))
        R.copy_(torch.as_tensor(p["R"]))
        graph.replay()
        phi.zero_()
        st = sw.sw_gcr_solve(g, o, R, phi)
        prob = O.Problem(p)
        res = np.linalg.norm(prob.operator(phi.cpu().numpy()) - p["R"]) / np.linalg.norm(p["R"])
        assert st.status == sw.SW_OK
        assert res <= 1.01e-8                      # the exit test's tolerance, and rounding
        sw.sw_precond_apply(g, o, r, q)
        fresh = sw.sw_grid_create(nx, ny)
        sw.sw_elliptic_set_coeffs(fresh, *co)
        ref = torch.empty_like(q)
        sw.sw_precond_apply(fresh, o, r, ref)
        assert torch.equal(q, ref)
