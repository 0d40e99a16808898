"""sw_precond_apply is ordered on its stream and does not wait for it: calls with
other options straight behind one another, a second stream, capture in a CUDA
graph, and operands that start at any element."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402

F64, F16, BF16 = sw.SW_PREC_FP64, sw.SW_PREC_MIXED_FP16, sw.SW_PREC_MIXED_BF16


def coeffs(nx, ny, seed):
    P = synth.problem(nx, ny, seed)
    return [torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS], torch.as_tensor(P["R"], device="cuda")


def grid(nx, ny, co):
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *co)
    return g


def dtype(prec):
    return torch.float64 if prec == F64 else torch.float32


def alone(co, o, r):
    """the call on a grid of its own, waited for"""
    ny, nx = r.shape
    q = torch.empty_like(r)
    g = grid(nx, ny, co)
    sw.sw_precond_apply(g, o, r, q)
    torch.cuda.synchronize()
    return q


# (precision, option, stages, eta factor, k): later calls need a larger
# workspace, another eta (new factors) and another descriptor
CALLS = [(F16, 3, 2, 0.0, 1), (F16, 3, 3, 0.5, 1), (F64, 3, 2, 0.5, 4), (BF16, 1, 1, 0.5, 8), (F64, 2, 4, 0.5, 8),
         (F64, 3, 1, 0.25, 8), (F16, 3, 2, 0.25, 2), (F16, 0, 1, 0.25, 2)]


@pytest.mark.parametrize("nx,ny", [(130, 33), (512, 256)])
def test_calls_straight_behind_one_another(nx, ny):
    co, R = coeffs(nx, ny, 61)
    g = grid(nx, ny, co)
    eta0 = sw.sw_grid_get_eta(g)
    todo = []
    for prec, pc, nst, f, k in CALLS:
        o = sw.sw_solve_opts_default(prec=prec, pc=pc, n_richardson=nst, eta=f * eta0, k=k)
        r = R.to(dtype(prec)) * (1.0 + len(todo))
        todo.append((o, r, torch.empty_like(r)))
    ref = [alone(co, o, r) for o, r, _ in todo]
    torch.cuda.synchronize()
    for o, r, q in todo:
        sw.sw_precond_apply(g, o, r, q)
    for (_, _, q), want in zip(todo, ref):
        assert torch.equal(q, want)


@pytest.mark.parametrize("prec", [F64, F16])
def test_second_stream_and_no_wait(prec):
    nx, ny = 256, 128
    co, R = coeffs(nx, ny, 62)
    o = sw.sw_solve_opts_default(prec=prec)
    src = R.to(dtype(prec))
    ref = alone(co, o, src)
    g = grid(nx, ny, co)
    r, q, out = torch.zeros_like(src), torch.zeros_like(src), torch.zeros_like(src)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):                     # the workspace exists, the kernels are loaded
        sw.sw_precond_apply(g, o, r, q)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(100_000_000)             # 50 ms in front of the operands
        r.copy_(src)
        sw.sw_precond_apply(g, o, r, q)
        assert not s.query()                       # returned while the stream is still busy
        out.copy_(q)
        done = torch.cuda.Event()
        done.record()
    torch.cuda.current_stream().wait_event(done)
    # the grid on another stream, ordered behind the first by the event
    q2 = torch.empty_like(src)
    sw.sw_precond_apply(g, o, src, q2)
    assert torch.equal(out, ref) and torch.equal(q2, ref)


@pytest.mark.parametrize("prec,nst", [(F64, 2), (F16, 2), (BF16, 1)])
def test_recorded_in_a_graph(prec, nst):
    nx, ny = 130, 33
    pr = [coeffs(nx, ny, 63 + q) for q in range(2)]
    o = sw.sw_solve_opts_default(prec=prec, n_richardson=nst)
    co = [t.clone() for t in pr[0][0]]
    g = grid(nx, ny, co)
    r = torch.zeros((ny, nx), dtype=dtype(prec), device="cuda")
    q = torch.empty_like(r)
    sw.sw_precond_apply(g, o, r, q)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sw.sw_precond_apply(g, o, r, q)
    for c2, R in pr:                               # a new residual, then new coefficients too
        sw.sw_elliptic_set_coeffs(g, *c2)
        r.copy_(R)
        graph.replay()
        assert torch.equal(q, alone(c2, o, r))


@pytest.mark.parametrize("prec", [F64, F16, BF16])
@pytest.mark.parametrize("nst", [1, 2])
def test_operands_that_start_at_any_element(prec, nst):
    nx, ny = 128, 16
    co, R = coeffs(nx, ny, 65)
    o = sw.sw_solve_opts_default(prec=prec, n_richardson=nst)
    src = R.to(dtype(prec))
    ref = alone(co, o, src)
    g = grid(nx, ny, co)
    rb, qb = (torch.zeros(nx * ny + 2, dtype=src.dtype, device="cuda") for _ in range(2))
    r, q = rb[1:1 + nx * ny].view(ny, nx), qb[1:1 + nx * ny].view(ny, nx)
    r.copy_(src)
    sw.sw_precond_apply(g, o, r, q)
    assert torch.equal(q, ref)
    assert float(qb[0]) == 0.0 and float(qb[-1]) == 0.0
