"""The launch shape that the solver picks, read from a CUDA graph that the call
is recorded in (nothing runs)."""
import ctypes as C

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16120_gb300 as sw  # noqa: E402


class KernelNodeParams(C.Structure):
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p)]


def recorded_kernels(s, call):
    """(dynamic shared memory, blocks, threads) of every kernel that call records on stream s"""
    rt = C.CDLL("libcudart.so.13")
    graph, n, p = C.c_void_p(), C.c_size_t(), KernelNodeParams()
    st = C.c_void_p(s.cuda_stream)
    assert rt.cudaStreamBeginCapture(st, 2) == 0       # relaxed
    try:
        call()
    finally:
        assert rt.cudaStreamEndCapture(st, C.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, C.byref(n)) == 0
    found = []
    for q in nodes:
        kind = C.c_int()
        assert rt.cudaGraphNodeGetType(C.c_void_p(q), C.byref(kind)) == 0
        if kind.value == 0 and rt.cudaGraphKernelNodeGetParams(C.c_void_p(q), C.byref(p)) == 0:
            found.append((p.smem, p.grid[0], p.block[0]))
    assert rt.cudaGraphDestroy(graph) == 0
    return found


def solver_launch(nx, ny, **opts):
    """(blocks, threads, dynamic shared memory) of the solver kernel for a grid:
    of the recorded kernels the one with most shared memory"""
    P = synth.problem(nx, ny, 7)
    g = sw.sw_grid_create(nx, ny)
    sw.sw_elliptic_set_coeffs(g, *[torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS])
    R = torch.as_tensor(P["R"], device="cuda")
    phi = torch.zeros_like(R)
    o = sw.sw_solve_opts_default(max_iters=1, **opts)
    sw.sw_gcr_solve(g, o, R, phi)                      # the workspace exists from here on
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    smem, blocks, threads = max(recorded_kernels(s, lambda: sw.sw_ensemble_solve_async([g], o, [R], [phi], stream=s)))
    return blocks, threads, smem


# rows of 2600 to 3400 points: two blocks fit an SM unless the launch counts the
# scan products, which blocks of several rows do not keep; fewer rows than a
# second block per SM pays for (three rounds of rows against two) stay with one
@pytest.mark.parametrize("nx,ny,per_sm", [(2048, 1024, 2), (2600, 1300, 2), (3400, 800, 2), (2600, 400, 1),
                                          (3400, 400, 1)])
def test_fp64_blocks_per_sm_of_several_rows_each(nx, ny, per_sm):
    blocks, threads, _ = solver_launch(nx, ny, prec=sw.SW_PREC_FP64)
    assert threads == 256
    assert blocks == per_sm * torch.cuda.get_device_properties(0).multi_processor_count


def test_scan_products_are_kept_where_they_are_used():
    """One row per block, with two blocks an SM at most and with four: 14 doubles
    a thread for the zonal solve of option 3, none for option 1."""
    for ny in (64, 512):
        blocks, threads, smem3 = solver_launch(1024, ny, prec=sw.SW_PREC_FP64)
        assert blocks == ny
        assert smem3 - solver_launch(1024, ny, prec=sw.SW_PREC_FP64, pc=sw.SW_PC_DIAG)[2] == 14 * 8 * threads


def ensemble_launch(sizes):
    """(blocks, threads) of an ensemble's solver kernel, recorded"""
    gs, Rs, phis = [], [], []
    for q, (nx, ny) in enumerate(sizes):
        P = synth.problem(nx, ny, 7)
        g = sw.sw_grid_create(nx, ny)
        sw.sw_elliptic_set_coeffs(g, *[torch.as_tensor(P[k], device="cuda") for k in sw.COEFF_KEYS])
        gs.append(g)
        Rs.append(torch.as_tensor(P["R"], device="cuda"))
        phis.append(torch.zeros_like(Rs[-1]))
    o = sw.sw_solve_opts_default(prec=sw.SW_PREC_MIXED_FP16, max_iters=1)
    sw.sw_ensemble_solve_async(gs, o, Rs, phis)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    smem, blocks, threads = max(recorded_kernels(s, lambda: sw.sw_ensemble_solve_async(gs, o, Rs, phis, stream=s)))
    return blocks, threads


# 304 blocks at the full register budget, 608 at half of it
@pytest.mark.parametrize("counts,half", [((8, 40), False), ((0, 40), False), ((32, 32), True), ((0, 200), True)])
def test_ensembles_take_half_the_registers_where_rounds_pay(counts, half):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks, threads = ensemble_launch([(128, 64)] * counts[0] + [(256, 128)] * counts[1])
    assert threads == 128
    assert (blocks > 2 * sms) == half and blocks <= 4 * sms


# about four points a thread above 512
# points where the rows have a block each with that, else four warps; three
# where only those give every row a block
@pytest.mark.parametrize("nx,ny,prec,threads", [(512, 256, 1, 128), (520, 64, 1, 160), (640, 320, 1, 160), (640, 500, 1, 128),
                                                (640, 640, 1, 160), (768, 120, 0, 192), (768, 384, 1, 128),
                                                (1000, 64, 0, 256), (1024, 512, 0, 128), (360, 640, 1, 96),
                                                (1440, 400, 1, 256)])
def test_threads_of_a_row(nx, ny, prec, threads):
    assert solver_launch(nx, ny, prec=prec)[1] == threads
