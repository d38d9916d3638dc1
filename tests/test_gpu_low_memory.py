"""The element operator without its scratch: not wanted, no room for it, or given back to an
allocation that the library cannot do without.  Bars as in the parity tests."""
import numpy as np
import pytest

from oracle import operator as op
from workloads import cases, meshgen as mg

from gpu_util import mass_coef, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

TOL = {64: 1e-12, 32: 1e-5}


@pytest.mark.parametrize("N,bits", [(3, 64), (7, 64), (7, 32), (10, 64), (10, 32)])
def test_without_scratch(N, bits):
    import torch
    import paper_2311_09465_gb300 as ts
    dtype = torch.float64 if bits == 64 else torch.float32
    case = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mg.pipe(nc=1, nr=1, nz=3))
    case.resistance = {mg.TAG_OUTLET1: 0.4}
    y = case.y0 + 0.5 * cases.random_state(case.mesh, N, seed=71)
    y[:, :, 0, 1] = 0.0
    v = cases.random_state(case.mesh, N, seed=72, smooth=False)
    prob = op.problem_from_case(case)
    lin = op.linearize(prob, y)
    r_ref, h_ref = op.residual(prob, y), op.jvp(prob, lin, v, "lin_a", mass_coef(case, 0.6))
    g = ts.GLSProblem(case, variant="lin_a", dt_pseudo=0.6)
    for wanted in (True, False, True):
        g.option(element_scratch=wanted)
        assert wanted or ts.ts_scratch_bytes(g.prob) == 0
        assert rel_l2(to_np(g.residual(to_dev(y, dtype))), r_ref) <= TOL[bits]
        assert (ts.ts_scratch_bytes(g.prob) > 0) == wanted
        vd = to_dev(v, dtype)
        hv = torch.empty_like(vd)
        graph = torch.cuda.CUDAGraph()                # a product allocates nothing, its first one either
        with torch.cuda.graph(graph):
            g.jvp(vd, hv)
        graph.replay()
        assert rel_l2(to_np(hv), h_ref) <= TOL[bits]
        assert rel_l2(to_np(g.jvp(vd)), h_ref) <= TOL[bits]
        del graph
    g.close()


def test_a_captured_residual_keeps_its_scratch():
    import torch
    import paper_2311_09465_gb300 as ts
    case = cases.pipe_case(N=3, Re=100.0, Wo=5.0, mesh=mg.pipe(nc=1, nr=1, nz=3))
    y = to_dev(case.y0 + 0.5 * cases.random_state(case.mesh, 3, seed=73), torch.float64)
    g = ts.GLSProblem(case)
    ref = g.residual(y)
    r = torch.empty_like(y)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.residual(y, r)
    held = ts.ts_scratch_bytes(g.prob)
    g.option(element_scratch=False)
    assert held > 0 and ts.ts_scratch_bytes(g.prob) == held
    graph.replay()
    assert torch.equal(r, ref)
    g.close()


def _solve(g, y0, krylov):
    y = y0.clone()
    rep = g.solve(y, precision=64, tol=1e-300, max_steps=1, krylov=krylov, eps_ls=1e-30, max_matvec=3, precond=1,
                  raise_on_noconv=False, reject=0.0)
    assert rep["matvecs"] == 3
    return y


def test_scratch_makes_room_for_the_krylov_basis():
    import torch
    import paper_2311_09465_gb300 as ts
    N = 7
    case = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mg.pipe(nc=10, nr=10, nz=20))
    y0 = to_dev(case.y0 + 0.1 * cases.random_state(case.mesh, N, seed=74), torch.float64)
    field = y0.numel() * 8
    small = ts.GLSProblem(case, dt_pseudo=0.5)        # every kernel loaded, with and without scratch
    ref = _solve(small, y0, 4)
    small.option(element_scratch=False)
    native = _solve(small, y0, 4)
    assert rel_l2(to_np(native - y0), to_np(ref - y0)) <= 1e-6
    small.close()

    g = ts.GLSProblem(case, dt_pseudo=0.5)
    g.residual(y0)
    scratch = ts.ts_scratch_bytes(g.prob)
    slack = 64 << 20
    assert scratch > 20 * field
    krylov = (slack + scratch // 4) // field          # the basis fits only into the slack and the scratch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - slack, dtype=torch.uint8, device="cuda")
    try:
        y = _solve(g, y0, krylov)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert rel_l2(to_np(y - y0), to_np(ref - y0)) <= 1e-6
    g.residual(y0)                                    # there is room again
    assert ts.ts_scratch_bytes(g.prob) == scratch
    g.close()


def test_calls_work_again_after_memory_ran_out():
    import torch
    import paper_2311_09465_gb300 as ts
    case = cases.pipe_case(N=7, Re=100.0, Wo=5.0, mesh=mg.pipe(nc=10, nr=10, nz=20))
    y0 = to_dev(case.y0 + 0.1 * cases.random_state(case.mesh, 7, seed=75), torch.float64)
    g, h = ts.GLSProblem(case, dt_pseudo=0.5), ts.GLSProblem(case, dt_pseudo=0.5)
    ref = _solve(g, y0, 4)                            # kernels loaded; a basis of 5 vectors
    r_ref = g.residual(y0)
    g.option(element_scratch=False)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - (64 << 20), dtype=torch.uint8, device="cuda")
    try:
        for call in (lambda: _solve(g, y0, 60),       # 61 vectors of 4.7 MB
                     lambda: h.residual(y0)):         # tau alone takes 170 MB
            with pytest.raises(ts.TsError) as ei:
                call()
            assert ei.value.code == ts.TS_ERR_OOM
    finally:
        del hog
        torch.cuda.empty_cache()
    g.option(element_scratch=True)
    assert rel_l2(to_np(_solve(g, y0, 4) - y0), to_np(ref - y0)) <= 1e-6
    assert rel_l2(to_np(h.residual(y0)), to_np(r_ref)) <= 1e-12
    g.close()
    h.close()
