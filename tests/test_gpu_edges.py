"""The CUDA kernels at the edges of their tiles, against the FP64 CPU oracle.

A warp holds 32 // N quadrature points, a block of the element operator 2 or 4
elements (8 of the tracer's), a block of the nodal kernels 4 nodes, a warp of the
assembled product a run of rows: meshes whose counts leave remainders, and every
mode count that is built.  Bars as in the parity tests: relative L2 1e-12 in
FP64 and 1e-5 in FP32 per operator application, 1e-4 for inverted blocks.
"""
import math

import numpy as np
import pytest

from oracle import operator as op
from oracle import solver as sv
from oracle import tracer as tr
from workloads import cases, meshgen as mg

from gpu_util import mass_coef, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

TOL = {64: 1e-12, 32: 1e-5}
# 30, 90 and 1205 tetrahedra: 2, 2 and 1 mod 4, 6, 2 and 5 mod 8; 16, 32 and 34 nodes and an odd count
MESHES = {
    "tiny": lambda: mg.pipe(nc=1, nr=1, nz=1),
    "pipe": lambda: mg.pipe(nc=1, nr=1, nz=3),
    "odd": lambda: mg.junction(h=0.7, seed=3),
}
MODES = [(N, "tiny") for N in (1, 2, 3, 4, 5, 7, 10, 15)] + [(2, "odd"), (3, "odd"), (5, "odd"), (7, "pipe")]


def _case(N, mesh):
    m = MESHES[mesh]()
    if mesh == "odd":
        return cases.junction_case(N=N, Re=300.0, Wo=8.0, mesh=m)
    c = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=m)
    c.resistance = {mg.TAG_OUTLET1: 0.4}
    return c


def _state(case, seed):
    y = case.y0 + 0.8 * cases.random_state(case.mesh, case.N, seed=seed)
    y[case.dirichlet_mask, 0:3] = case.y0[case.dirichlet_mask, 0:3]
    y[:, :, 0, 1] = 0.0
    return y


def _dtype(bits):
    import torch
    return torch.float64 if bits == 64 else torch.float32


@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("N,mesh", MODES)
def test_residual_and_product_with_ragged_counts(N, mesh, bits):
    import paper_2311_09465_gb300 as ts
    case = _case(N, mesh)
    y = _state(case, seed=31)
    v = cases.random_state(case.mesh, N, seed=32, smooth=False)
    prob = op.problem_from_case(case)
    lin = op.linearize(prob, y)
    g = ts.GLSProblem(case, variant="lin_a", dt_pseudo=0.6)
    yd, vd = to_dev(y, _dtype(bits)), to_dev(v, _dtype(bits))
    r = to_np(g.residual(yd))
    hv = to_np(g.jvp(vd))
    assert rel_l2(r, op.residual(prob, y)) <= TOL[bits]
    assert rel_l2(hv, op.jvp(prob, lin, v, "lin_a", mass_coef(case, 0.6))) <= TOL[bits]
    g.close()


@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("N", [3, 5, 7, 10])
def test_a_bad_node_stays_in_its_elements(N, bits):
    # NaN at one node: the rows of its elements' nodes and no others are not finite
    import paper_2311_09465_gb300 as ts
    case = _case(N, "pipe")
    y = _state(case, seed=33)
    node = int(np.flatnonzero(~np.asarray(case.dirichlet_mask))[0])
    y[node, 1, 0, 0] = np.nan
    touched = np.zeros(case.mesh.n_nodes, dtype=bool)
    tets = np.asarray(case.mesh.tets)
    touched[tets[(tets == node).any(axis=1)].ravel()] = True
    case.resistance = {}
    g = ts.GLSProblem(case)
    r = to_np(g.residual(to_dev(y, _dtype(bits))))
    bad = ~np.isfinite(r).reshape(len(touched), -1).all(axis=1)
    np.testing.assert_array_equal(bad, touched)
    g.close()


@pytest.mark.parametrize("N,bits", [(3, 64), (7, 64), (10, 64), (10, 32)])
def test_the_first_product_can_be_captured(N, bits):
    # a product after a residual of its own precision allocates nothing
    import torch
    import paper_2311_09465_gb300 as ts
    case = _case(N, "tiny")
    g = ts.GLSProblem(case, variant="frozen", dt_pseudo=0.6)
    g.residual(to_dev(_state(case, seed=41), _dtype(bits)))
    v = to_dev(cases.random_state(case.mesh, N, seed=42, smooth=False), _dtype(bits))
    hv = torch.empty_like(v)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.jvp(v, hv)
    hv.zero_()
    graph.replay()
    np.testing.assert_array_equal(to_np(hv), to_np(g.jvp(v)))
    g.close()


@pytest.mark.parametrize("bits", [64, 32])
def test_outlet_with_more_nodes_than_threads(bits):
    import paper_2311_09465_gb300 as ts
    mesh = mg.pipe(nc=16, nr=14, nz=1)
    case = cases.pipe_case(N=2, Re=100.0, Wo=5.0, mesh=mesh)
    case.resistance = {mg.TAG_OUTLET1: 0.7}
    assert np.sum(cases.nodes_with_tag(mesh, mg.TAG_OUTLET1)) > 1024
    y = _state(case, seed=34)
    prob = op.problem_from_case(case)
    g = ts.GLSProblem(case)
    r = to_np(g.residual(to_dev(y, _dtype(bits))))
    assert rel_l2(r, op.residual(prob, y)) <= TOL[bits]
    g.close()


@pytest.mark.parametrize("variant", ["frozen", "paper"])
@pytest.mark.parametrize("N,mesh,bits", [(1, "tiny", 32), (2, "tiny", 64), (2, "pipe", 32), (3, "pipe", 32),
                                         (4, "tiny", 64), (5, "tiny", 32), (7, "tiny", 64)])
def test_nodal_blocks_and_inverses(N, mesh, bits, variant):
    import paper_2311_09465_gb300 as ts
    case = _case(N, mesh)
    y = _state(case, seed=35)
    V, nb = case.mesh.n_nodes, 8 * N
    prob = op.problem_from_case(case)
    H = sv.dense_matrix(prob, op.linearize(prob, y), variant, mass_coef(case, 0.9)).reshape(V, nb, V, nb)
    ref = np.stack([H[A, :, A, :] for A in range(V)])
    g = ts.GLSProblem(case, variant=variant, dt_pseudo=0.9)
    g.residual(to_dev(y, _dtype(bits)))
    got = to_np(g.block_diagonal(invert=False))
    assert rel_l2(got, ref) <= 1e-5
    inv = to_np(g.block_diagonal(invert=True)).transpose(0, 2, 1)
    fixed = np.zeros((V, 4, N, 2), dtype=bool)
    fixed[:, :, 0, 1] = True
    fixed[case.dirichlet_mask, 0:3] = True
    fixed = fixed.reshape(V, nb)
    for A in range(V):
        B = got[A].copy()
        B[fixed[A], :] = 0.0
        B[:, fixed[A]] = 0.0
        B[fixed[A], fixed[A]] = 1.0
        assert np.linalg.norm(inv[A] @ B - np.eye(nb)) / math.sqrt(nb) <= 1e-4
    g.close()


@pytest.mark.parametrize("N,mesh", [(1, "tiny"), (2, "pipe"), (3, "odd"), (4, "tiny"), (5, "odd"), (10, "tiny"),
                                    (15, "tiny")])
def test_assembled_product_with_ragged_rows(N, mesh):
    import torch
    import paper_2311_09465_gb300 as ts
    case = _case(N, mesh)
    case.resistance = {}
    y = _state(case, seed=36)
    v = cases.random_state(case.mesh, N, seed=37, smooth=False)
    prob = op.problem_from_case(case)
    ref = op.jvp(prob, op.linearize(prob, y), v, "paper", mass_coef(case, 0.8))
    g = ts.GLSProblem(case, variant="paper", dt_pseudo=0.8)
    g.residual(to_dev(y, torch.float64))
    g.assemble()
    v[case.dirichlet_mask, 0:3] = np.nan         # inputs that the product ignores
    v[:, :, 0, 1] = np.inf
    got = to_np(g.spmv(to_dev(v, torch.float32)))
    assert rel_l2(got, ref) <= 1e-5
    g.close()


@pytest.mark.parametrize("N", [4, 5])
def test_assembled_product_with_several_rows_a_warp(N):
    # more rows than warps of one wave: the ring runs on across row ends
    import torch
    import paper_2311_09465_gb300 as ts
    case = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mg.pipe(nc=6, nr=6, nz=60))
    assert case.mesh.n_nodes > 2 * 152 * 9 * 4
    g = ts.GLSProblem(case, variant="paper", dt_pseudo=0.8)
    g.residual(to_dev(_state(case, seed=38), torch.float64))
    g.assemble()
    v = to_dev(cases.random_state(case.mesh, N, seed=39, smooth=False), torch.float32)
    assert rel_l2(to_np(g.spmv(v)), to_np(g.jvp(v))) <= 1e-5
    g.close()


@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("N,mesh", MODES)
def test_tracer_with_ragged_counts(N, mesh, bits):
    import paper_2311_09465_gb300 as ts
    m = MESHES[mesh]()
    rng = np.random.default_rng(40)
    decay = (1.0 / (1.0 + np.arange(N)) ** 2)[:, None]
    a = 2.0 * rng.standard_normal((m.n_nodes, 3, N, 2)) * decay
    phi = rng.standard_normal((m.n_nodes, N, 2)) * decay
    a[..., 0, 1] = 0.0
    phi[..., 0, 1] = 0.0
    dmask = cases.dirichlet_nodes(m, (mg.TAG_INLET1,))
    tp = tr.make_tracer_problem(m.xyz, m.tets, N, 0.03, 0.8, dmask, 3.0)
    h = ts.ts_mesh_load(m.xyz, m.tets, m.bfaces, m.btag)
    t = ts.Tracer(h, m.n_nodes, N, 0.03, 0.8, 3.0, dirichlet_tags=(mg.TAG_INLET1,))
    got = to_np(t.residual(to_dev(a, _dtype(bits)), to_dev(phi, _dtype(bits))))
    assert rel_l2(got, tr.tracer_residual(tp, a, phi)) <= TOL[bits]
    t.close()
    ts.ts_mesh_free(h)


@pytest.mark.parametrize("krylov", [1, 3, 5, 66])
def test_gram_schmidt_group_remainders(krylov):
    # dot products run four basis vectors at a time and 64 between barriers: with every
    # remainder the solve reaches the root
    import torch
    import paper_2311_09465_gb300 as ts
    case = _case(3, "pipe")
    g = ts.GLSProblem(case, variant="lin_a", dt_pseudo=0.3)
    y = to_dev(case.y0, torch.float64)
    rep = g.solve(y, precision=64, tol=1e-6, max_steps=400, krylov=krylov, eps_ls=0.05, max_matvec=4000, precond=1)
    r = to_np(g.residual(y))
    assert rep["status"] == 0
    assert np.linalg.norm(r) <= 1.0001 * rep["r_final"] * rep["r_ref"]
    assert rel_l2(r, op.residual(op.problem_from_case(case), to_np(y))) <= 1e-5   # small against r itself
    g.close()
