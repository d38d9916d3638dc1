"""tau in flows that make its matrix M ill-conditioned: one harmonic without a
mean, and a mean that the harmonic reverses, at large cell Peclet numbers u h / nu.

M is known to n eps |M| in FP64 (n = 2N - 1), so tau's relative error is at most
n eps cond(M) / 2 in any backward-stable form, the oracle's as well; the bar is the
parity tests' own plus the sum of both, on the least-squares part of the residual.
"""
import dataclasses

import numpy as np
import pytest

from oracle import operator as op
from oracle import tracer as tr
from oracle.spectral import conv_matrix, to_complex
from oracle.tau import tau_argument
from workloads import cases, meshgen as mg

from gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52
FLOWS = ("harmonic", "reversing")


def _flow(mesh, N, flow):
    """Axial velocity [V, 3, N, 2] of one phase everywhere, order 1."""
    x = mesh.xyz
    w = 1.0 + 0.3 * np.sin(2.0 * x[:, 0] + x[:, 1]) * np.cos(x[:, 2])
    a = np.zeros((mesh.n_nodes, 3, N, 2))
    a[:, 2, 1, 0], a[:, 2, 1, 1] = 0.45 * w, 0.2 * w
    if flow == "reversing":                          # an eigenvalue of the harmonic's own matrix
        a[:, 2, 0, 0] = 2.0 * np.hypot(0.45, 0.2) * np.cos(np.pi / (2 * N)) * w
    return a


def _cond(prob, kappa, vel):
    u = np.einsum("qa,eaim->eqim", op.QP_BARY, to_complex(vel, prob.N)[prob.tets])
    M = tau_argument(conv_matrix(u), np.broadcast_to(prob.G[:, None], u.shape[:2] + (3, 3)), kappa, prob.C_I)
    lam = np.linalg.eigvalsh(0.5 * (M + np.conj(np.swapaxes(M, -1, -2))))
    return float((lam[..., -1] / lam[..., 0]).max())


def _setup(N, flow, peclet):
    mesh = mg.pipe(nc=1, nr=1, nz=1)
    case = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mesh)
    prob = op.problem_from_case(case)
    nu = float(np.mean(prob.vol) ** (1 / 3)) / peclet
    case.mu, case.omega = case.rho * nu, 1.0
    prob = op.problem_from_case(case)
    vel = _flow(mesh, N, flow)
    return case, prob, nu, vel, _cond(prob, nu, vel)


def _bar(N, cond, r, galerkin, tol=1e-12):
    return tol + (2 * N - 1) * EPS * cond * np.linalg.norm(r - galerkin) / np.linalg.norm(r)


@pytest.mark.parametrize("peclet", [1e3, 3e3, 1e4, 1e5, 3e5])
@pytest.mark.parametrize("flow", FLOWS)
@pytest.mark.parametrize("N", [2, 3, 5, 7, 10, 15])
def test_fp64_residuals_of_ill_conditioned_flows(N, flow, peclet):
    import torch
    import paper_2311_09465_gb300 as ts
    case, prob, nu, vel, cond = _setup(N, flow, peclet)
    y = cases.random_state(case.mesh, N, seed=51)
    y[:, :3] = vel
    y[:, :, 0, 1] = 0.0
    ref = op.residual(prob, y)
    bar = _bar(N, cond, ref, op.residual(dataclasses.replace(prob, C_I=1e30), y))
    assert bar < 1e-4
    g = ts.GLSProblem(case)
    got = to_np(g.residual(to_dev(y, torch.float64)))
    assert np.linalg.norm(got - ref) <= bar * np.linalg.norm(ref)
    g.close()

    phi = cases.random_state(case.mesh, N, seed=52)[:, 3]
    phi[:, 0, 1] = 0.0
    tp = tr.make_tracer_problem(case.mesh.xyz, case.mesh.tets, N, nu, 1.0, case.dirichlet_mask, 3.0)
    ref = tr.tracer_residual(tp, vel, phi)
    bar = _bar(N, cond, ref, tr.tracer_residual(dataclasses.replace(tp, C_I=1e30), vel, phi))
    h = ts.ts_mesh_load(case.mesh.xyz, case.mesh.tets, case.mesh.bfaces, case.mesh.btag)
    t = ts.Tracer(h, case.mesh.n_nodes, N, nu, 1.0, 3.0, dirichlet_tags=case.dirichlet_tags)
    got = to_np(t.residual(to_dev(vel, torch.float64), to_dev(phi, torch.float64)))
    assert np.linalg.norm(got - ref) <= bar * np.linalg.norm(ref)
    t.close()
    ts.ts_mesh_free(h)


def _cosine_rows(tp, a, h, phi):
    """Tracer rows in closed form: velocity a cos(h t) along z, h = N - 1, and phi uniform
    with harmonic h alone.  The sine is in the null space of the convolution and the
    cosine and the mean have its square 2 a^2, so tau is 1 / sqrt(c) and
    1 / sqrt(2 a^2 G_zz + c)."""
    s = tp.omega * h
    c = tp.C_I * tp.kappa ** 2 * np.einsum("eij,eij->e", tp.G, tp.G)
    res = np.array([-s * phi[1], s * phi[0]])
    T = np.stack([res[0] / np.sqrt(2 * a * a * tp.G[:, 2, 2] + c), res[1] / np.sqrt(c)])
    r = np.zeros((tp.xyz.shape[0], tp.N, 2))
    for k in range(4):
        np.add.at(r[:, h, 0], tp.tets[:, k], tp.vol / 4 * (res[0] + s * T[1]))
        np.add.at(r[:, h, 1], tp.tets[:, k], tp.vol / 4 * (res[1] - s * T[0]))
        np.add.at(r[:, 0, 0], tp.tets[:, k], tp.vol * tp.dN[:, k, 2] * 2 * a * T[0])
    return r


@pytest.mark.parametrize("peclet", [1e2, 3e2, 1e4])
@pytest.mark.parametrize("N", [2, 3, 5])
def test_fp64_tau_of_a_cosine_without_a_mean(N, peclet):
    # an eigenvalue alone in its row keeps its relative accuracy: 2^-46 holds the 2^-53 of
    # sums of some 30 terms and tau's 2^-54 over a diagonal entry of at least 2^-8
    import torch
    import paper_2311_09465_gb300 as ts
    mesh = mg.pipe(nc=1, nr=1, nz=1)
    h = N - 1
    size = float(np.mean(op.problem_from_case(cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mesh)).vol) ** (1 / 3))
    tp = tr.make_tracer_problem(mesh.xyz, mesh.tets, N, size / peclet, 1.0, np.zeros(mesh.n_nodes, dtype=bool), 3.0)
    vel = np.zeros((mesh.n_nodes, 3, N, 2))
    vel[:, 2, h, 0] = 0.5
    phi = np.zeros((mesh.n_nodes, N, 2))
    phi[:, h] = 1.0, 1.0
    ref = _cosine_rows(tp, 0.5, h, (1.0, 1.0))
    hm = ts.ts_mesh_load(mesh.xyz, mesh.tets, mesh.bfaces, mesh.btag)
    t = ts.Tracer(hm, mesh.n_nodes, N, tp.kappa, 1.0, 3.0)
    got = to_np(t.residual(to_dev(vel, torch.float64), to_dev(phi, torch.float64)))
    assert np.linalg.norm(got - ref) <= 2.0 ** -46 * np.linalg.norm(ref)
    t.close()
    ts.ts_mesh_free(hm)


@pytest.mark.parametrize("size", [1e-10, 1e-9, 1e9, 1e10])
@pytest.mark.parametrize("N", [3, 7])
def test_fp64_tau_at_small_and_large_lengths(N, size):
    # G:G leaves FP32's range below h = 1e-9 and its low part from h = 1e8 on; the continuity
    # rows (velocity gradients and tau) stay inside it at both ends
    import torch
    import paper_2311_09465_gb300 as ts
    case = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mg.pipe(nc=1, nr=1, nz=1))
    case.mesh.xyz = case.mesh.xyz * size
    case.mu, case.omega = 0.3 * case.rho * size, 1.0 / size
    y = cases.random_state(case.mesh, N, seed=54)
    y[:, :, 0, 1] = 0.0
    ref = op.residual(op.problem_from_case(case), y)[:, 3]
    g = ts.GLSProblem(case)
    got = to_np(g.residual(to_dev(y, torch.float64)))[:, 3]
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    g.close()
