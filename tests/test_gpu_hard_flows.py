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


@pytest.mark.parametrize("peclet", [1e3, 1e5, 3e5])
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
