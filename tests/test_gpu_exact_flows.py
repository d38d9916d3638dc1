"""The exact tangent's derivative of tau in flows that make M ill-conditioned, after an
FP64 residual: eigenpairs of points that tau_fx takes and of points it leaves to FP64.

Reference: the Daleckii-Krein formula on the oracle's complex M in FP64, through the
least-squares terms of the oracle's operator (they are linear in tau).  The product is
FP32: M and its derivative known to n eps32 |M| (n = 2N - 1) make the derivative of
tau uncertain by n eps32 cond(M), beside the exact test's own 1e-5.
"""
import dataclasses
import math

import numpy as np
import pytest

from oracle import operator as op
from oracle.spectral import conv_matrix, to_complex
from oracle.tau import tau_argument
from workloads import cases

from gpu_util import to_dev, to_np
from test_gpu_hard_flows import FLOWS, _setup

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -24


def _dtau_part(prob, y, v):
    lin = op.linearize(prob, y)
    v = v.copy()
    v[prob.dmask, :3] = 0.0
    uq = np.einsum("qa,eaim->eqim", op.QP_BARY, to_complex(v, prob.N)[prob.tets][:, :, :3])
    G = np.broadcast_to(prob.G[:, None], lin.A.shape[:2] + (3, 3))
    M = tau_argument(lin.A, G, prob.mu / prob.rho, prob.C_I)
    dM = np.einsum("...ij,...imn,...jnk->...mk", G, conv_matrix(uq), lin.A)
    adj = lambda a: np.conj(np.swapaxes(a, -1, -2))                                # noqa: E731
    lam, V = np.linalg.eigh(0.5 * (M + adj(M)))
    s = np.sqrt(lam)
    phi = -1.0 / (s[..., :, None] * s[..., None, :] * (s[..., :, None] + s[..., None, :]))
    dtau = V @ ((adj(V) @ (dM + adj(dM)) @ V) * phi) @ adj(V)
    return (op.apply(prob, dataclasses.replace(lin, tau=dtau), y, "frozen")
            - op.apply(prob, dataclasses.replace(lin, tau=0 * dtau), y, "frozen"))


@pytest.mark.parametrize("peclet", [1e2, 1e3, 3e3])
@pytest.mark.parametrize("flow", FLOWS)
@pytest.mark.parametrize("N", [2, 3, 5, 7])
def test_tau_derivative_after_an_fp64_residual(N, flow, peclet):
    import torch
    import paper_2311_09465_gb300 as ts
    case, prob, _, vel, cond = _setup(N, flow, peclet)
    y = cases.random_state(case.mesh, N, seed=51)
    y[:, :3] = vel
    y[:, :, 0, 1] = 0.0
    v = cases.random_state(case.mesh, N, seed=52)
    v[:, :, 0, 1] = 0.0
    ref = _dtau_part(prob, y, v)
    g = ts.GLSProblem(case, variant="exact", dt_pseudo=math.inf)
    g.residual(to_dev(y, torch.float64))
    got = to_np(g.jvp(to_dev(v, torch.float32)))
    g.set(dt_pseudo=math.inf, variant="lin_a")
    got -= to_np(g.jvp(to_dev(v, torch.float32)))
    assert np.linalg.norm(got - ref) <= (1e-5 + (2 * N - 1) * EPS32 * cond) * np.linalg.norm(ref)
    g.close()
