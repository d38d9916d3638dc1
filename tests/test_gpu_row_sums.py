"""Node sums of the FP64 element operator where the element rows cancel, as in a converged
state: a pressure that is the same everywhere.

Rows are double-float: geometry, products and the stored row are each rounded to 2^-49 of
the row at most, nine roundings of 2^-49 / sqrt3 rms together at the outside.  The sum adds
nothing to that: rms error below sqrt(9 / 3) 2^-49 of the root of the rows' sum of squares."""
import numpy as np
import pytest

from oracle import operator as op
from workloads import cases, meshgen as mg

from gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 3, 7, 15])
def test_rows_that_cancel(N):
    import torch
    import paper_2311_09465_gb300 as ts
    mesh = mg.pipe(nc=4, nr=3, nz=8)
    case = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mesh)
    prob = op.problem_from_case(case)
    p = np.random.default_rng(3).standard_normal((N, 2))
    p[0, 1] = 0.0
    y = np.zeros((mesh.n_nodes, 4, N, 2))
    y[:, 3] = p
    inner = np.ones(mesh.n_nodes, bool)
    inner[np.asarray(mesh.bfaces).ravel()] = False
    squares = np.zeros((mesh.n_nodes, 3))
    np.add.at(squares, prob.tets, (prob.dN * prob.vol[:, None, None]) ** 2)
    g = ts.GLSProblem(case)
    r = to_np(g.residual(to_dev(y, torch.float64)))
    g.close()
    size = np.sqrt((squares[inner][:, :, None, None] * p ** 2).sum())
    assert np.linalg.norm(r[inner]) <= np.sqrt(3.0) * 2.0 ** -49 * size
