"""Products of one problem on several streams, live and captured, without ordering among
them: each result is the one that a single stream gives, bit for bit (every sum of the
one-launch element operator has a fixed order)."""
import pytest

from workloads import cases, meshgen as mg

from gpu_util import to_dev

pytestmark = pytest.mark.gpu

REPEATS = 30


@pytest.mark.parametrize("N,bits,variant", [(3, 64, "lin_a"), (7, 64, "frozen"), (7, 64, "lin_a"), (10, 32, "lin_a")])
def test_products_on_several_streams(N, bits, variant):
    import torch
    import paper_2311_09465_gb300 as ts
    dtype = torch.float64 if bits == 64 else torch.float32
    case = cases.pipe_case(N=N, Re=100.0, Wo=5.0, mesh=mg.pipe(nc=4, nr=3, nz=10))
    case.resistance = {mg.TAG_OUTLET1: 0.4}
    y = case.y0 + 0.5 * cases.random_state(case.mesh, N, seed=61)
    g = ts.GLSProblem(case, variant=variant, dt_pseudo=0.6)
    g.residual(to_dev(y, dtype))
    v = [to_dev(cases.random_state(case.mesh, N, seed=62 + k, smooth=False), dtype) for k in range(4)]
    ref = [g.jvp(x, torch.empty_like(x)) for x in v]
    out = [[torch.zeros_like(x) for _ in range(REPEATS)] for x in v]
    captured = [torch.empty_like(x) for x in v[2:]]
    graphs = []
    for x, h in zip(v[2:], captured):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            g.jvp(x, h)
        graphs.append(graph)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in v]
    for k in range(REPEATS):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                if i < 2:
                    g.jvp(v[i], out[i][k])
                else:
                    graphs[i - 2].replay()
                    out[i][k].copy_(captured[i - 2])
    torch.cuda.synchronize()
    for i in range(4):
        assert all(torch.equal(h, ref[i]) for h in out[i]), i
    del graphs
    g.close()
