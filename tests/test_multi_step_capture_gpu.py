"""Multi-step calls plan their launches by the host's launch cost, or by a graph
node's while the stream is captured, and with totals take them in a last single
step or by a pass of their own: whatever the plan, the state is the same bit for
bit, the totals to the order of their FP64 sums."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nb", [(4, 32, 1), (64, 64, 1), (3, 1000, 1), (200, 200, 1), (100, 90, 3),
                                      (512, 512, 1), (1290, 1024, 1)])
@pytest.mark.parametrize("steps", [2, 5, 13])
def test_captured_call_equals_the_eager_one(lbmlib, cuda, nx, ny, nb, steps):
    import torch
    L = lbmlib
    n = nx * ny * nb
    s = L.shape(nx, ny, nb)
    g = torch.Generator(device=cuda)
    g.manual_seed(nx + steps)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, device=cuda).view(9, 1)
    f = (w * (1 + 0.1 * torch.rand(9, n, generator=g, device=cuda))).reshape(-1)
    for call, more in ((L.lbm_step_bgk, ()), (L.lbm_step_channel, (1e-4,))):
        a, b = f.clone(), torch.empty_like(f)
        for _ in range(steps):
            call(a, b, None, s, 0.7, None, *more, nsteps=1)
            a, b = b, a
        want = torch.zeros(5, dtype=torch.float64, device=cuda)
        L.lbm_moments(a, s, totals=want)
        for totals in (False, True):
            eager, captured, tmp = (torch.empty_like(f) for _ in range(3))
            t, u = (torch.full((5,), 9.0, dtype=torch.float64, device=cuda) if totals else None
                    for _ in range(2))
            call(f, eager, tmp, s, 0.7, None, *more, nsteps=steps, totals=t)
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
                call(f, captured, tmp, s, 0.7, None, *more, nsteps=steps, totals=u)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(eager, a) and torch.equal(captured, a), (call.__name__, totals)
            for got in (t, u):
                if totals:  # FP64 sums of n masses in two orders; FP32 energy per node
                    d = (got - want).abs()
                    assert float(d[:3].max()) <= 1e-12 * want[0].item()
                    assert float(d[3]) <= 1e-6 * want[3].item()
    assert L.lbm_get_status() == 0
