"""FP64 totals of a state (lbm_moments, lbm_step_bgk): against exact and FP64
sums, on lattices where a thread takes several nodes, and into a buffer that
held other values (the totals are overwritten)."""
from fractions import Fraction

import pytest

pytestmark = pytest.mark.gpu

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)


def _state(n, dev, seed):
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, device=dev).view(9, 1)
    return (w * (1 + 0.1 * torch.rand(9, n, generator=g, device=dev))).reshape(-1)


def _fp64(f, n):
    import torch
    v = f.view(9, n)
    ok = torch.isfinite(v).all(0)
    v = v.double()[:, ok]
    jx = sum(EX[q] * v[q] for q in range(9) if EX[q])
    jy = sum(EY[q] * v[q] for q in range(9) if EY[q])
    rho = v.sum(0)
    e = 0.5 * (jx * jx + jy * jy) / rho
    return [rho.sum().item(), jx.sum().item(), jy.sum().item(), e.sum().item(),
            float(n - int(ok.sum()))], v.abs().sum().item()


# one node per thread, several (311,296 threads on 152 SMs), and an odd stack
@pytest.mark.parametrize("nx,ny,nb", [(301, 217, 2), (2048, 1031, 1), (1023, 517, 3)])
@pytest.mark.parametrize("steps", [0, 1, 3])
def test_totals_against_fp64(lbmlib, cuda, nx, ny, nb, steps):
    """Mass and momentum: a node's nine additions round at 2^-24 of lo <= 8 2^-24
    of the node (2^-42), the sums over nodes less than that; torch's own FP64 sums
    (a tree) less than 2^-45.  Energy: a few FP32 roundings per node."""
    import torch
    L = lbmlib
    n = nx * ny * nb
    s = L.shape(nx, ny, nb)
    f = _state(n, cuda, seed=nx + steps)
    f.view(9, n)[4, n // 3] = float("inf")
    out, tmp = torch.empty_like(f), torch.empty_like(f)
    t = torch.full((5,), 123.0, dtype=torch.float64, device=cuda)
    L.lbm_step_bgk(f, out, tmp, s, 0.8, None, steps, t)
    u = torch.full((5,), -7.0, dtype=torch.float64, device=cuda)
    L.lbm_moments(out, s, totals=u)
    want, size = _fp64(out, n)
    for got in (t.tolist(), u.tolist()):
        assert got[4] == want[4] > 0
        for k in range(3):
            assert abs(got[k] - want[k]) <= 2 ** -41 * size, (k, got, want)
        assert abs(got[3] - want[3]) <= 8 * 2 ** -24 * want[3]
    assert L.lbm_get_status() == L.LBM_ERR_NONFINITE


@pytest.mark.parametrize("draw", range(6))
def test_sum_over_the_nodes_of_one_thread(lbmlib, cuda, draw):
    """4096^2 nodes, of which those 8 x 152 x 256 apart (54 of them, on 152 SMs
    one thread's) hold a mass of 48 significant bits and all others 2^-100:
    the sum is within 2^-48 (the thread's sum in two FP32 words) and a few FP64
    roundings of the exact one, however the nodes are shared out."""
    import torch
    L = lbmlib
    side, stride = 4096, 8 * 152 * 256
    n = side * side
    g = torch.Generator()
    g.manual_seed(draw)
    r = torch.rand(2, generator=g)
    hi, lo = 0.25 + 0.25 * r[0], (1 + r[1]) * 2.0 ** -27
    f = torch.zeros(9, n, device=cuda)
    f[0] = 2.0 ** -100
    f[0, 1000 * draw::stride], f[1, 1000 * draw::stride] = hi, lo
    count = len(range(1000 * draw, n, stride))
    t = torch.zeros(5, dtype=torch.float64, device=cuda)
    L.lbm_moments(f.view(-1), L.shape(side, side), totals=t)
    want = count * (Fraction(hi.item()) + Fraction(lo.item()))
    err = abs(Fraction(t[0].item()) - want) / want
    assert err <= Fraction(11, 10) / 2 ** 48, float(err * 2 ** 48)


@pytest.mark.parametrize("nx,ny,nb", [(1, 1, 1), (255, 1, 1), (257, 3, 2), (1023, 517, 3)])
def test_fields_with_and_without_totals(lbmlib, cuda, nx, ny, nb):
    """The two instances of the moments kernel give the same fields."""
    import torch
    L = lbmlib
    n = nx * ny * nb
    s = L.shape(nx, ny, nb)
    f = _state(n, cuda, seed=nx)
    got = [torch.full((n,), -7.0, device=cuda) for _ in range(6)]
    L.lbm_moments(f, s, *got[:3])
    L.lbm_moments(f, s, *got[3:], totals=torch.zeros(5, dtype=torch.float64, device=cuda))
    for a, b in zip(got[:3], got[3:]):
        assert torch.equal(a, b)
    rho = f.view(9, n).double().sum(0)
    assert float(((got[0].double() - rho).abs() / rho).max()) <= 8 * 2 ** -24
