"""Multi-step calls (lbm_step_bgk and lbm_step_channel with nsteps > 1) keep
the state on chip between steps (multi_step.cu): the same collisions in the
same order, so they equal repeated single-step calls bit for bit, at the
edges of what each form takes -- lattices of one row or column, strips and
row ranges with remainders, odd sizes, padded plane strides, buffers off the
vector alignment, stacks with their own relaxation times, and states with
infinities and NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (3, 2, 2), (4, 32, 1), (64, 64, 1), (65, 63, 3), (150, 150, 1), (64, 64, 40),
          (24, 96, 8),                                                 # on chip for all steps
          (56, 700, 1), (57, 701, 2), (112, 441, 1), (3, 9001, 1), (9001, 3, 1), (1023, 67, 2),
          (260, 256, 1), (1290, 1024, 1), (1291, 1023, 1)]            # several steps per pass


def _state(n, ps, dev, seed, off=0, bad=False):
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, device=dev).view(9, 1)
    buf = torch.zeros(9 * ps + off, device=dev)
    f = buf[off:].view(9, ps)
    f[:, :n] = w * (1 + 0.1 * torch.rand(9, n, generator=g, device=dev))
    if bad:
        f[3, n // 3], f[5, n // 2], f[0, n - 1] = float("inf"), float("nan"), 3e38
        f[:, n // 5] = 0.0
    return buf[off:]


def _same(a, b, n, ps):
    import torch
    x, y = a.view(9, ps)[:, :n], b.view(9, ps)[:, :n]
    return bool(torch.equal(x.isnan(), y.isnan())) and bool(
        torch.equal(x.nan_to_num(0.0, 1.0, -1.0), y.nan_to_num(0.0, 1.0, -1.0)))


@pytest.mark.parametrize("nx,ny,nb", SHAPES)
@pytest.mark.parametrize("steps", [2, 3, 4, 9, 14])
def test_equals_single_steps(lbmlib, cuda, nx, ny, nb, steps):
    import torch
    L = lbmlib
    n = nx * ny * nb
    taus = (0.51 + 0.5 * torch.rand(nb, device=cuda)) if nb > 1 else None
    for pad, off, bad in ((0, 0, False), (3, 0, True), (0, 1, False)):
        ps = n + pad
        s = L.shape(nx, ny, nb, ps)
        for call, more in ((L.lbm_step_bgk, ()), (L.lbm_step_channel, (1e-4,))):
            f = _state(n, ps, cuda, seed=nx + steps, off=off, bad=bad)
            out, tmp = torch.empty_like(f), torch.empty_like(f)
            call(f, out, tmp, s, 0.7, taus, *more, nsteps=steps)
            a, b = f.clone(), torch.empty_like(f)
            for _ in range(steps):
                call(a, b, None, s, 0.7, taus, *more, nsteps=1)
                a, b = b, a
            assert _same(out, a, n, ps), (call.__name__, pad, off, bad)
    L.lbm_get_status()


@pytest.mark.parametrize("nx,ny,nb", [(64, 64, 3), (1023, 67, 2)])
def test_totals_of_the_last_state(lbmlib, cuda, nx, ny, nb):
    import torch
    L = lbmlib
    n = nx * ny * nb
    s = L.shape(nx, ny, nb)
    for call, more in ((L.lbm_step_bgk, ()), (L.lbm_step_channel, (1e-4,))):
        f = _state(n, n, cuda, seed=5)
        out, tmp = torch.empty_like(f), torch.empty_like(f)
        t, want = (torch.zeros(5, dtype=torch.float64, device=cuda) for _ in range(2))
        call(f, out, tmp, s, 0.7, None, *more, nsteps=7, totals=t)
        L.lbm_moments(out, s, totals=want)
        # two orders of the same FP64 sums of n positive masses
        scale = want[0].item()
        assert np.abs((t - want).cpu().numpy()).max() <= 1e-12 * scale
    assert L.lbm_get_status() == 0


@pytest.mark.parametrize("nx,ny,nb", [(64, 16, 1), (61, 17, 1), (37, 31, 2), (128, 128, 1), (190, 250, 1),
                                      (3, 3000, 1), (191, 256, 1), (96, 96, 20)])
def test_clusters_of_sixteen_equal_single_steps(lbmlib, cuda, nx, ny, nb):
    import torch
    L = lbmlib
    n = nx * ny * nb
    s = L.shape(nx, ny, nb)
    for steps in (2, 25):
        for call, more in ((L.lbm_step_bgk, ()), (L.lbm_step_channel, (1e-4,))):
            f = _state(n, n, cuda, seed=nx + steps)
            out, tmp = torch.empty_like(f), torch.empty_like(f)
            call(f, out, tmp, s, 0.7, None, *more, nsteps=steps)
            a, b = f.clone(), torch.empty_like(f)
            for _ in range(steps):
                call(a, b, None, s, 0.7, None, *more, nsteps=1)
                a, b = b, a
            assert _same(out, a, n, n), (call.__name__, steps)
    assert L.lbm_get_status() == 0
