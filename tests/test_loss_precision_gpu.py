"""The Eq. 4 loss holds a node's nine squared errors to FP64 accuracy
(gnn_collide_loss_kernel), inside and outside the range in which it carries
them in FP32 words.  All nodes but one (or one per lattice) have their target
met exactly, so that the exact loss is a short sum of rationals and no other
sum rounds."""
from fractions import Fraction

import pytest

from paper_2504_14494_gb300 import inputs

pytestmark = pytest.mark.gpu

ULP = Fraction(1, 2 ** 53)
NX, NY, NB = 37, 11, 2
PER, N = NX * NY, NX * NY * NB


def _setup(L, torch, cuda, scale):
    g = torch.Generator(device=cuda)
    g.manual_seed(1)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, device=cuda).view(9, 1)
    f = (scale * w * (1 + 0.05 * torch.rand(9, N, generator=g, device=cuda))).reshape(-1)
    theta = torch.from_numpy(inputs.xavier_params(3, bias_scale=0.1)).to(cuda)
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=cuda)
    L.gnn_pack(theta, packed)
    return g, f, theta, packed


def _loss(L, torch, f, y, tgt, packed, pred=None):
    s = L.shape(NX, NY, NB)
    ws = torch.empty(L.gnn_loss_workspace_bytes(s), dtype=torch.uint8, device=f.device)
    loss = torch.zeros(1, dtype=torch.float64, device=f.device)
    L.gnn_collide_loss(f, y, tgt, s, 0.7, None, packed, loss, None, pred, ws)
    return loss.item()


def _squares(r):
    return sum(Fraction(x) ** 2 for x in r.cpu().double().tolist())


# populations scaled into the FP32 words' range, and below and above it
@pytest.mark.parametrize("scale,ulps", [(1.0, 3.1), (1e-14, 11.1), (1e16, 11.1)])
@pytest.mark.parametrize("node", [0, 255, 256, N - 1])
def test_loss_of_one_node(lbmlib, cuda, scale, ulps, node):
    """Rounding: the node's value (2.1, or 10 by FP64 products), the division by 9 N (1)."""
    import torch
    L = lbmlib
    g, f, _, packed = _setup(L, torch, cuda, scale)
    y = torch.zeros(10 * N, device=cuda)
    y[:N] = torch.randn(N, generator=g, device=cuda)
    pred = torch.empty_like(f)
    _loss(L, torch, f, y, f, packed, pred)
    for draw in range(24):
        tgt = pred.clone()
        step = scale * 10.0 ** -(draw % 6) * torch.randn(9, generator=g, device=cuda)
        tgt.view(9, N)[:, node] += step
        r = pred.view(9, N)[:, node] - tgt.view(9, N)[:, node]
        want = _squares(r) / (9 * N)
        got = Fraction(_loss(L, torch, f, y, tgt, packed))
        assert abs(got - want) <= Fraction(ulps) * ULP * want, (draw, float((got - want) / want / ULP))


def test_weighted_loss_of_two_nodes(lbmlib, cuda):
    """As above, with a weight per lattice: one rounding more per node, one for the sum."""
    import torch
    L = lbmlib
    g, f, theta, packed = _setup(L, torch, cuda, 1.0)
    s = L.shape(NX, NY, NB)
    pre, y, pred = torch.empty_like(f), torch.empty(10 * N, device=cuda), torch.empty_like(f)
    L.lbm_stream(f, pre, s)
    saved = torch.empty(L.gnn_saved_bytes(s), dtype=torch.uint8, device=cuda)
    L.gnn_forward(pre, s, packed, saved, y)
    _loss(L, torch, pre, y, pre, packed, pred)
    ws = torch.empty(L.gnn_train_workspace_bytes(s), dtype=torch.uint8, device=cuda)
    for draw in range(8):
        lw = 10.0 ** (draw - 4) * (0.5 + torch.rand(NB, generator=g, device=cuda))
        tgt = pred.clone()
        want = Fraction(0)
        for b, node in enumerate((PER - 1, PER + 5)):
            tgt.view(9, N)[:, node] += 1e-3 * torch.randn(9, generator=g, device=cuda)
            r = pred.view(9, N)[:, node] - tgt.view(9, N)[:, node]
            want += Fraction(lw[b].item()) * _squares(r) / (9 * N)
        loss = torch.zeros(1, dtype=torch.float64, device=cuda)
        p, pk = theta.clone(), packed.clone()
        m, v = (torch.zeros(L.gnn_trainable_count(), device=cuda) for _ in range(2))
        L.gnn_train_step_weighted(f, tgt, s, 0.7, None, lw, p, pk, m, v, 1, 1e-3, 0.0, loss, None, ws)
        got = Fraction(loss.item())
        assert abs(got - want) <= Fraction(5.1) * ULP * want, (draw, float((got - want) / want / ULP))
    assert L.lbm_get_status() == 0
