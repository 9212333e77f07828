"""The message-passing kernels take one, two or four threads per node and one
to four tiles per SM by the number of 128-node tiles: one per SM, two, an odd
number up to 13, and the rest.  Every value of a node is computed the same way
in each, so a stack's results are bitwise those of its lattices stepped alone
(32 tiles).  Stacks of 64 x 64 lattices on either side of each line."""
import pytest

from paper_2504_14494_gb300 import inputs

pytestmark = pytest.mark.gpu

# lattices per stack: 32 tiles each; on 152 SMs 1, 1 / 2, 2 / 3, 3, 4, 5, 13, 14, 17 tiles per SM
STACKS = [2, 4, 5, 9, 10, 14, 16, 22, 61, 64, 80]


@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("nb", STACKS)
def test_stack_equals_its_lattices(lbmlib, cuda, nb, variant):
    import torch
    L = lbmlib
    n, per = 64, 64 * 64
    g = torch.Generator(device=cuda)
    g.manual_seed(nb)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, device=cuda).view(9, 1)
    f = w * (1 + 0.05 * torch.rand(9, nb * per, generator=g, device=cuda))
    dy = torch.randn(10, nb * per, generator=g, device=cuda)
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=cuda)
    L.gnn_pack(torch.from_numpy(inputs.xavier_params(3, bias_scale=0.1, variant=variant)).to(cuda),
               packed)

    def run(f, dy, s):
        f, dy = f.reshape(-1).contiguous(), dy.reshape(-1).contiguous()
        out, df = torch.empty_like(f), torch.empty_like(f)
        ws = torch.empty(L.gnn_step_workspace_bytes(s), dtype=torch.uint8, device=cuda)
        L.lbm_step_gnn(f, out, s, 0.7, None, packed, None, ws)
        saved = torch.empty(L.gnn_saved_bytes(s), dtype=torch.uint8, device=cuda)
        y = torch.empty_like(dy)
        L.gnn_forward(f, s, packed, saved, y)
        grad = torch.empty(L.gnn_trainable_count(), device=cuda)
        wb = torch.empty(L.gnn_backward_workspace_bytes(s), dtype=torch.uint8, device=cuda)
        L.gnn_backward(f, s, packed, saved, dy, grad, df, wb)
        return [out.view(9, -1), y.view(10, -1), df.view(9, -1)]

    stack = run(f, dy, L.shape(n, n, nb))
    for b in {0, nb // 2, nb - 1}:
        part = slice(b * per, (b + 1) * per)
        alone = run(f[:, part], dy[:, part], L.shape(n, n))
        for x, want in zip(stack, alone):
            assert torch.equal(x[:, part], want)
    assert L.lbm_get_status() == 0
