"""Node lookup of the batched kernels by 128-node blocks: lattices that begin
on, before and after a block's first node, blocks with many lattices, and a
block that holds the border of the BGK and GNN groups.  Each lattice equals
its own single-lattice run (each tensor-core row depends only on its own
node) to FP32 rounding, 1e-6 relative."""
import numpy as np
import pytest

from paper_2504_14494_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = {
    "aligned": [(16, 8, 0, 0.8), (128, 1, 0, 0.7), (16, 16, 1, 0.9), (8, 16, 1, 0.6)],
    "one_off": [(127, 1, 0, 0.8), (2, 1, 0, 0.7), (1, 127, 1, 0.9), (129, 1, 1, 0.6), (4, 32, 1, 1.1)],
    "many_per_block": [(1 + i % 3, 1 + i % 2, i % 2, 0.6 + 0.01 * i) for i in range(90)],
    "one_group": [(3, 5, 1, 0.8), (40, 30, 1, 0.7), (7, 1, 1, 0.65)],
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_nodes_find_their_lattice(lbmlib, cuda, case):
    import torch
    L, lattices = lbmlib, CASES[case]
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=cuda)
    L.gnn_pack(torch.from_numpy(inputs.xavier_params(23, s_df=1e-3, bias_scale=0.1)).to(cuda), packed)
    plan = L.lbm_batch_plan_create(lattices)
    try:
        n = L.lbm_batch_nodes(plan)
        off = L.lbm_batch_offsets(plan, len(lattices))
        gen = torch.Generator(device=cuda).manual_seed(5)
        f0 = 0.11 + 0.01 * torch.rand(9, n, device=cuda, generator=gen)
        f1, f2 = torch.empty_like(f0), torch.empty_like(f0)
        ws = torch.empty(max(L.lbm_batch_workspace_bytes(plan), 16), dtype=torch.uint8, device=cuda)
        L.lbm_batch_run(plan, f0.view(-1), f1.view(-1), f2.view(-1), 1, packed, ws)
        assert L.lbm_get_status() == 0
        for i, (nx, ny, col, tau) in enumerate(lattices):
            a = f0[:, off[i]:off[i] + nx * ny].contiguous().view(-1)
            b, s = torch.empty_like(a), L.shape(nx, ny)
            if col == 0:
                L.lbm_step_bgk(a, b, None, s, tau)
            else:
                w = torch.empty(L.gnn_step_workspace_bytes(s), dtype=torch.uint8, device=cuda)
                L.lbm_step_gnn(a, b, s, tau, None, packed, None, w)
            got = f1[:, off[i]:off[i] + nx * ny]
            np.testing.assert_allclose(got.cpu().numpy(), b.view(9, -1).cpu().numpy(), rtol=1e-6, atol=0,
                                       err_msg=str((i, nx, ny, col)))
    finally:
        L.lbm_batch_plan_destroy(plan)
