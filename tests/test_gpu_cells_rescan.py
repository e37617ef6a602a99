"""Cells around the number of points that a warp sorts, in maps whose cells are sorted one by one, and overfull cells of maps
above 9472 cells, which the cell-binned path orders too; FP32 inputs against the FP64 oracle, the FP32 tolerance."""
import pytest
import torch

import oracle
from gpu_util import TOL_FP32, ensure_lib, oracle_backward, relerr
from paper_2601_10819_gb300 import inputs, msda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(33, 29), (64, 176), (100, 100)])  # 1020, 11505 and 10201 cells
@pytest.mark.parametrize("n", [255, 256, 257, 400])
def test_a_cell_of_n_points_among_others(n, H, W):
    """n of 630 points, spread over the anchors, in one cell and the others elsewhere."""
    ensure_lib()
    oracle.build()
    A, P = 90, 7
    gen = torch.Generator().manual_seed(1900 + n)
    pr = inputs.make_problem(gen, B=1, cam_maps=[[(H, W)]], C=32, G=4, A=A, P=P, loc_range=(0.0, 0.4))
    loc = pr.sampling_location.view(-1, 2).clone()
    some = torch.randperm(A * P, generator=gen)[:n]
    x, y = W // 2 + 0.1 + 0.8 * torch.rand(2, n, generator=gen)  # pixels W // 2 and H // 2
    loc[some] = torch.stack([(x + 0.5) / W, (y - W // 2 + H // 2 + 0.5) / H], -1)
    pr = inputs.Problem(pr.feat, pr.spatial_shape, pr.scale_start_index, loc.view_as(pr.sampling_location), pr.weights,
                        pr.grad_out)
    cx, cy = (loc[:, 0] * W - 0.5).floor(), (loc[:, 1] * H - 0.5).floor()
    assert int(((cx == W // 2) & (cy == H // 2)).sum()) == n
    d = pr.to("cuda")
    ws = torch.full((msda.backward_workspace_size(1, H * W, 32, 1, 1, A, P, 4, True),), 0x7f, dtype=torch.uint8,
                    device="cuda")
    g = [t.clone() for t in msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)]
    assert int(ws[:4].view(torch.int32).item()) == 1  # the cell-binned path ran
    h = msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)
    assert all(torch.equal(a, b) for a, b in zip(g, h))
    for a, r in zip(g, oracle_backward(pr)):
        assert relerr(a.cpu().double().numpy(), r) <= TOL_FP32
