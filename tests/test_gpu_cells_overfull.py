"""Overfull cells: in maps above 9472 cells the binning blocks that meet one clear the plan's flag while other blocks of the
same grid are starting, and the gradient is the corner-slot form's; in smaller maps the cell-binned path orders them."""
import pytest
import torch

import oracle

from gpu_util import TOL_FP32, ensure_lib, oracle_backward, relerr
from paper_2601_10819_gb300 import inputs, msda

pytestmark = pytest.mark.gpu


def test_flag_cleared_while_other_blocks_start():
    """More (batch element, map) blocks than the GPU holds at once (two per SM), every third camera with 320 points in
    one cell of a 100x100 map; the same bits in each of 30 calls, and the corner-slot form's gradient."""
    ensure_lib()
    gen = torch.Generator().manual_seed(1605)
    B, K = 12, 36
    pr = inputs.make_problem(gen, B=B, cam_maps=[[(100, 100)]] * K, C=16, G=2, A=40, P=8, loc_range=(0.0, 1.0))
    loc = pr.sampling_location.clone()
    loc[:, :, :, ::3] = 0.5051 + (torch.rand(loc[:, :, :, ::3].shape, generator=gen) - 0.5) * 2e-5
    d = inputs.Problem(pr.feat, pr.spatial_shape, pr.scale_start_index, loc.contiguous(), pr.weights, pr.grad_out).to("cuda")
    ref = msda.backward(*d.tensors(), d.grad_out, deterministic=True, variant=5)
    first = None
    for _ in range(30):
        g = msda.backward(*d.tensors(), d.grad_out, deterministic=True)
        torch.cuda.synchronize()
        if first is None:
            first = [t.clone() for t in g]
        assert all(torch.equal(x, y) for x, y in zip(g, first))
    assert relerr(first[0].cpu().double().numpy(), ref[0].cpu().double().numpy()) <= TOL_FP32
    assert msda.device_status() == 0


@pytest.mark.parametrize("B,A,maps,spread", [
    (1, 257, [[(25, 25)]], 1e-6),             # every point in one cell, one more than a warp sorts
    (2, 900, [[(24, 31), (95, 96)]], 1e-3),   # the widest map that is read again; cells of 1 to thousands of points
    (1, 64, [[(30, 40)], [(33, 29)]], 5e-3),  # ap not a multiple of 32 with P = 5
])
def test_cells_of_more_points_than_a_warp_sorts(B, A, maps, spread):
    """Crowded cells of maps of up to 9472 cells stay on the cell-binned path; FP32 inputs, the FP32 tolerance, and the
    bits of a second call."""
    ensure_lib()
    oracle.build()
    P = 5 if A == 64 else 1 if A == 257 else 7
    gen = torch.Generator().manual_seed(1700 + A)
    pr = inputs.make_problem(gen, B=B, cam_maps=maps, C=32, G=4, A=A, P=P, loc_range=(0.0, 1.0))
    loc = pr.sampling_location.clone()
    crowd = torch.rand(loc.shape[:-1], generator=gen) < (1.0 if A == 257 else 0.9)
    loc[crowd] = 0.5031 + (loc[crowd] - 0.5) * spread
    pr = inputs.Problem(pr.feat, pr.spatial_shape, pr.scale_start_index, loc.contiguous(), pr.weights, pr.grad_out)
    d = pr.to("cuda")
    Bd, rows, C = d.feat.shape
    K, S = d.spatial_shape.shape[:2]
    ws = torch.full((msda.backward_workspace_size(Bd, rows, C, K, S, A, P, 4, True),), 0x7f, dtype=torch.uint8,
                    device="cuda")
    g = [t.clone() for t in msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)]
    assert int(ws[:4].view(torch.int32).item()) == 1  # the cell-binned path ran
    h = msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)
    assert all(torch.equal(x, y) for x, y in zip(g, h))
    for x, r in zip(g, oracle_backward(pr)):
        assert relerr(x.cpu().double().numpy(), r) <= TOL_FP32
