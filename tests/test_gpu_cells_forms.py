"""The forms in which the cell-binned reduce sums a map, each at every lane-group width, against the FP64 oracle (FP32
inputs, the FP32 tolerance): by columns (a lane group or a warp each) and by cells (a lane group or a warp each)."""
import pytest
import torch

import oracle
from gpu_util import TOL_FP32, ensure_lib, oracle_backward, relerr
from paper_2601_10819_gb300 import inputs, msda

pytestmark = pytest.mark.gpu

# about 0.9, 8, 16, 124, 325 and 868 records per row under 5200 points: columns, cells and a warp per cell in turn, from
# another map on for each width; with half of the points in one cell a warp takes a column, of several bands or one
MAPS = [(60, 97), (25, 26), (16, 20), (6, 7), (4, 4), (3, 2)]


@pytest.mark.parametrize("crowded", [False, True])
@pytest.mark.parametrize("C,G", [(32, 8), (32, 4), (64, 4), (128, 4), (64, 1), (128, 1)])  # 1, 2, 4, 8, 16, 32 lanes
def test_forms_against_oracle(C, G, crowded):
    ensure_lib()
    oracle.build()
    A, P = (200, 26) if C // G == 128 else (650, 8)  # one group's grad_out fits a block's shared memory
    gen = torch.Generator().manual_seed(1800 + C + G)
    pr = inputs.make_problem(gen, B=2, cam_maps=[MAPS], C=C, G=G, A=A, P=P, loc_range=(0.0, 1.0))
    if crowded:
        loc = pr.sampling_location.clone()
        some = torch.rand(loc.shape[:-1], generator=gen) < 0.5
        loc[some] = 0.5131 + (loc[some] - 0.5) * 1e-4
        pr = inputs.Problem(pr.feat, pr.spatial_shape, pr.scale_start_index, loc, pr.weights, pr.grad_out)
    d = pr.to("cuda")
    need = msda.backward_workspace_size(2, d.feat.shape[1], C, 1, len(MAPS), A, P, G, True)
    ws = torch.full((need,), 0x7f, dtype=torch.uint8, device="cuda")
    g = [t.clone() for t in msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)]
    assert int(ws[:4].view(torch.int32).item()) == 1  # the cell-binned path ran
    h = msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)
    assert all(torch.equal(x, y) for x, y in zip(g, h))
    for x, r in zip(g, oracle_backward(pr)):
        assert relerr(x.cpu().double().numpy(), r) <= TOL_FP32
    assert msda.device_status() == 0
