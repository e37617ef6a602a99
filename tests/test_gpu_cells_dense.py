"""Dense maps of the cell-binned deterministic backward: cells summed by lane groups and by warps, at every lane-group
width, with passes of one cell row and of the whole map, against the FP64 oracle (FP32 inputs, the FP32 tolerance)."""
import pytest
import torch

import oracle
from gpu_util import TOL_FP32, ensure_lib, oracle_backward, relerr
from paper_2601_10819_gb300 import inputs, msda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("maps,A,P,lo,hi", [
    ([(1, 1), (7, 3), (12, 11)], 64, 8, 0.0, 1.0),    # about 128, 16 and 3 records per cell: a warp, its line, the sweep
    ([(9, 100), (40, 4)], 330, 12, -0.05, 1.05),      # the widest rows a pass takes (at C/G = 32); many short ones
    ([(5, 210), (3, 2)], 500, 16, 0.4, 0.6),          # rows too wide for a pass (C/G = 32): the sweep; crowded cells
])
@pytest.mark.parametrize("C,G", [(32, 8), (32, 4), (64, 4), (128, 4), (128, 2), (128, 1)])
def test_dense_maps_against_oracle(C, G, maps, A, P, lo, hi):
    ensure_lib()
    oracle.build()
    gen = torch.Generator().manual_seed(C * 31 + G + A)
    pr = inputs.make_problem(gen, B=2, cam_maps=[maps, maps[::-1]], C=C, G=G, A=A, P=P, loc_range=(lo, hi))
    d = pr.to("cuda")
    need = msda.backward_workspace_size(2, d.feat.shape[1], C, 2, len(maps), A, P, G, True)
    ws = torch.full((need,), 0x7f, dtype=torch.uint8, device="cuda")
    g = [t.clone() for t in msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)]
    if A * C // G * 4 < 200_000:  # one group's grad_out fits a block's shared memory: the cell-binned path ran
        assert int(ws[:4].view(torch.int32).item()) == 1
    h = msda.backward(*d.tensors(), d.grad_out, deterministic=True, workspace=ws)
    assert all(torch.equal(x, y) for x, y in zip(g, h))
    rf = oracle_backward(pr)[0]
    assert relerr(g[0].cpu().double().numpy(), rf) <= TOL_FP32
    assert msda.device_status() == 0
