"""A band of the cell-binned reduce that is read in place, when the waits of the bands around it give up: its barrier phase
completes with a plain arrival, so the buffers' phases stay in step, and the next call matches the oracle."""
import pytest
import torch

import oracle
from gpu_util import TOL_FP32, ensure_lib, oracle_backward, relerr
from paper_2601_10819_gb300 import inputs, msda

pytestmark = pytest.mark.gpu

TIMEOUT = 4


def test_in_place_bands_among_staged_ones_give_up_then_recover():
    """Rows of 500 (too wide for the sums by cells at C/G = 32 and 400 anchors), 1300 points on the map's upper half and 3900
    in one cell of its lower half: that row's records exceed a band buffer, the rows around it come staged."""
    ensure_lib()
    oracle.build()
    gen = torch.Generator().manual_seed(1606)
    pr = inputs.make_problem(gen, B=1, cam_maps=[[(12, 500)]], C=32, G=1, A=400, P=13, loc_range=(0.0, 1.0))
    loc = pr.sampling_location.clone()
    loc[:, 100:] = torch.tensor([0.5012, 0.7]) + (loc[:, 100:] - 0.5) * 1e-5
    pr = inputs.Problem(pr.feat, pr.spatial_shape, pr.scale_start_index, loc, pr.weights, pr.grad_out)
    d = pr.to("cuda")
    call = lambda: msda.backward(*d.tensors(), d.grad_out, deterministic=True)
    msda.device_status()  # clear
    msda.debug_set_wait_limit(0)
    try:
        call()
        assert msda.device_status() == TIMEOUT
    finally:
        msda.debug_set_wait_limit(-1)
    g = call()
    torch.cuda.synchronize()
    assert msda.device_status() == 0
    for x, r in zip(g, oracle_backward(pr)):
        assert relerr(x.cpu().double().numpy(), r) <= TOL_FP32
