"""grad_feat written in the features' type: bitwise the FP32 gradient rounded once, on every path that writes it."""
import pytest
import torch

from gpu_util import ensure_lib
from paper_2601_10819_gb300 import inputs, msda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["bf16", "f16"])
# sweeps and dense maps; bands in place (a sweep whose rows exceed a buffer); overlapping maps (corner-slot form issued
# from the device); the corner-slot form forced; rows of no map
@pytest.mark.parametrize("kind", ["plain", "in-place", "overlap", "slots", "gaps"])
@pytest.mark.parametrize("C,G", [(64, 8), (256, 8), (32, 1)])
def test_bits_of_the_rounded_gradient(C, G, kind, dt):
    ensure_lib()
    gen = torch.Generator().manual_seed(C + G)
    maps = [(1, 500), (2, 3)] if kind == "in-place" else [(9, 14), (5, 7), (2, 3)]
    A, P = (400, 13) if kind == "in-place" else (60, 7)
    pr = inputs.make_problem(gen, B=2, cam_maps=[maps] * 2, C=C, G=G, A=A, P=P, loc_range=(-0.1, 1.1), feat_dtype=dt,
                             w_dtype=dt)
    start = pr.scale_start_index.clone()
    if kind == "overlap":
        start[1, 0] = 2
    if kind == "gaps":
        start += 5
        pr.feat = torch.cat([pr.feat, torch.zeros(2, 12, C, dtype=pr.feat.dtype)], 1)
    d = inputs.Problem(pr.feat, pr.spatial_shape, start, pr.sampling_location, pr.weights, pr.grad_out).to("cuda")
    variant = 5 if kind == "slots" else 0
    ref = msda.backward(*d.tensors(), d.grad_out, deterministic=True, variant=variant)
    gf = torch.full(d.feat.shape, float("nan"), dtype=d.feat.dtype, device="cuda")
    got = msda.backward(*d.tensors(), d.grad_out, deterministic=True, variant=variant,
                        grads=(gf, torch.empty_like(ref[1]), torch.empty_like(ref[2])),
                        flags=msda.FLAG_GRAD_FEAT_IN_FEAT_TYPE)
    torch.cuda.synchronize()
    assert torch.equal(gf, ref[0].to(gf.dtype)) and torch.equal(got[1], ref[1]) and torch.equal(got[2], ref[2])


def test_refused_where_it_is_not_built():
    ensure_lib()
    gen = torch.Generator().manual_seed(3)
    d = inputs.make_problem(gen, B=1, cam_maps=[[(6, 5), (3, 2)]], C=32, G=4, A=5, P=3, feat_dtype="bf16").to("cuda")
    gf, gl, gw = (torch.empty(d.feat.shape, dtype=torch.bfloat16, device="cuda"),
                  torch.empty(d.sampling_location.shape, device="cuda"), torch.empty(d.weights.shape, device="cuda"))
    for kw in (dict(deterministic=False), dict(deterministic=True, variant=2)):
        with pytest.raises(msda.MSDAError):
            msda.backward(*d.tensors(), d.grad_out, grads=(gf, gl, gw), flags=msda.FLAG_GRAD_FEAT_IN_FEAT_TYPE, **kw)
