"""The gradient buffers that msda.backward allocates, takes and refuses, with the library's call replaced by a recorder
(nothing runs on a GPU: a buffer of the wrong type or size would be overrun there)."""
import pytest
import torch

from paper_2601_10819_gb300 import msda

B, ROWS, C, K, S, A, P, G = 2, 6, 8, 1, 1, 3, 2, 1
SIZES = [(B, ROWS, C), (B, A, P, K, 2), (B, A, P, K, S, G)]


class Recorder:
    def __init__(self):
        self.calls = []

    def msda_backward_workspace_size(self, *args):
        return 0

    def msda_backward(self, *args):
        self.calls.append(args)
        return 0


@pytest.fixture
def lib(monkeypatch):
    r = Recorder()
    monkeypatch.setattr(msda, "load", lambda path=None: r)
    monkeypatch.setattr(msda, "_dims", lambda *t: (B, ROWS, C, K, S, A, P, G))
    monkeypatch.setattr(msda, "_stream", lambda device: 0)
    return r


def call(feat_dtype, flag, grads=None):
    feat = torch.zeros(B, ROWS, C, dtype=feat_dtype)
    none = torch.zeros(1)
    return msda.backward(feat, none, none, none, torch.zeros(1, dtype=feat_dtype), torch.zeros(B, A, C),
                         deterministic=True, grads=grads, flags=msda.FLAG_GRAD_FEAT_IN_FEAT_TYPE if flag else 0)


def buffers(feat_grad_dtype):
    return [torch.empty(s, dtype=feat_grad_dtype if i == 0 else torch.float32) for i, s in enumerate(SIZES)]


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("flag", [False, True])
def test_the_feature_gradient_has_the_type_that_is_written(lib, dt, flag):
    written = dt if flag else torch.float32
    got = call(dt, flag)
    assert [t.dtype for t in got] == [written, torch.float32, torch.float32]
    assert [tuple(t.shape) for t in got] == SIZES
    mine = buffers(written)
    assert all(x is y for x, y in zip(call(dt, flag, mine), mine))
    # a buffer of another shape or with room to spare is filled from its start
    call(dt, flag, [torch.empty(B * ROWS * C + 5, dtype=written), mine[1].view(-1), mine[2]])
    assert len(lib.calls) == 3


@pytest.mark.parametrize("flag,i,bad", [
    (True, 0, torch.empty(SIZES[0])),                                # FP32, but 16 bits are written
    (False, 0, torch.empty(SIZES[0], dtype=torch.bfloat16)),         # 16 bits, but twice as much is written
    (True, 0, torch.empty(SIZES[0], dtype=torch.float16)),           # the other 16-bit type
    (False, 0, torch.empty(B, ROWS, C - 1)),                         # too small
    (True, 0, torch.empty(B, C, ROWS, dtype=torch.bfloat16).transpose(1, 2)),
    (False, 1, torch.empty(SIZES[1], dtype=torch.bfloat16)),
    (False, 1, torch.empty(B, A, P, 2, K).transpose(3, 4)[:, ::2]),
    (True, 2, torch.empty(B, A, P, K, S)[..., :0]),
    (False, 2, torch.empty(SIZES[2], device="meta")),                # on another device
])
def test_a_buffer_that_does_not_match_is_refused_before_the_call(lib, flag, i, bad):
    grads = buffers(torch.bfloat16 if flag else torch.float32)
    grads[i] = bad
    with pytest.raises(ValueError):
        call(torch.bfloat16, flag, grads)
    assert not lib.calls
