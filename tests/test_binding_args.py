"""Arguments that the binding converts by itself (no GPU needed)."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2605_22718_b200 import binding

POSE = [0.5, -1.0, 2.0, 0.0, 1.0, 0.0, 0.25, 0.0]


@pytest.mark.parametrize("pose", [
    POSE,
    tuple(POSE),
    [Fraction(x) for x in POSE],
    np.array(POSE),
    np.array(POSE, dtype=np.float32),
    np.array([Fraction(x) for x in POSE], dtype=object),
    np.array([str(x) for x in POSE]),
    torch.tensor(POSE),
    torch.tensor(POSE).reshape(8, 1),
    torch.tensor(POSE, dtype=torch.bfloat16, requires_grad=True),
])
def test_poses_of_every_kind(pose):
    assert list(binding._pose_arg(pose)) == POSE


@pytest.mark.parametrize("pose", [POSE + [0.0], ["x"] * 8, [None] * 8])
def test_poses_that_are_refused(pose):
    with pytest.raises((IndexError, TypeError, ValueError)):
        binding._pose_arg(pose)


def test_a_stream_that_is_not_given(monkeypatch):
    """None and 0 both stand for the current stream."""
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 7, raising=False)
    assert binding._stream(None) == binding._stream(0) == 7
