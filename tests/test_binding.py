"""What the binding takes as a device pointer: a tensor, an int, None; nothing that int()
happens to accept."""

import numpy as np
import pytest
import torch


@pytest.fixture(scope="module")
def C():
    from paper_2608_13578_gb300 import build
    build.build()
    from paper_2608_13578_gb300 import bcmt
    return bcmt


def test_pointers(C):
    t = torch.zeros(4)
    assert C._ptr(t) == t.data_ptr() and C._ptr(1 << 20) == 1 << 20 and C._ptr(None) is None


@pytest.mark.parametrize("bad", [3.0, "4096", b"4096", np.float32(16.0), np.int64(16), [16]])
def test_other_values_are_refused(C, bad):
    with pytest.raises(AttributeError):
        C._ptr(bad)
    p = C.make_params(2, 64, 256, 4, 16, "bf16")
    with pytest.raises(AttributeError):
        C.bcmt_forward(p, bad, *([1 << 20] * 11), 0)
