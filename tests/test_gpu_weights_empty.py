"""Connection weights of so many pairs that the lights would be packed first, where there are no
lights (or no eyes): every pair is out of range, which the call refuses, and the next call is
answered."""
import numpy as np
import pytest

from gpu_util import dev
from test_gpu_connect import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, (1 << 20) + 1])
def test_no_lights_or_no_eyes(ctx, n):  # noqa: F811
    import torch
    import paper_1907_12343_gb300 as hrr
    one = torch.ones(1, device=dev())
    pairs = torch.zeros((n, 2), dtype=torch.int32, device=dev())
    sums = torch.zeros(1, device=dev())
    E, L, p = hrr.hrr_eyes(*[one.data_ptr()] * 3, None, None), hrr.hrr_lights(*[one.data_ptr()] * 4), pairs.data_ptr()
    for n_e, n_l, want in ((1, 0, hrr.HRR_ERR_INVALID_ARG), (0, 1, hrr.HRR_ERR_INVALID_ARG), (1, 1, hrr.HRR_OK)):
        st = hrr.hrr_connect(ctx.handle, E, n_e, L, n_l, 0.5, p, n, None, None, None, sums.data_ptr())
        assert st == want, (n_e, n_l, hrr.hrr_last_error(ctx.handle))
    # p = min(1, 0.5 / 1e-4) = 1, so each pair's weight is 1 / 1e-4; partial sums of at most 2^21
    # such values in float32 stay within 2^21 2^-24 of their sum
    assert abs(float(sums[0]) / (n * 1e4) - 1) < 0.125
