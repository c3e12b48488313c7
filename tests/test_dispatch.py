"""Which kernels a call launches (see dispatch.py): the rules on sizes and parameters."""
import pytest

import dispatch as D
from paper_2102_01747_gb300 import workloads as W


@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("max_iter,unroll", [(1, 2), (2, 2), (3, 8), (11, 8)])
def test_julia_steps_per_escape_test_follow_the_cap(max_iter, unroll, p):
    s = dict(W.julia_256(), p=p, max_iter=max_iter)
    assert D.launches(s) == [("plain_kernel", (0, unroll, 0, 0, 0, 0))]
