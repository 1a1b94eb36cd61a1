"""Axes padded to 192, 384 and 768 points, at both ends of each range, as row, middle and core axis, against the oracle with
the gates of parity_util and test_gpu_backward."""
import pytest

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

from parity_util import check
from test_gpu_backward import check_backward

# 2-D grids; general 3-D grids; planes of 192 x 192 points; planes of 128 x 128 points with a core axis of 192
GRIDS = [(65, 96), (96, 65), (96, 97), (129, 70), (70, 192), (192, 129), (33, 257), (384, 18), (17, 384), (257, 66),
         (66, 20, 96), (17, 129, 66), (3, 260, 20), (5, 96, 96), (4, 65, 67), (2, 80, 95), (65, 33, 64)]


@pytest.mark.parametrize("dtype,shared", [("f32", False), ("bf16", True)])
@pytest.mark.parametrize("dims", GRIDS, ids=str)
def test_forward(dims, dtype, shared):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=3, dtype=dtype, h_shared=shared, seed=131)
    check(w, q, k, v, h)


@pytest.mark.parametrize("dtype,shared", [("f32", False), ("bf16", True)])
@pytest.mark.parametrize("dims", GRIDS, ids=str)
def test_gradients(dims, dtype, shared):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=1 if len(dims) == 3 else 3, dtype=dtype, h_shared=shared, seed=132)
    check_backward(w, q, k, v, h, seed=132)
