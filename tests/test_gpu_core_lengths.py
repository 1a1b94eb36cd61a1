"""Tensor-copy spectral core at every axis length it takes, at both ends of the extents padded to it and with tile widths
that do not divide the bins of a row, against the oracle with the gates of parity_util."""
import pytest

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

from parity_util import check

# (core axis, ...): padded to 64, 128, 256, 512, 1024; general 2-D, general 3-D and plane-fused grids
LINEAR = [(17, 130), (32, 300), (33, 130), (64, 33), (65, 70), (128, 33), (129, 140), (256, 17), (257, 17), (300, 40),
          (17, 33, 20), (32, 20, 33), (33, 17, 40), (64, 33, 17), (20, 33, 64), (40, 70, 65)]
PERIODIC = [(64, 256), (128, 128), (256, 64), (512, 64), (64, 32, 64), (128, 16, 32), (512, 16, 8)]


@pytest.mark.parametrize("dtype,shared", [("f32", False), ("bf16", True)])
@pytest.mark.parametrize("dims", LINEAR, ids=str)
def test_padded(dims, dtype, shared):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=3, dtype=dtype, h_shared=shared, seed=121)
    check(w, q, k, v, h)


@pytest.mark.parametrize("dtype,shared", [("f32", False), ("bf16", True)])
@pytest.mark.parametrize("dims", PERIODIC, ids=str)
def test_periodic(dims, dtype, shared):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=3, dtype=dtype, h_shared=shared, seed=122, circular=True)
    check(w, q, k, v, h)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("causal,shared", [(True, True), (False, False)])
@pytest.mark.parametrize("L", [4097, 8191, 8194, 20001, 65539, 131071, 262146], ids=str)
def test_long_lines_of_any_length(L, causal, shared, dtype):
    """Long 1-D grids whose slices start on no particular boundary, on the warp-engine kernels."""
    w, (q, k, v, h) = W.random_problem((L,), B=2, C=2, dtype=dtype, causal=causal, h_shared=shared, seed=123)
    check(w, q, k, v, h)
