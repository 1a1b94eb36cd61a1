"""Slice-fused forward (one kernel, spectra in shared memory only) at the edges of its instances, against the oracle with
the gates of parity_util."""
import pytest
import torch

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

from parity_util import check

# smallest and largest extents of each padded length, odd and even rows; 2-D and 3-D: both ends of every axis instance
LINES = [64, 65, 127, 128, 129, 256, 257, 511, 512, 1023, 1025, 2047, 2048, 2049, 4095, 4096]
PLANES = [(2, 1), (8, 16), (5, 32), (16, 17), (9, 31), (16, 16), (17, 16), (32, 32), (31, 64), (33, 15), (64, 17), (33, 64), (65, 13),
          (128, 32), (127, 31)]
VOLUMES = [(2, 2, 1), (8, 8, 16), (7, 8, 15), (8, 9, 16), (8, 16, 13), (9, 8, 16), (16, 5, 7), (8, 7, 17), (5, 8, 32)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("causal,shared", [(True, True), (False, False)])
@pytest.mark.parametrize("L", LINES)
def test_lines(L, causal, shared, dtype):
    # 7 batch entries: several per filter transform and a ragged last group where the filter is shared
    w, (q, k, v, h) = W.random_problem((L,), B=7 if shared else 2, C=3, dtype=dtype, causal=causal, h_shared=shared, seed=101)
    check(w, q, k, v, h)


@pytest.mark.parametrize("dtype,shared", [("f32", False), ("bf16", True)])
@pytest.mark.parametrize("dims", PLANES + VOLUMES, ids=str)
def test_grids(dims, dtype, shared):
    w, (q, k, v, h) = W.random_problem(dims, B=3, C=5, dtype=dtype, h_shared=shared, seed=102)
    check(w, q, k, v, h)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("dims", [(128,), (8192,), (16, 32), (32, 64), (64, 128), (128, 32), (16, 16, 32), (32, 16, 32), (16, 16, 64)], ids=str)
def test_periodic_grids(dims, dtype):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=3, dtype=dtype, seed=103, circular=True)
    check(w, q, k, v, h)


def test_many_slices_shared_filter():
    """More units of work than the GPU has room for: every batch entry of every channel is written once."""
    w, (q, k, v, h) = W.random_problem((100,), B=37, C=211, dtype="bf16", causal=True, h_shared=True, seed=104)
    check(w, q, k, v, h)
