"""Backward of 2-D and 3-D grids from one set of spectra (three spectral products in one core), at both ends of every
core length and path, against the oracle with the gates of test_gpu_backward."""
import pytest

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

from test_gpu_backward import check_backward

# core axis padded to 64, 128, 256, 512, 1024; general 2-D, general 3-D and plane-fused grids
GRIDS = [(17, 70), (32, 129), (33, 70), (65, 30), (128, 65), (129, 140), (257, 20), (400, 17),
         (17, 17, 20), (20, 33, 17), (33, 20, 40), (17, 33, 64), (18, 70, 65), (33, 40, 50), (65, 33, 33)]


@pytest.mark.parametrize("dtype,shared", [("f32", False), ("bf16", False), ("bf16", True)])
@pytest.mark.parametrize("dims", GRIDS, ids=str)
def test_gradients(dims, dtype, shared):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=3, dtype=dtype, h_shared=shared, seed=111)
    check_backward(w, q, k, v, h, seed=111)


@pytest.mark.parametrize("dims", [(64, 256), (128, 128), (256, 64), (512, 64), (64, 32, 64), (128, 16, 32)], ids=str)
def test_gradients_periodic(dims):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=2, dtype="f32", seed=112, circular=True)
    check_backward(w, q, k, v, h, seed=112)


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("dims", [(40, 70), (20, 40, 50), (17, 20, 40)], ids=str)
def test_several_groups_and_passes(dims, shared, monkeypatch):
    """Groups of slices that start at a channel offset, ragged last ones, passes over the batch for a shared filter."""
    monkeypatch.setenv("HYENAND_BACKWARD_RING_SLICES", "4")
    monkeypatch.setenv("HYENAND_BACKWARD_MAX_BATCH", "2")
    w, (q, k, v, h) = W.random_problem(dims, B=5, C=3, dtype="bf16", h_shared=shared, seed=113)
    check_backward(w, q, k, v, h, seed=113)
