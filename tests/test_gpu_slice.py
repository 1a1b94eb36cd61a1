"""Slice-fused forward (one kernel, spectra in shared memory only) at the edges of its instances, against the oracle with
the gates of parity_util."""
import pytest
import torch

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

from parity_util import check
from test_gpu_backward import check_backward

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


@pytest.mark.parametrize("dtype,shared", [("f32", True), ("bf16", False), ("bf16", True)])
@pytest.mark.parametrize("dims,causal", [((64,), False), ((65,), True), ((257,), True), ((512,), False), ((1025,), True), ((2048,), False),
                                         ((3000,), True), ((4096,), True), ((2, 1), False), ((8, 16), False), ((16, 17), False),
                                         ((17, 16), False), ((33, 15), False), ((33, 64), False), ((64, 33), False), ((128, 32), False),
                                         ((8, 8, 16), False), ((7, 9, 15), False), ((8, 7, 17), False)], ids=str)
def test_backward(dims, causal, dtype, shared):
    w, (q, k, v, h) = W.random_problem(dims, B=3, C=5, dtype=dtype, causal=causal, h_shared=shared, seed=105)
    check_backward(w, q, k, v, h, seed=105)


@pytest.mark.parametrize("dims", [(128,), (16, 32), (16, 16, 32)], ids=str)
def test_backward_periodic(dims):
    w, (q, k, v, h) = W.random_problem(dims, B=2, C=3, dtype="f32", seed=106, circular=True)
    check_backward(w, q, k, v, h, seed=106)


@pytest.mark.parametrize("C,path", [(37, "fused2d"), (38, "nd_generic")])
def test_many_planes_of_64_points(C, path):
    """Either side of the number of slices from which 64-point planes leave the fused 2-D kernel."""
    from paper_2607_19378_b200 import hyenand as hn
    w, (q, k, v, h) = W.random_problem((30, 20), B=4, C=C, dtype="bf16", seed=107)
    plan = hn.Plan(w.dims, w.B, w.C, dtype=w.torch_dtype)
    assert hn.hyenand_plan_path(plan.handle) == path
    plan.close()
    check(w, q, k, v, h)


@pytest.mark.parametrize("dims,B,C,dtype,causal", [((2000,), 4, 2048, "f32", True), ((31, 64), 3, 6000, "bf16", False)], ids=str)
def test_shared_filter_over_ranges_inside_a_batch_entry(dims, B, C, dtype, causal):
    """hyenand_forward_host works off a large batch in ranges of slices that start and end inside a batch entry: channels
    without a slice in the range sit next to channels with one, in more units than the GPU has room for."""
    from paper_2607_19378_b200 import hyenand as hn
    w = W.Workload("ranges", dims, B, C, dtype, seed=108, causal=causal, h_shared=True)
    q, k, v, h = (t.cpu() for t in W.make_inputs(w, device="cuda"))
    plan = hn.Plan(dims, B, C, causal=causal, dtype=w.torch_dtype)
    try:
        y_dev = plan.forward(*(t.cuda() for t in (q, k, v, h)))
        host = [t.contiguous().pin_memory() for t in (q, k, v, h)]
        y = torch.full_like(q, float("nan")).pin_memory()
        plan.forward_host(*host, y)
    finally:
        plan.close()
    assert torch.equal(y, y_dev.cpu())
