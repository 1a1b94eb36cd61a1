"""Which kernels serve a grid: results agree between the paths, so only this tells when a grid falls back to another one."""
import pytest
import torch

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

ROWS = {"rows_fwd(h)", "rows_fwd(k*v)", "axis_core", "rows_inv"}
PLANES = {"plane_fwd(h)", "plane_fwd(k*v)", "axis_core", "plane_inv"}
# dims, batch, channels, causal, kernels of a forward, points per axis
FORWARD = [((2000,), 2, 3, True, {"slice_fused"}, (4096,)), ((15, 14), 2, 3, False, {"slice_fused"}, (32, 32)),
           ((30, 20), 4, 37, False, {"fused2d"}, (64, 64)), ((30, 20), 4, 38, False, {"slice_fused"}, (64, 64)),
           ((64, 64), 4, 38, False, {"fused2d"}, (128, 128)), ((8, 8, 16), 2, 3, False, {"slice_fused"}, (16, 16, 32)),
           ((96, 96, 96), 1, 2, False, PLANES, (192, 192, 192)), ((20, 128, 120), 1, 2, False, PLANES, (64, 256, 256)),
           ((300, 40), 1, 2, False, ROWS, (768, 128)), ((113, 112), 1, 2, False, ROWS, (256, 256)),
           ((40001,), 1, 2, True, {"ct_cols_fwd(h)", "ct_cols_fwd(k*v)", "ct_hspec", "ct_core", "ct_cols_inv"}, (131072,))]


@pytest.mark.parametrize("case", FORWARD, ids=lambda c: f"{c[0]}-{c[2]}")
def test_forward(case):
    from paper_2607_19378_b200 import hyenand as hn
    dims, B, C, causal, kernels, points = case
    plan = hn.Plan(dims, B, C, causal=causal, dtype=torch.bfloat16)
    infos = [hn.hyenand_plan_kernel_info(plan.handle, i, False) for i in range(hn.hyenand_plan_kernel_count(plan.handle))]
    assert {name for name, launches, _, _ in infos if launches > 0} == kernels
    assert hn.hyenand_plan_fft_dims(plan.handle, len(dims)) == points
    plan.close()


def kernel_names(call):
    from torch.profiler import ProfilerActivity, profile
    call()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return " ".join(e.key for e in prof.key_averages())


@pytest.mark.parametrize("dims,causal,kernels", [((2000,), True, ["slice_bwd_kernel"]), ((64, 64), False, ["slice_bwd_kernel"]),
                                                 ((8, 8, 16), False, ["slice_bwd_kernel"]), ((40, 90), False, ["axis_core3_tma_kernel"]),
                                                 ((20, 40, 50), False, ["axis_core3_tma_kernel"]),
                                                 ((40, 96, 96), False, ["axis_core3_tma_kernel", "hplane_inv_kernel"]),
                                                 ((9000,), True, ["ct_core_w_kernel"])], ids=str)
def test_backward(dims, causal, kernels):
    from paper_2607_19378_b200 import hyenand as hn
    w, arrays = W.random_problem(dims, B=1, C=2, dtype="bf16", causal=causal, seed=161)
    q, k, v, h = (t.cuda() for t in arrays)
    grad = hn.Backward(dims, w.B, w.C, mode=w.mode, dtype=w.torch_dtype)
    names = kernel_names(lambda: grad(q, k, v, h, q))
    assert all(name in names for name in kernels), names
    grad.close()


@pytest.mark.parametrize("dims,kernels,absent", [((15, 14), ["slice_fwd_kernel", "token_scale_kernel"], "widen"),
                                                 ((40, 50), ["fused2d_kernel", "token_scale_kernel"], "widen"),
                                                 ((256, 512), ["token_solo_kernel", "post_solo_kernel"], "slice_fwd")], ids=str)
def test_operator(dims, kernels, absent):
    from paper_2607_19378_b200 import hyenand as hn
    w, arrays = W.random_problem(dims, B=1, C=3, dtype="bf16", seed=162)
    q, k, v, h = (t.cuda() for t in arrays)
    g = torch.ones(w.C, device="cuda")
    mixer = hn.Mixer(dims, w.B, w.C, mode=w.mode, dtype=w.torch_dtype)
    names = kernel_names(lambda: mixer.forward(q, k, v, h, g, g))
    assert all(name in names for name in kernels) and absent not in names, names
    mixer.close()
