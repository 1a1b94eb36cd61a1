"""Long 1-D plans whose shared filters meet groups of slices that are no whole batch entries."""
import pytest
import torch

from parity_util import assert_parity
import oracle
from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu


def make(L, B, C, dtype="bf16", seed=221):
    from paper_2607_19378_b200 import hyenand as hn
    w = W.Workload("groups", (L,), B, C, dtype, causal=True, h_shared=True, seed=seed, filt="causal_exp", alpha=(0.5, 8.0))
    return hn, w, W.make_inputs(w, device="cuda"), hn.Plan(w.dims, B, C, causal=True, dtype=w.torch_dtype)


def core_ms(L, B, C):
    """Device time of the core kernel in one forward (the fastest of three)."""
    hn, w, (q, k, v, h), plan = make(L, B, C)
    kid = [i for i in range(hn.hyenand_plan_kernel_count(plan.handle)) if hn.hyenand_plan_kernel_info(plan.handle, i, True)[0] == "ct_core"][0]
    y = plan.forward(q, k, v, h)
    best = float("inf")
    for _ in range(3):
        hn.hyenand_plan_set_timing(plan.handle, 2)
        plan.forward(q, k, v, h, y)
        torch.cuda.synchronize()
        ms, n = hn.hyenand_plan_kernel_time(plan.handle, kid)
        best = min(best, ms)
    plan.close()
    return best, int(n)


def test_core_works_on_the_slices_of_its_group_alone():
    """1000 channels of 262144 values go through the core in two groups, 765 in one: 1.31 times the rows.  A core that took every
    channel through each group would take about twice that."""
    one, n1 = core_ms(262144, 1, 765)
    two, n2 = core_ms(262144, 1, 1000)
    assert (n1, n2) == (1, 2)
    assert two <= 1.31 * 1.25 * one, (one, two)


# padded 2^20: groups of 383 slices.  Two entries in groups that start inside one; more channels than a group holds (spectra made
# once); one entry of them (each filter has one slice)
@pytest.mark.parametrize("B,C", [(2, 200), (2, 390), (1, 390)])
def test_groups(B, C):
    hn, w, (q, k, v, h), plan = make(524288, B, C)
    y = plan.forward(q, k, v, h)
    torch.cuda.synchronize()
    assert hn.hyenand_plan_device_status(plan.handle) == 0 and hn.hyenand_plan_guard_damage(plan.handle) == 0
    plan.close()
    assert bool(torch.isfinite(y.float()).all())
    for s in sorted({0, 382, 383, B * C - 1}):
        b, c = divmod(s, C)
        one = [t[b:b + 1, c:c + 1].cpu() for t in (q, k, v)]
        ws = W.Workload("one", w.dims, 1, 1, w.dtype, causal=True)
        assert_parity(y[b:b + 1, c:c + 1].cpu(), oracle.conv_fft(*one, h[c].cpu()[None, None], "causal"), one[0], ws, what=f"slice {s}")


@pytest.mark.parametrize("L,B,C", [(65536, 3, 50), (262144, 2, 17)])
def test_host_call_in_groups_has_the_same_bits(L, B, C):
    """hyenand_forward_host works on ranges of slices that start and end inside batch entries."""
    hn, w, (q, k, v, h), plan = make(L, B, C)
    y = plan.forward(q, k, v, h)
    hq, hk, hv, hh = (t.cpu().pin_memory() for t in (q, k, v, h))
    hy = torch.empty_like(hq).pin_memory()
    hn.hyenand_forward_host(plan.handle, hq, hk, hv, hh, 0, hy)
    plan.close()
    assert torch.equal(hy, y.cpu())


@pytest.mark.parametrize("dtype,shared", [("f32", True), ("bf16", False)])
def test_a_driver_that_takes_no_map_of_the_workspace(dtype, shared):
    """Such a plan runs on the kernels without tensor copies; it is not an error."""
    from parity_util import check
    w, arrays = W.random_problem((20000,), B=2, C=2, dtype=dtype, causal=True, h_shared=shared, seed=222)
    check(w, *arrays, env={"HYENAND_REFUSE_MAPS": "1"})
