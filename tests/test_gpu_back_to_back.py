"""Calls that read the previous call's result, enqueued without a pause: the same bits as with the device idle between them
(kernels start while their predecessors drain and must not read or write early)."""
import pytest

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

GRIDS = [(8, 8), (32, 32), (17, 40), (40, 90), (200,), (9, 20, 12), (5, 40, 70), (3, 90, 70), (6000,)]


def chain(step, x, calls, pause):
    import torch
    out = []
    for _ in range(calls):
        x = step(x)
        out.append(x)
        if pause:
            torch.cuda.synchronize()
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("B,C", [(1, 1), (2, 3), (4, 48)])
@pytest.mark.parametrize("dims", GRIDS, ids=str)
def test_plan(dims, B, C):
    import torch
    from paper_2607_19378_b200 import hyenand as hn
    w, arrays = W.random_problem(dims, B=B, C=C, dtype="f32", seed=141)
    q, k, v, h = (torch.as_tensor(a).cuda().contiguous() for a in arrays)
    h /= h.abs().sum(dim=tuple(range(2, h.dim())), keepdim=True)      # no gain of the convolution above 1
    plan = hn.Plan(dims, B, C, dtype=torch.float32)
    grad = hn.Backward(dims, B, C, dtype=torch.float32)

    def step(x):
        return grad(q, x, v, h, plan.forward(q, x, v, h))[1]

    for a, b in zip(chain(step, k, 6, True), chain(step, k, 6, False)):
        assert torch.isfinite(a).all() and torch.equal(a, b)


def test_allocation_free_entry_point():
    """Its twiddle table is rewritten by a kernel of every call."""
    import torch
    from paper_2607_19378_b200 import hyenand as hn
    sets = []
    for dims in [(20, 70), (9, 33, 12), (40, 17)]:
        w, arrays = W.random_problem(dims, B=1, C=2, dtype="f32", seed=142)
        t = [torch.as_tensor(a).cuda().contiguous() for a in arrays]
        sets.append((dims, t, t[3].stride(0)))

    def run(pause):
        out = []
        for _ in range(5):
            for dims, (q, k, v, h), stride in sets:
                y = torch.zeros_like(q)
                hn.hyenand_forward_noalloc(dims, 1, 2, 0, 0, q, k, v, h, stride, y)
                out.append(y)
                if pause:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return out

    for a, b in zip(run(True), run(False)):
        assert torch.equal(a, b)
