"""Calls inside a stream capture: forward, operator and backward on every path, the first call with a filter shared over the
batch among them (it allocates), replayed on new values in the same buffers."""
import pytest
import torch

from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

# one-kernel grids, general 2-D and 3-D, planes, long lines
GRIDS = [((100,), True), ((2000,), True), ((20, 30), False), ((64, 64), False), ((40, 90), False), ((300, 40), False), ((9, 20, 12), False),
         ((20, 40, 50), False), ((5, 96, 96), False), ((66, 70, 65), False), ((6001,), True)]


def captured(call):
    """replay() runs the captured call and returns its outputs"""
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out = call()

    def replay():
        graph.replay()
        torch.cuda.synchronize()
        return [t.clone() for t in (out if isinstance(out, tuple) else (out,))]
    replay.call = call                                       # the objects the captured kernels use live as long
    return replay


def check_replay(make, tensors):
    """make() -> a call on fresh objects.  Its first call is captured; replays equal calls outside a capture."""
    direct = make()
    direct()                                                 # loads the kernels
    replay = captured(make())
    for seed in (1, 2):
        g = torch.Generator(device="cuda").manual_seed(seed)
        for t in tensors:
            t.copy_(torch.randn(t.shape, generator=g, device="cuda"))
        got, want = replay(), direct()
        torch.cuda.synchronize()
        for a, b in zip(got, want if isinstance(want, tuple) else (want,)):
            assert torch.isfinite(b).all() and torch.equal(a, b)


@pytest.mark.parametrize("dtype,shared", [("f32", True), ("bf16", False), ("bf16", True)])
@pytest.mark.parametrize("dims,causal", GRIDS, ids=str)
def test_first_calls(dims, causal, dtype, shared):
    from paper_2607_19378_b200 import hyenand as hn
    w, arrays = W.random_problem(dims, B=2, C=3, dtype=dtype, causal=causal, h_shared=shared, seed=151)
    q, k, v, h = (t.cuda() for t in arrays)
    g = torch.ones(w.C, device="cuda")

    def forward():
        plan = hn.Plan(dims, w.B, w.C, causal=causal, dtype=w.torch_dtype)
        return lambda: plan.forward(q, k, v, h)

    def operator():
        mixer = hn.Mixer(dims, w.B, w.C, mode=w.mode, dtype=w.torch_dtype)
        return lambda: mixer.forward(q, k, v, h, g, g)

    def backward():
        grad = hn.Backward(dims, w.B, w.C, mode=w.mode, dtype=w.torch_dtype)
        return lambda: grad(q, k, v, h, q)

    for make in (forward, operator, backward):
        check_replay(make, (q, k, v))


def test_groups_on_two_lanes(monkeypatch):
    """Several groups: the filter of all channels needs more room than a group's, taken inside the capture."""
    from paper_2607_19378_b200 import hyenand as hn
    monkeypatch.setenv("HYENAND_GROUP_SLICES", "2")
    monkeypatch.setenv("HYENAND_LANES", "2")
    for dims in [(40, 90), (5, 96, 96)]:
        w, arrays = W.random_problem(dims, B=2, C=5, dtype="f32", h_shared=True, seed=152)
        q, k, v, h = (t.cuda() for t in arrays)

        def forward():
            plan = hn.Plan(dims, w.B, w.C, dtype=w.torch_dtype)
            return lambda: plan.forward(q, k, v, h)
        check_replay(forward, (q, k, v))
