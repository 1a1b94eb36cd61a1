"""Which of their two variants the forward row kernels take: rows that travel ahead wait for their copies, so a call takes them
only where a wait that gives up has a status word to say so in, and where they are the faster ones."""
import pytest
import torch

from parity_util import assert_parity
import oracle
from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

AHEAD, STAGED = 128, 256                                       # threads per CTA


def row_kernels(call):
    """Threads per CTA of the forward row kernels that call() launches, from its capture into a graph."""
    from cuda.bindings import driver
    call()                                                     # loads the kernels
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    raw = driver.CUgraph(g.raw_cuda_graph())
    _, _, n = driver.cuGraphGetNodes(raw)
    err, nodes, n = driver.cuGraphGetNodes(raw, n)
    assert err == driver.CUresult.CUDA_SUCCESS
    threads = []
    for node in nodes[:n]:
        if driver.cuGraphNodeGetType(node)[1] != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        params = driver.cuGraphKernelNodeGetParams(node)[1]
        if b"rows_fwd_w_kernel" in driver.cuFuncGetName(params.func)[1]:
            threads.append(params.blockDimX)
    g.replay()
    torch.cuda.synchronize()
    return threads


@pytest.mark.parametrize("dims,dtype", [((40, 500), "f32"), ((40, 500), "bf16"), ((300, 512), "f32"), ((80, 256), "f32")], ids=str)
def test_calls_without_a_status_word_make_no_wait_for_copies(dims, dtype):
    from paper_2607_19378_b200 import hyenand as hn
    w, (q, k, v, h) = W.random_problem(dims, B=1, C=2, dtype=dtype, seed=231)
    dev = [t.cuda() for t in (q, k, v, h)]
    y = torch.empty_like(dev[0])
    code = hn.HYENAND_F32 if dtype == "f32" else hn.HYENAND_BF16
    found = row_kernels(lambda: hn.hyenand_forward_noalloc(w.dims, 1, 2, 0, code, *dev, dev[3][0].numel(), y))
    assert found and set(found) == {STAGED}, found
    assert_parity(y.cpu(), oracle.conv_fft(q, k, v, h, "linear"), q, w)


# filter rows, k*v rows.  fp32 of 512 points: ahead for the filter's alone, from three rounds of the GPU's groups on; 1024 points:
# ahead, but for rows that are one round of the staged groups and more than one of those, or that let the next kernel in early
ROUTES = [((256, 256), 16, "f32", STAGED, STAGED), ((70, 199), 160, "f32", AHEAD, STAGED), ((70, 199), 160, "bf16", STAGED, STAGED),
          ((300, 512), 3, "f32", STAGED, STAGED), ((512, 512), 4, "f32", STAGED, STAGED), ((300, 512), 4, "bf16", AHEAD, STAGED),
          ((300, 511), 8, "bf16", AHEAD, AHEAD), ((40, 511), 5, "f32", AHEAD, STAGED)]


@pytest.mark.parametrize("dims,C,dtype,h_rows,kv_rows", ROUTES, ids=str)
def test_rows_ahead_where_they_are_the_faster_ones(dims, C, dtype, h_rows, kv_rows):
    from paper_2607_19378_b200 import hyenand as hn
    w, (q, k, v, h) = W.random_problem(dims, B=1, C=C, dtype=dtype, seed=232)
    dev = [t.cuda() for t in (q, k, v, h)]
    plan = hn.Plan(w.dims, 1, C, dtype=w.torch_dtype)
    y = torch.empty_like(dev[0])
    found = row_kernels(lambda: plan.forward(*dev, y))
    status, damage = hn.hyenand_plan_device_status(plan.handle), hn.hyenand_plan_guard_damage(plan.handle)
    plan.close()
    assert (status, damage) == (0, 0)
    assert sorted(found) == sorted((h_rows, kv_rows)), found
    for c in sorted({0, 1, C - 1}):
        one = [t[:, c:c + 1] for t in (q, k, v, h)]
        ws = W.Workload("one", w.dims, 1, 1, dtype)
        assert_parity(y[:, c:c + 1].cpu(), oracle.conv_fft(*one, "linear"), one[0], ws, what=f"channel {c}")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("dims", [(3, 511), (33, 401)], ids=str)
def test_groups_that_start_off_a_granule(dims, dtype, monkeypatch):
    """Slices of an odd volume in groups of two and one: tensors whose first and last granule are cut."""
    from paper_2607_19378_b200 import hyenand as hn
    for group in ("1", "2"):
        monkeypatch.setenv("HYENAND_GROUP_SLICES", group)
        w, arrays = W.random_problem(dims, B=1, C=5, dtype=dtype, seed=233)
        plan = hn.Plan(w.dims, 1, 5, dtype=w.torch_dtype)
        y = plan.forward(*(t.cuda() for t in arrays))
        torch.cuda.synchronize()
        assert hn.hyenand_plan_device_status(plan.handle) == 0 and hn.hyenand_plan_guard_damage(plan.handle) == 0
        plan.close()
        assert_parity(y.cpu(), oracle.conv_fft(*arrays, "linear"), arrays[0], w, what=f"groups of {group}")
