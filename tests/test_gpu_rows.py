"""Row kernels whose rows travel ahead as copies of whole 16-byte granules: last rows of tensors that end off a granule, odd row
lengths, an odd number of rows, and the gates of rows back in rounds."""
import pytest
import torch

from parity_util import assert_parity
import oracle
from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

# rows padded to 1024 (385 .. 512), 512 (193 .. 256), 768 and 384 points
DIMS = [(3, 511), (1, 3, 385), (5, 512), (70, 509), (3, 255), (66, 200), (41, 256), (3, 300), (20, 150)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("dims", DIMS, ids=str)
def test_rows_at_the_ends_of_their_tensors(dims, dtype):
    from paper_2607_19378_b200 import hyenand as hn
    w, arrays = W.random_problem(dims, B=1, C=3, dtype=dtype, seed=181)
    plan = hn.Plan(w.dims, w.B, w.C, dtype=w.torch_dtype)
    y = plan.forward(*(t.cuda() for t in arrays))
    torch.cuda.synchronize()
    assert hn.hyenand_plan_device_status(plan.handle) == 0 and hn.hyenand_plan_guard_damage(plan.handle) == 0
    plan.close()
    assert_parity(y.cpu(), oracle.conv_fft(*arrays, "linear"), arrays[0], w)
