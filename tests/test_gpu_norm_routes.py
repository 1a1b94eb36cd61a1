"""Norms of Eq. 2 on tiles of 64 tokens and 16 warps: channels kept in registers (24 per thread), and the kernel that writes the
gates out (grids of several kernels), each at the edges of its tiles and read once and twice."""
import pytest
import torch

import oracle
from oracle import mixer as omx
from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [((64, 64), 2, 257, "bf16"), ((50, 82), 2, 384, "bf16"), ((14, 15), 32, 192, "bf16"), ((14, 15), 32, 256, "f32"),     # one kernel
         ((80, 81), 2, 260, "bf16"), ((45, 90), 2, 161, "bf16"), ((45, 90), 2, 129, "f32"), ((16, 16, 25), 3, 256, "bf16"),       # several
         ((14, 14), 8, 768, "bf16"), ((14, 15), 32, 400, "f32")]                                                      # past the rule


@pytest.mark.parametrize("dims,B,C,dtype", CASES, ids=str)
def test_tiles(dims, B, C, dtype):
    from paper_2607_19378_b200 import hyenand as hn
    w, (q, k, v, h) = W.random_problem(dims, B=B, C=C, dtype=dtype, seed=211)
    g_in, g_out = torch.linspace(0.5, 1.5, C), torch.linspace(1.5, 0.5, C)
    mx = hn.Mixer(w.dims, B, C, mode=w.mode, dtype=w.torch_dtype, eps=1e-6)
    y = mx.forward(q.cuda(), k.cuda(), v.cuda(), h.cuda(), g_in.cuda(), g_out.cuda())
    torch.cuda.synchronize()
    mx.close()
    ref = omx.hyena_mixer(q, k, v, h, g_in, g_out, eps=1e-6)
    assert oracle.rel_l2(y.cpu(), ref) <= (1e-5 if dtype == "f32" else 2e-3)
