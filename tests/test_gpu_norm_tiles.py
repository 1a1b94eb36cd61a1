"""Norms of Eq. 2 on tiles of 64 tokens and 16 warps (many channels, few tokens): channels kept in registers and read twice, rows
that end inside a tile."""
import pytest
import torch

import oracle
from oracle import mixer as omx
from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,B,C,dtype", [((64, 64), 2, 130, "bf16"), ((50, 41), 4, 200, "f32"), ((32, 32), 8, 400, "bf16"), ((1030,), 8, 128, "f32")], ids=str)
def test_many_channels(dims, B, C, dtype):
    from paper_2607_19378_b200 import hyenand as hn
    w, (q, k, v, h) = W.random_problem(dims, B=B, C=C, dtype=dtype, seed=191)
    g_in, g_out = torch.linspace(0.5, 1.5, C), torch.linspace(1.5, 0.5, C)
    mx = hn.Mixer(w.dims, B, C, mode=w.mode, dtype=w.torch_dtype, eps=1e-6)
    y = mx.forward(q.cuda(), k.cuda(), v.cuda(), h.cuda(), g_in.cuda(), g_out.cuda())
    torch.cuda.synchronize()
    mx.close()
    ref = omx.hyena_mixer(q, k, v, h, g_in, g_out, eps=1e-6)
    assert oracle.rel_l2(y.cpu(), ref) <= (1e-5 if dtype == "f32" else 2e-3)
