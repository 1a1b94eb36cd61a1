"""Kernel synthesis on the tensor cores with several tiles of taps, and several chunks of channels in each, per CTA."""
import numpy as np
import pytest
import torch

from test_gpu_synthesis import gpu_synthesize, make_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("C", [5, 32, 70, 100])
@pytest.mark.parametrize("dims,mode,Hf", [((20, 20), "linear", 32), ((2000,), "causal", 32), ((9, 10, 11), "linear", 64)], ids=str)
def test_many_tiles_per_cta(dims, mode, Hf, C, dtype):
    """A batch of 300 entries leaves each of them one or two CTAs for all of its tiles; one entry alone has a CTA per tile."""
    B = 300
    p = make_params(len(dims), Hf, 2, C, 1, mode, seed=241)
    one = gpu_synthesize(dims, mode, 1, C, Hf, 2, p, dtype)
    many = dict(p, gamma=np.repeat(p["gamma"], B, 0), beta=np.repeat(p["beta"], B, 0))
    assert bool(torch.isfinite(one.float()).all())
    assert torch.equal(gpu_synthesize(dims, mode, B, C, Hf, 2, many, dtype), one.expand((B,) + one.shape[1:]))
