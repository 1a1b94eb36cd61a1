"""The window of the kernel synthesis in its two variants (up to 16 hidden units on the ALUs, more on the tensor cores)."""
import numpy as np
import pytest
import torch

from test_gpu_synthesis import gpu_synthesize, make_params

pytestmark = pytest.mark.gpu


def window_only(N, Hf, C, mode, sigma=None):
    """A network whose value is bout exactly: what is left of K is the window."""
    p = make_params(N, Hf, 2, C, 1, mode, seed=201)
    g = np.random.default_rng(202)                            # (the same window and biases at every width)
    p["Wout"] = np.zeros_like(p["Wout"])
    p["bout"] = g.uniform(0.5, 2.0, C).astype(np.float32)
    shape = (C,) if mode == "causal" else (N, C)
    p["window"] = np.exp(g.uniform(-2.0, 1.0, shape)).astype(np.float32) if sigma is None else np.full(shape, sigma, np.float32)
    return p


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("dims,mode", [((300,), "causal"), ((300,), "linear"), ((17, 20), "linear"), ((16, 32), "circular"), ((9, 10, 11), "linear")], ids=str)
def test_both_variants_have_the_same_window(dims, mode, dtype):
    """One arithmetic for w(c): not a bit depends on how wide the network is."""
    C = 40
    narrow, wide, wider = (gpu_synthesize(dims, mode, 1, C, Hf, 2, window_only(len(dims), Hf, C, mode), dtype) for Hf in (16, 32, 64))
    assert torch.equal(narrow, wide) and torch.equal(narrow, wider)


@pytest.mark.parametrize("Hf", [16, 32, 64])
@pytest.mark.parametrize("sigma", [1e-12, 1e-20, 1e-30])
def test_window_narrower_than_the_grid(sigma, Hf):
    """1 / sigma^2 overflows fp32: the centre tap is the network's value and all others are zero."""
    dims, C = (6, 5), 3
    p = window_only(2, Hf, C, "linear", sigma)
    h = gpu_synthesize(dims, "linear", 1, C, Hf, 2, p, "f32").cpu()
    want = torch.zeros_like(h)
    want[0, :, 5, 4] = torch.from_numpy(p["bout"])
    assert torch.equal(h, want)
