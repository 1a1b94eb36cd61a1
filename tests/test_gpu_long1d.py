"""Long 1-D kernels at the edges of their tiles: slices that are whole rows of the second transform (tensor copies), whole
multiples of 8 bytes, of pairs, and neither, for every first-transform length; filters whose rows serve several batch entries."""
import pytest
import torch

from parity_util import assert_parity, run_gpu
import oracle
from paper_2607_19378_b200 import workloads as W

pytestmark = pytest.mark.gpu

# padded 2^14 .. 2^20: first transforms of 128, 256, 512 and 1024 points
LENGTHS = [8192, 8196, 8198, 16384, 16381, 32768, 32766, 65536, 65533, 131072, 131074, 262144, 262139, 262148, 524288, 524285]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("L", LENGTHS)
def test_tiles(L, dtype):
    w, (q, k, v, h) = W.random_problem((L,), B=2, C=1, dtype=dtype, causal=True, h_shared=L % 8 == 0, seed=171)
    y, path = run_gpu(w, q, k, v, h)
    assert path == "ct1d"
    assert_parity(y, oracle.conv_fft(q, k, v, h, "causal"), q, w)


@pytest.mark.parametrize("L,B,C,dtype", [(9001, 5, 96, "f32"), (20000, 7, 40, "bf16"), (40000, 3, 33, "f32"), (270000, 2, 17, "bf16")])
def test_filter_rows_that_serve_several_entries(L, B, C, dtype):
    """More rows than lane groups in flight: a unit is one row of the filter and that row of several batch entries."""
    w, (q, k, v, h) = W.random_problem((L,), B=B, C=C, dtype=dtype, causal=True, h_shared=True, seed=172)
    y, _ = run_gpu(w, q, k, v, h)
    sel = [0, C // 2, C - 1]                                  # whole slices of three channels, every entry of the batch
    pick = lambda t: t[..., sel, :].contiguous()
    w3 = W.Workload("pick", (L,), B, 3, dtype, causal=True, h_shared=True, seed=172)
    assert_parity(pick(y), oracle.conv_fft(pick(q), pick(k), pick(v), pick(h), "causal"), pick(q), w3)
    assert bool(torch.isfinite(y.float()).all())
