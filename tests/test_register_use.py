"""Register spills of kernels that run at their register limit, as ptxas reported them when the library was built (no GPU).
The bounds are what the kernels need by themselves: twiddles held in registers across a wait, or a second copy of a row's first
pass, showed as two to forty times as much and cost measured time."""
import os
import re

import pytest


def spill_loads(source):
    """mangled kernel name -> bytes of spill loads, from the build's ptxas output"""
    from paper_2607_19378_b200 import build as bld
    bld.build()
    log = os.path.join(bld.OBJ, source + ".ptxas.log")
    if not os.path.exists(log):
        pytest.skip("the objects were built elsewhere")
    out, name = {}, None
    for line in open(log):
        m = re.search(r"Compiling entry function '(\S+)'", line)
        name = m.group(1) if m else name
        m = re.search(r"(\d+) bytes spill loads", line)
        if m and name:
            out[name] = int(m.group(1))
    assert out
    return out


@pytest.mark.parametrize("kernel,limit", [("rows_fwd_w_kernelIfLi10ELi0ELb1E", 200), ("rows_fwd_w_kernelIfLi10ELi1ELb1E", 112),
                                          ("rows_inv_w_kernelIfLi10ELi0ELb1E", 136), ("rows_inv_w_kernelIfLi10ELi1ELb1E", 144)])
def test_rows_of_1024_points(kernel, limit):
    """Grids that fill the GPU: no more than before the kernels waited for their predecessors (dependent launches)."""
    found = [v for k, v in spill_loads("rows_w").items() if kernel in k]
    assert len(found) == 1 and found[0] <= limit, found


def test_rows_of_three_times_a_power_of_two():
    rows = {k: v for k, v in spill_loads("rows_w").items() if re.search(r"Li2[234]E", k)}
    assert len(rows) == 2 * 3 * 5 and max(rows.values()) <= 16, {k: v for k, v in rows.items() if v > 16}


def test_norms_keep_their_channels_in_registers():
    """mixer_post_kernel<T, VEC, NW, KEEP>: KEEP channels of a thread stay in registers between the sum and the result."""
    kept = {k: v for k, v in spill_loads("mixer").items() if re.search(r"mixer_post_kernelI\w+?Li\dELi\d+ELi(4|16|24)E", k)}
    assert len(kept) >= 2 * 2 * 5 and max(kept.values()) == 0, {k: v for k, v in kept.items() if v}


def test_rows_that_travel_ahead_spill_nothing():
    """rows_fwd_w_kernel<T, LOG2P, MODE, LATE, AHEAD>: four warps with 168 registers a thread.  Periodic rows, which have no such
    variant, at what they have had from the start."""
    rows = spill_loads("rows_w")
    ahead = {k: v for k, v in rows.items() if re.search(r"rows_fwd_w_kernelI\w+?Li\d+ELi\dELb\dELb1E", k)}
    assert len(ahead) == 2 * 3 + 1 and max(ahead.values()) == 0, ahead
    periodic = {k: v for k, v in rows.items() if re.search(r"rows_fwd_w_kernelI\w+?Li10ELi3E", k)}
    assert len(periodic) == 4 and max(periodic.values()) <= 232, periodic
