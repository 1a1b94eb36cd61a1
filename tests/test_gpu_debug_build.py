"""The checked build (-DHYENAND_DEBUG): every kernel's global-memory accesses compared with the ranges its call may
touch.  The parity suites run once more against that library in a child process; tests/conftest.py fails any test
after which the checker has counted an access."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SUITES = ["tests/test_gpu_parity.py", "tests/test_gpu_mixer.py", "tests/test_gpu_synthesis.py", "tests/test_gpu_backward.py",
          "tests/test_gpu_slice.py", "tests/test_gpu_core_lengths.py", "tests/test_gpu_backward_spectral.py", "tests/test_gpu_len3.py",
          "tests/test_zz_no_alloc.py"]
# the largest long 1-D cases run for minutes under the checker and add no kernel the smaller ones leave out
SKIP = "not large_padded_sizes and not above_2_pow_20 and not tensor_maps_follow"


def _child(code_or_args):
    env = dict(os.environ, HYENAND_LIB="debug")
    return subprocess.run([sys.executable] + code_or_args, cwd=ROOT, env=env, capture_output=True, text=True, timeout=3000)


@pytest.mark.gpu
def test_checker_counts_an_access_outside_the_registered_ranges():
    r = _child(["-c", "from paper_2607_19378_b200 import hyenand as H; print(H.hyenand_debug_build(), H.hyenand_debug_selftest())"])
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split()[-2:] == ["True", "1000"], r.stdout


@pytest.mark.gpu
def test_product_library_has_no_checker():
    from paper_2607_19378_b200 import hyenand as H
    if os.environ.get("HYENAND_LIB") == "debug":
        pytest.skip("running against the checked build")
    assert not H.hyenand_debug_build()
    assert H.hyenand_debug_violations()[0] == -1 and H.hyenand_debug_selftest() == -1


@pytest.mark.gpu
def test_parity_suites_pass_with_no_out_of_range_access():
    r = _child(["-m", "pytest", "-m", "gpu", "-x", "-q", "-p", "no:cacheprovider", "-k", SKIP] + SUITES)
    assert r.returncode == 0, (r.stdout[-3000:], r.stderr[-2000:])
