"""Kernels that the dispatch rules keep from small shapes, on the small shapes of the other GPU tests, on a B200: the same tests in child
processes with the batch kernel left out (the prefill kernels and the warp-level batch kernel serve its calls) and with it
wherever it can serve.  What runs then is checked without a device in test_routes_cpu.py."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WITHOUT = {
    "test_prefill_gpu.py": "small_and_ragged or narrow_tiles or one_hot or split_k or zero_input or outside_y or group_prefill_parity",
    "test_prefill_ta_gpu.py": "widths or guard_band or keep_their_bits",
    "test_gated_gpu.py": "gated_parity or outside_y",
    "test_kv_gpu.py": "prefill_kernels_see",
    "test_kv_append_gpu.py": "batch_of_rows_see",
    "test_mid_gpu.py": "oracle or lines or outside",
}
ALWAYS = {"test_narrow_gpu.py": "", "test_kv_append_gpu.py": "batch_of_rows_see", "test_gated_gpu.py": "gated_parity", "test_kv_gpu.py": "prefill_kernels_see", "test_prefill_gpu.py": "one_hot or zero_input"}


def child(setting, name, chosen):
    env = dict(os.environ, QLINEAR_GEMM_NARROW=setting)
    cmd = [sys.executable, "-m", "pytest", os.path.join("tests", name), "-m", "gpu", "-x", "-q", "-p", "no:cacheprovider"]
    r = subprocess.run(cmd + (["-k", chosen] if chosen else []), env=env, cwd=ROOT, timeout=600, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    assert r.returncode == 0, r.stdout[-4000:]


@pytest.mark.parametrize("name", WITHOUT)
def test_with_the_batch_kernel_left_out(_built_library, name):
    child("0", name, WITHOUT[name])


@pytest.mark.parametrize("name", ALWAYS)
def test_with_the_batch_kernel_wherever_it_can_serve(_built_library, name):
    child("2", name, ALWAYS[name])
