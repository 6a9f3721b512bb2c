"""Kernels that hold several code paths at once stay within their registers:
the persistent batch kernel has the products of one to eight digits and the
element-wise operations, and none of its values lives in local memory."""
import os
import subprocess

from paper_2407_13055_gb300 import build


def test_persistent_kernel_does_not_spill(tmp_path):
    src = os.path.join(build.CSRC, "k_keyswitch.cu")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-cubin", src, "-o",
                        str(tmp_path / "k.cubin")], capture_output=True, text=True, check=True)
    lines = r.stderr.splitlines()
    at = [i for i, s in enumerate(lines) if "Function properties for" in s and "k_persistent" in s]
    assert len(at) == 1
    assert lines[at[0] + 1].strip().startswith("0 bytes stack frame, 0 bytes spill stores, 0 bytes spill loads")
