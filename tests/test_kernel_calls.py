"""The block-per-ant kernels are compiled without out-of-line calls: forms of
them with calls have faulted on the GPU for a reason that was not found."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2203_02228_gb300 import build


@pytest.mark.skipif(shutil.which(os.environ.get("NVCC", "nvcc")) is None, reason="needs nvcc")
def test_block_kernels_make_no_calls(tmp_path):
    cmd = [os.environ.get("NVCC", "nvcc")] + build.NVCC_FLAGS + [
        "-I", build.INCLUDE, "-Xptxas", "-v", "-cubin", "-o", str(tmp_path / "ants.cubin"),
        os.path.join(build.CSRC, "ants.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    kernel, seen = None, set()
    for line in (r.stdout + r.stderr).splitlines():
        m = re.search(r"Compiling entry function '(\w+)'", line)
        if m:
            kernel = m.group(1)
        m = re.search(r"Function properties for (\w+)", line)
        if m and "k_ants_blk" in kernel:
            assert m.group(1) == kernel, "%s calls %s" % (kernel, m.group(1))
            seen.add(kernel)
    assert len(seen) == 8  # list width, registers, one colony or a batch
