"""The transform kernels of the largest rings keep their words in registers (read from the assembler's own report)."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2606_10477_gb300 import build

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc not available")
@pytest.mark.parametrize("log_n", [16, 17])
def test_transform_kernels_do_not_spill(log_n, tmp_path):
    """A few constants of a lane may go to the stack; the words and the open sums of 128 bits (at least 16 words) may not."""
    src = os.path.join(build.SRC, f"ntt_inst_{log_n}.cu")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", src, "-o", str(tmp_path / "x.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    names = re.findall(r"Compiling entry function '(\w+)'", r.stderr)
    frames = re.findall(r"(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr)
    assert len(names) == len(frames) and len(names) >= 10
    for name, f in zip(names, frames):
        assert max(map(int, f)) <= 64, (name, f)
