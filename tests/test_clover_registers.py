"""The inverse clover blocks are formed in registers, as csrc/clover_inverse.cuh says:
ptxas reports no stack frame for the kernel of the FP64 even-odd set-up (the other
user inlines the same function)."""
import os
import re
import subprocess

from paper_2412_06347_gb300 import build as b


def test_no_stack_frame(tmp_path):
    r = subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-Xptxas", "-v", "-c", os.path.join(b.CSRC, "evenodd.cu"), "-o",
                        str(tmp_path / "o.o")], capture_output=True, text=True, check=True)
    m = re.search(r"Function properties for \S*clover_inverse_kernel\S*\s+(\d+) bytes stack frame", r.stderr)
    assert m and int(m.group(1)) == 0, m and m.group(0)
