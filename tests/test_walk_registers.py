"""The walks of sampled drafts hold a CTA's share of the vocabulary in registers (csrc/sampled_q.cu): no instance of them
may need local memory, by the compiler's own account."""
import os
import re
import subprocess

import pytest

from paper_2509_18824_b200 import build


def test_walks_use_no_local_memory(tmp_path):
    nvcc = build._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    r = subprocess.run([nvcc] + build.NVCC_FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, "sampled_q.cu"), "-o", str(tmp_path / "q.o")],
                       capture_output=True, text=True, check=True)
    per_kernel = re.findall(r"Function properties for (\S*walk_q\S*)\n\s+(\d+) bytes stack frame, (\d+) bytes spill stores", r.stdout + r.stderr)
    assert len(per_kernel) == 6, r.stderr               # trees and chains, 8, 16 and 40 entries per thread
    assert all(int(stack) == 0 and int(spill) == 0 for _, stack, spill in per_kernel), per_kernel
