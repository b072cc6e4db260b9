"""The plan kernel keeps its parameters where they were passed (CPU: compiled, not run): each
block picks one plan of the launch's set, and with the set passed by value it would copy the
whole set to its stack first, which costs every attention call ~2 us."""
import os
import re
import subprocess

import pytest

import __graft_entry__


def test_plan_kernel_has_no_stack(tmp_path):
    b = __graft_entry__._build_module()
    if not os.path.exists(b._nvcc()):
        pytest.skip("no nvcc")
    src = os.path.join(b.CSRC, "importance.cu")
    r = subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-Xptxas", "-v", "-c", src, "-o", str(tmp_path / "o.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    log = r.stdout + r.stderr
    found = re.findall(r"Function properties for \S*attn_plan_kernel\S*\s+(\d+) bytes stack frame, "
                       r"(\d+) bytes spill stores", log)
    assert found == [("0", "0")], found
