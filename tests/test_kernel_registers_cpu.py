"""What ptxas reports for the kernels whose inner loops must not touch local memory (their shared memory leaves almost no L1): spilled
registers and arrays with a changing index both show up as a stack frame.  Compiles a source file; needs nvcc, no GPU."""
import re
import shutil
import subprocess

import pytest

from paper_2505_16381_b200 import build

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")


def stack_frames(source, tmp_path):
    """{(kernel, template arguments): bytes of stack}"""
    r = subprocess.run(["nvcc", *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", str(build.CSRC / source), "-o", str(tmp_path / "out.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    found = re.findall(r"Compiling entry function '\S*?\d+([a-z]\w*?_kernel)I(\w+?)Ev?v?N\S*' for 'sm_100a'\n.*\n\s*(\d+) bytes stack frame",
                       r.stderr + r.stdout)
    return {(name, args): int(n) for name, args, n in found}


@pytest.mark.parametrize("source,kernel,limits", [
    ("levels.cu", "key_cache_kernel", {"Li64E": 0, "Li128E": 0}),
    ("chunk_chain.cu", "chunk_chain_kernel", {"Li64E": 0}),
    ("chunk_prep.cu", "chunk_prep_kernel", {"Li64E": 8, "Li128E": 0}),   # (8: one pointer that all roles of the block share)
])
def test_stack_frames(source, kernel, limits, tmp_path):
    frames = stack_frames(source, tmp_path)
    for instance, limit in limits.items():
        mine = {n: b for n, b in frames.items() if n[0].endswith(kernel) and n[1].startswith(instance)}
        assert mine, (instance, sorted(frames))
        assert max(mine.values()) <= limit, mine
