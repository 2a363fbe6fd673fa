"""What the native code remembers in the process. A kernel's shared-memory limit belongs to a device: code that raises it
once a process leaves every further device at the default, and launches there fail (a host of several GPUs is not at
hand, so the sources are read)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2404_08299_gb300", "csrc")


def functions(text):
    """Bodies of the namespace-level functions (their closing brace stands at the line's start)."""
    return re.findall(r"^[A-Za-z].*?\{\n.*?^\}", text, re.M | re.S)


def test_shared_memory_limits_are_not_kept_by_process():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for body in functions(text):
            if "cudaFuncAttributeMaxDynamicSharedMemorySize" not in body:
                continue
            seen += 1
            assert not re.search(r"\bstatic\s+(const\s+)?(bool|int|auto|std::once_flag)\b", body), path
            assert "once_flag" not in body and "call_once" not in body, path
    assert seen >= 3  # the weighted radix scatter, the small batch's preparation, the block sort
