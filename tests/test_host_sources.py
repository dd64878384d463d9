"""Rules that the CUDA sources keep, checked on the text (one GPU cannot show them)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2412_19027_gb300", "csrc", "*.cu*")))


def test_kernel_attributes_are_set_per_device():
    """A kernel's shared-memory limit belongs to one device: no process-wide flag of a function decides whether it
    is set (the one flag there is, g_noalloc_ready, is an array over devices)."""
    assert SOURCES
    for path in SOURCES:
        text = open(path).read()
        if "cudaFuncSetAttribute" not in text:
            continue
        flags = re.findall(r"^\s+static\s+(?:bool|int|std::once_flag)\s+(\w+)\s*(?:=[^;]*)?;", text, re.M)
        assert not flags, (os.path.basename(path), flags)
