"""Properties of the kernel sources that no run can show (CPU only)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_08733_gb300", "csrc")


def _sources(*ext):
    return {os.path.basename(f): open(f).read() for e in ext for f in glob.glob(os.path.join(CSRC, "*" + e))}


def test_no_restrict_name_for_a_buffer_the_kernel_writes():
    """A kernel that reads the residuals (or the auxiliaries' residuals) also writes them, and
    what it reads may be what the launch before it still writes: no name of such a
    buffer may promise the compiler that nothing else touches it."""
    for name, text in _sources(".cuh").items():
        bound = re.findall(r"__restrict__\s+\w+\s*=\s*static_cast<[^>]*>\(prm\.(\w+)\)", text)
        assert not bound, (name, bound)
