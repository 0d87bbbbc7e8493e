"""Rules that the kernel sources keep and no run can show."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_16213_gb300", "csrc")


def test_no_read_only_loads():
    """Kernels are brought up while their predecessor still writes what they will read, so none loads
    through the read-only path, which is for data that does not change while the kernel is resident."""
    for name in sorted(os.listdir(CSRC)):
        code = re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())
        assert not re.search(r"__ldg\b|__restrict__|ld\.global(\.\w+)*\.nc\b", code), name
