"""State that belongs to a device lives in the context, not in the process."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_09290_b200", "csrc")


def test_kernel_attributes_are_remembered_per_context():
    """A function attribute is set on the current device: remembered in a function-local static, the first context's device would be the
    only one on which the launches that need it work, and two host threads would race on the flag."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = open(path).read()
        assert not re.search(r"\bstatic\s+(bool|int|unsigned)\s+\w+(\[\w+\])?\s*=", src), os.path.basename(path)
        for m in re.finditer(r"cudaFuncSetAttribute", src):
            around = src[max(0, m.start() - 400):m.end() + 400]
            assert "attr_done" in around, f"{os.path.basename(path)}: an attribute outside the context's record"
