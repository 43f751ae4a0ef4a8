"""State that belongs to a device is not remembered for the whole process.

A kernel's dynamic shared-memory limit (cudaFuncSetAttribute) holds for the
device that was current when it was set.  Code that remembers in a static
variable that it has set one launches with the default limit of 48 KB on the
next device, and the launch is rejected.  Read from the sources: no function
that sets an attribute has a mutable static local.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_00495_gb300", "csrc")


def functions(text):
    """Bodies of the top-level functions (braces at column 0 of their closing line)."""
    return re.findall(r"^[^\s#/}].*?\{\n(.*?)^\}", text, flags=re.M | re.S)


def test_attributes_are_set_for_the_current_device():
    seen = 0
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//.*|\"[^\"\n]*\"", "", open(f).read())
        for body in functions(text):
            if "cudaFuncSetAttribute" in body:
                seen += 1
                assert not re.search(r"\bstatic\s+(?!constexpr|const\b)", body), (f, body[:200])
    assert seen >= 5
