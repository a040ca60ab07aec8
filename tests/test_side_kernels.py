"""What the kernels over one operand's blocks may read: the 3xTF32 split runs without the digit
kernels' exponent arrays, so the argument that it takes does not hold them (a helper shared with
those kernels could read them through a null pointer otherwise)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1910_13555_gb300", "csrc", "numeric_emu.cu")


def _struct(src, name):
    return re.search(r"struct %s\b[^{]*\{(.*?)\n\};" % name, src, re.S).group(1)


def test_tf32_split_cannot_reach_what_its_launch_does_not_set():
    src = open(SRC).read()
    arg = re.search(r"__global__ void k_tf32_split\((?:const )?(\w+) &?S\)", src).group(1)
    fields = set(re.findall(r"[\s*](\w+)(?=[,;])", _struct(src, arg)))
    launch = re.search(r"\nvoid execute_tf32x3\(.*?\n\}", src, re.S).group(0)
    common = re.search(r"\nSideArgs side_args\(.*?\n\}", src, re.S).group(0)
    assert fields <= set(re.findall(r"\bS\.(\w+) = ", launch + common))
