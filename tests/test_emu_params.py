"""Every field of the emulated kernels' argument is read by some kernel: it is copied with every
launch and every plan of a batch."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1910_13555_gb300", "csrc", "numeric_emu.cu")


def test_no_field_is_only_set():
    src = open(SRC).read()
    body = re.search(r"struct EmuParams \{(.*?)\n\};", src, re.S).group(1)
    fields = set(re.findall(r"[\s*](\w+)(?=[,;])", re.sub(r"//[^\n]*", "", body)))
    assert {"Cin", "desc", "ents", "a_tf"} <= fields
    read = set(re.findall(r"\bP\.(\w+)\b(?! = )", src)) | set(re.findall(r"get\([^)]*\)\.(\w+)", src))
    assert fields <= read
