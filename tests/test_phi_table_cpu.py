"""The generated table of phi/Phi and log Phi (csrc/phi_table.h), as text."""
import os
import re

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_04582_gb300", "csrc",
                      "phi_table.h")


def _read():
    with open(HEADER) as f:
        text = f.read()
    return text, [int(w, 16) for w in re.findall(r"0x([0-9a-f]{16})ull", text)]


def test_table_type_is_aligned_for_16_byte_loads():
    # an array of 8-byte words is only 8-byte aligned by its type, and the kernels load 16 bytes at a time
    text, words = _read()
    decl = re.search(r"__device__ const (\w+) g_phi_table\[", text)
    assert decl and decl.group(1) == "ulonglong2"
    nodes, row = (int(v) for v in re.search(r"kPhiNodes = (\d+).*kPhiRow = (\d+)", text).groups())
    assert len(words) == nodes * row and row % 2 == 0
