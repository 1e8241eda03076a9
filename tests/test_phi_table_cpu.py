"""The generated table of phi/Phi and log Phi (csrc/phi_table.h), as text."""
import os
import re
import struct

import numpy as np
import pytest

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


def test_table_keeps_relative_precision():
    # the polynomials as the kernels sum them (FP32 from t^5 on) against 50 digits.  Bound: 16 of FP64's
    # half-ulps; the interpolation takes 2.3e-16, the FP32 powers (z / 128)^5 / 5! 2^-24, 1.1e-15 at z = 10
    mp = pytest.importorskip("mpmath")
    _, words = _read()
    f64 = lambda w: struct.unpack("<d", struct.pack("<Q", w))[0]
    f32 = lambda w: [np.float32(v) for v in struct.unpack("<ff", struct.pack("<Q", w))]
    rng = np.random.default_rng(1)
    with mp.workdps(50):
        cdf = lambda z: mp.erfc(-z / mp.sqrt(2)) / 2
        exact = (lambda z: mp.exp(-z * z / 2) / mp.sqrt(2 * mp.pi) / cdf(z), lambda z: mp.log1p(cdf(z) - 1))
        for i in list(rng.integers(0, 641, 60)) + [0, 1, 63, 512, 639, 640]:
            row = words[14 * i:14 * i + 14]
            a7, a6 = f32(row[10])
            a5, b5 = f32(row[11])
            b7, b6 = f32(row[12])
            low = [f64(w) for w in row[:10]]
            polys = ([a7, a6, a5], low[:5]), ([b7, b6, b5], low[6:10] + [low[5]])
            for t in rng.uniform(-1 / 128, 1 / 128, 8):
                t = abs(t) if i == 0 else -abs(t) if i == 640 else t
                z = mp.mpf(int(i)) / 64 + mp.mpf(float(t))
                for (high, rest), fn in zip(polys, exact):
                    u = np.float32(0)
                    for c in high:
                        u = np.float32(np.float32(u * np.float32(t)) + c)
                    v = mp.mpf(float(u))
                    for c in rest:
                        v = mp.mpf(float(v * mp.mpf(float(t)) + mp.mpf(c)))
                    assert abs(v / fn(z) - 1) <= 16 * 2.0 ** -53, (i, t)
