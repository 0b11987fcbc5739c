"""The stats kernel screens FP64 cells for the band 1e-6 < phi < 1 - 1e-6 by the
upper words of its limits (hex literals in stats.cu)."""
import os
import re
import struct

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_upper_words_are_the_limits():
    src = open(os.path.join(ROOT, "paper_1910_05180_gb300", "csrc", "stats.cu")).read()
    m = re.search(r"kBandLo = (0x[0-9a-f]+)u, kBandHi = (0x[0-9a-f]+)u;", src)
    for text, limit in zip(m.groups(), (1e-6, 1.0 - 1e-6)):
        assert int(text, 16) == struct.unpack(">Q", struct.pack(">d", limit))[0] >> 32
