"""The logarithm's table: its entries are read as 16-byte words, so their type is
16-byte aligned (checked by the compiler), and they are what their comment says."""
import math
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1703_02920_gb300", "csrc")


def test_entries_are_aligned_for_their_loads(tmp_path):
    from paper_1703_02920_gb300 import build
    src = tmp_path / "align.cu"
    src.write_text('#include "logratio.cuh"\n'
                   'static_assert(alignof(msk::LogEntry) == sizeof(double2), "16-byte loads");\n'
                   'static_assert(sizeof(msk::LogEntry) == sizeof(double2), "two doubles");\n')
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", CSRC, "-c", str(src), "-o",
                        str(tmp_path / "align.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_entries():
    text = open(os.path.join(CSRC, "logratio.cuh")).read()
    rows = re.findall(r"\{(-?[0-9.e-]+), (-?[0-9.e-]+)\}", text)
    assert len(rows) == 93
    for i, (r, l) in enumerate(rows, 90):
        r, l = float(r), float(l)
        assert abs(r * i / 128 - 1) < 2.0 ** -23
        m, _ = math.frexp(r)
        assert m * 2.0 ** 24 == int(m * 2.0 ** 24)  # 24 bits: z = m r - 1 rounds once
        assert abs(l + math.log(r)) <= 2.0 ** -54
