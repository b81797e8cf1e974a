"""Every device helper of the shared headers has a caller."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_02920_gb300", "csrc")


def test_shared_helpers_have_callers():
    text = {f: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
            for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h"))}
    whole = "\n".join(text.values())
    for header in ("common.cuh", "reduce.cuh", "logratio.cuh"):
        names = re.findall(r"__device__[^;{(]*?\b(\w+)\s*\([^;{]*\)\s*\{", text[header])
        assert names
        for name in set(names):
            assert len(re.findall(rf"\b{name}\b", whole)) > names.count(name), (header, name)
