"""Chained kernels (those that call chain_wait) are resident while the kernels
before them on the stream still write, so only what a context uploads once is
read-only during their life.  In the sources: a chained kernel's const
__restrict__ parameters and every __ldg are of such data."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_02920_gb300", "csrc")
# work lists, offsets and weight sums: uploaded once per context
CONSTANT = {"tiles", "units", "cta_unit_off", "cb_unit_off", "wsum"}


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, name)).read()
            yield name, re.sub(r"//[^\n]*", "", text)


def _body(text, start):
    """From the opening brace at or after start to its closing one."""
    i = text.index("{", start)
    depth = 0
    for k in range(i, len(text)):
        depth += (text[k] == "{") - (text[k] == "}")
        if depth == 0:
            return text[i:k + 1]
    raise AssertionError("unbalanced braces")


def _kernels():
    for name, text in _sources():
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
            end = text.index(")", m.end())
            yield name, m.group(1), text[m.end():end], _body(text, end)


def test_chained_kernels_promise_no_read_only_chain_data():
    chained = 0
    for name, kernel, params, body in _kernels():
        if "chain_wait()" not in body:
            continue
        chained += 1
        for p in params.split(","):
            if "const" in p.split() and "__restrict__" in p:
                assert p.split()[-1] in CONSTANT, (name, kernel, p.strip())
    assert chained >= 15


def test_ldg_only_of_constant_tables():
    for name, text in _sources():
        assert name == "logratio.cuh" or "__ldg(" not in text, name


def test_device_helpers_take_plain_pointers():
    for name, text in _sources():
        for m in re.finditer(r"__device__[^;{(]*\b(\w+)\s*\(([^)]*)\)", text):
            assert not re.search(r"const \w+\* __restrict__", m.group(2)), (name, m.group(1))
