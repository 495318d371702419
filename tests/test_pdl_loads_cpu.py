"""Kernels that wait for the kernel before them (griddepcontrol.wait) start while that kernel still
writes.  The non-coherent load path wants memory that nobody writes while the kernel runs, so in
such a kernel only data that is complete before a call's first step may take it: W, the sponge
tables, the receiver map and the tap tables.  A wrong load shows in no result as long as the
compiler happens to leave it behind the wait, hence this check of the sources.  (The cache-hint
intrinsics are not volatile either, so they may move above the wait too.)"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1912_08063_gb300", "csrc")
CONSTANT = re.compile(r"\b(W|Wp|sig_[xyz]|s[xyz]|rec_map|pts)\b")


def _without_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _closing(text, i, pair):
    depth = 0
    for k in range(i, len(text)):
        depth += (text[k] == pair[0]) - (text[k] == pair[1])
        if depth == 0:
            return k
    raise AssertionError("unbalanced source")


def kernels(text):
    """(parameters, body) of every kernel defined in a source file."""
    for m in re.finditer(r"__global__", text):
        name = re.compile(r"\b(k_\w+)\s*\(").search(text, m.end())
        end = _closing(text, name.end() - 1, "()")
        b = text.index("{", end)
        yield text[name.end():end], text[b:_closing(text, b, "{}")]


def violations(text):
    text = _without_comments(text)
    bad, waits = [], False
    for params, body in kernels(text):
        if "pdl_wait()" not in body:
            continue
        waits = True
        for d in re.findall(r"[^,;{}()]*__restrict__[^,;=)]*", params + ";" + body):
            if not CONSTANT.search(d.split("__restrict__")[1]):
                bad.append(" ".join(d.split()))
    if waits:   # the file's device functions serve its waiting kernels too
        for m in re.finditer(r"__ld(?:g|ca|cg|cs|lu)\(", text):
            arg = text[m.end():_closing(text, m.end() - 1, "()")]
            if not CONSTANT.search(arg):
                bad.append(m.group() + " ".join(arg.split()) + ")")
    return bad


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_waiting_kernels_read_written_data_plainly(name):
    with open(os.path.join(CSRC, name)) as f:
        assert violations(f.read()) == []


def test_the_check_finds_both_forms():
    src = """__global__ void k_a(const float *__restrict__ W, const float *__restrict__ f, float *o)
    { pdl_wait(); o[0] = f[0] * W[0] + __ldg(o + 1) + __ldg(W + 2) + __ldcg(o + 3); }
    __global__ void k_b(const float *__restrict__ f, float *o) { o[0] = f[0]; }"""
    assert violations(src) == ["const float *__restrict__ f", "__ldg(o + 1)", "__ldcg(o + 3)"]
