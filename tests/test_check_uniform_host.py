"""A WO_CHECK build's index check that leaves a kernel (``return``) must be one
decision for the whole block: a thread that left before the others' block
barriers and full-mask shuffles would make those undefined.  Read from the
sources: no such check may test a value that depends on the thread."""
import glob
import os
import re

import pytest

from paper_2412_09775_gb300.build import CSRC

NAME = re.compile(r"(?<![.\w])\w+")  # not a member: blockIdx.y is not the variable y
BLOCK = re.compile(r"#if defined\(WO_CHECK\) && WO_CHECK\n(.*?)#endif", re.S)


def thread_dependent(code):
    """The names assigned, directly or not, from the thread index."""
    pairs = [(n, e) for stmt in re.split(r"[;{}]", code)
             for n, e in re.findall(r"(\w+)\s*=(?!=)\s*((?:[^,()]|\((?:[^()]|\([^()]*\))*\))*)", stmt)]
    tainted = {"threadIdx"}
    while True:
        more = {n for n, e in pairs if set(NAME.findall(e)) & tainted} - tainted
        if not more:
            return tainted
        tainted |= more


def leaving_checks():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in BLOCK.finditer(src):
            if "return" in m.group(1) and "WO_IN" in m.group(1):
                body = src[src.rindex("__global__", 0, m.start()):m.start()] + m.group(1)
                line = src[:m.start()].count("\n") + 1
                yield pytest.param(body, m.group(1), id=f"{os.path.basename(path)}:{line}")


def test_the_reader_follows_assignments():
    t = thread_dependent("int l = threadIdx.x % T, c = b * 2; long long g = f(l, (3 + c)); x0 = blockIdx.x;")
    assert t == {"threadIdx", "l", "g"}


@pytest.mark.parametrize("body,check", list(leaving_checks()))
def test_leaving_checks_are_uniform(body, check):
    assert not thread_dependent(body) & set(NAME.findall(check))
