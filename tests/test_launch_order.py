"""Every kernel waits for its predecessor before it touches memory (kernels are launched with
programmatic dependence): the wait is the first statement, and every pointer argument goes
through it, since a `const T* __restrict__` argument lets a compiler move loads over an
ordinary memory clobber."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0710_3612_gb300", "csrc")


def _strip(src):
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


def _close(s, i, pair):
    """Index of the bracket that closes the one at i."""
    depth = 0
    for k in range(i, len(s)):
        depth += (s[k] == pair[0]) - (s[k] == pair[1])
        if depth == 0:
            return k
    raise AssertionError("unbalanced brackets")


def _split(params):
    out, depth, cur = [], 0, ""
    for ch in params:
        depth += (ch in "<(") - (ch in ">)")
        if ch == "," and depth == 0:
            out.append(cur)
            cur = ""
        else:
            cur += ch
    return [p.strip() for p in out + [cur]]


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = _strip(open(path).read())
        for m in re.finditer(r"__global__\s+void\b", src):
            i = m.end()
            b = re.compile(r"\s*__launch_bounds__\s*\(").match(src, i)
            if b:
                i = _close(src, b.end() - 1, "()") + 1
            name = re.compile(r"\s*(\w+)\s*\(").match(src, i)
            end = _close(src, name.end() - 1, "()")
            body = src[src.index("{", end) + 1:].lstrip()
            params = _split(src[name.end():end])
            if params[-1] != "int dependent":                # launched plainly, after whole kernels
                assert re.search(r"\b%s\s*<<<" % name[1], src) and "launch_after(" + name[1] not in src
                continue
            yield pytest.param(params, body, id=os.path.basename(path)[:-3] + "-" + name[1])


KERNELS = list(_kernels())


def test_kernels_are_found():
    assert len(KERNELS) > 60


@pytest.mark.parametrize("params,body", KERNELS)
def test_wait_comes_first_and_orders_every_pointer(params, body):
    m = re.match(r"pdl_wait\(([^;]*)\);", body)
    assert m, body[:60]
    pointers = [re.search(r"(\w+)$", p)[1] for p in params if "*" in p]
    assert [a.strip() for a in m[1].split(",")] == ["dependent"] + pointers
