"""Kernels that are launched early (programmatic dependent launch) must not read what the kernel before them writes until
grid_dep_wait() has returned.  A read-only load (__ldg, const __restrict__) carries no dependence the compiler would have to
keep behind that wait, so every pointer that is read that way has to come out of dep() after it; this looks at the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_00130_b200", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def body(text, at):
    """The braces from the first '{' at or after `at`."""
    i = text.index("{", at)
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
        j += 1


def early_kernels(text):
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\s*\(", text):
        depth, j = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[j], 0)
            j += 1
        code = body(text, j)
        if "grid_dep_wait()" in code:
            yield m.group(1), text[m.end():j - 1], code.split("grid_dep_wait();", 1)[1]


def loads(code):
    """Names at the root of the arguments of __ldg."""
    for m in re.finditer(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\(\s*)?([A-Za-z_][\w.]*)", code):
        yield m.group(1)


@pytest.mark.parametrize("name", FILES)
def test_read_only_loads_go_through_dep(name):
    text = open(os.path.join(CSRC, name)).read()
    for kernel, params, code in early_kernels(text):
        structs = re.findall(r"(?:const\s+)?(?:__grid_constant__\s+)?const\s+([A-Z]\w*)\s*&?\s*(\w+)", params)
        for _, p in structs:
            assert not [x for x in loads(code) if x.startswith(p + ".")], (kernel, "reads a parameter's pointer directly")
            # a parameter's epilogue operands are handed on only as a copy made after the wait
            assert not re.search(r"(?<!after_wait\()\b%s\.e\b(?!\.(?:M|N)\b)" % p, code), (kernel, "hands on " + p + ".e")
            for field in ("bias", "dsig", "cin"):
                for m in re.finditer(r"\b%s\.%s\b(?!_)" % (p, field), code):
                    line = code[code.rfind("\n", 0, m.start()):code.find("\n", m.end())]
                    assert "dep(" in line or re.search(r"\b%s\.%s \?" % (p, field), line), (kernel, line)
        for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params):
            assert re.search(r"\b%s = dep\(%s\)" % (p, p), code), (kernel, p)


def test_the_sources_are_seen():
    assert sum(len(list(early_kernels(open(os.path.join(CSRC, f)).read()))) for f in FILES) >= 20
