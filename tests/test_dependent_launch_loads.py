"""Read-only loads behind the wait of a programmatic dependent launch, looked up in the sources (no GPU).

A load through `const __restrict__`, or by __ldg / __ldcs / __ldcg, may be moved by the compiler in front of an asm statement that
only clobbers memory.  Every such load of the library therefore starts from a pointer whose value is taken behind the wait: a kernel
argument handed to pdl_wait(...), or a local one made by pdl_ptr(...).  A load moved in front of the wait would read what the
preceding kernel is still writing; that cannot be provoked, only ruled out."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_05203_b200", "csrc")
FILES = sorted(f for f in glob.glob(os.path.join(CSRC, "*")) if f.endswith((".cu", ".cuh", ".inc")))


def _source(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    return re.sub(r"__launch_bounds__\([^)]*\)", "", text)


def _call_argument(text, at):
    depth, end = 1, at
    while depth:
        depth += {"(": 1, ")": -1}.get(text[end], 0)
        end += 1
    return text[at:end - 1]


def _behind_wait(expression, text, at):
    """Whether the pointer that `expression`, at position `at`, starts from takes its value behind the wait."""
    for _ in range(6):
        if "pdl_ptr(" in expression:
            return True
        # the first name that is neither a cast nor the condition of a choice
        expression = re.sub(r"\b\w+_cast<[^>]*>|^[^?]*\?\s*(?:nullptr\s*:)?", "", expression)
        first = re.search(r"([A-Za-z_]\w*)\s*(\.?)", expression)
        if first is None or first.group(2) == ".":                  # straight from a struct of arguments
            return False
        name = first.group(1)
        if any(re.search(r"\b%s\b" % name, args) for args in re.findall(r"pdl_wait\(([^)]*)\)", text[:at])):
            return True
        # the definition before the load; behind it where the load stands in a lambda defined in front of a loop
        made = [m for m in re.finditer(r"\b%s\s*=(?!=)\s*([^;]*);" % name, text) if m.group(1) != "nullptr"]
        made = [m for m in made if m.start() < at][-1:] or made[:1]
        if not made:
            return False
        expression, at = made[0].group(1), made[0].start()
    return False


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_read_only_loads_start_behind_the_wait(path):
    text = _source(path)
    loads = [(m.start(), _call_argument(text, m.end())) for m in re.finditer(r"\b__ld(?:g|cs|cg)\(", text)]
    locals_ = [(m.start(), m.group(1)) for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+\w+\s*=\s*([^;]*);", text)]
    assert [e for at, e in loads + locals_ if not _behind_wait(e, text, at)] == []


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_pointer_arguments_go_through_the_wait(path):
    text = _source(path)
    for m in re.finditer(r"__global__\s+void\s+(\w+)\s*\(([^{;]*?)\)\s*\{", text):
        pointers = {re.search(r"(\w+)\s*$", q).group(1) for q in re.sub(r"/\*.*?\*/", "", m.group(2)).split(",") if "*" in q}
        wait = re.search(r"pdl_wait\(([^)]*)\)", text[m.end():])
        assert wait and pointers <= set(re.findall(r"\w+", wait.group(1))), m.group(1)
        assert "pdl_ptr(" not in text[m.end():m.end() + wait.start()], m.group(1)
