"""Loads behind the wait of a programmatic dependent launch, looked up in the sources (no GPU).

A load through `const __restrict__`, or by __ldg / __ldcs / __ldcg, may be moved by the compiler in front of an asm statement that
only clobbers memory.  Every such load of the library therefore starts from a pointer whose value is taken behind the wait: a kernel
argument handed to pdl_wait(...), or a local one made by pdl_ptr(...).  A load moved in front of the wait would read what the
preceding kernel is still writing; that cannot be provoked, only ruled out.

Some kernels read in front of the wait on purpose what no kernel has written since the shards were loaded (or, for lists of sampled rows,
since an earlier kernel of the call has waited): AHEAD names it, kernel by kernel.  A kernel that waits in one of two places is looked at
both ways."""
import glob
import itertools
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_05203_b200", "csrc")
FILES = sorted(f for f in glob.glob(os.path.join(CSRC, "*")) if f.endswith((".cu", ".cuh", ".inc")))


# arguments that may be read in front of the wait (status: errors are recorded by an atomic operation at any time)
AHEAD = {"grad_wide_kernel": {"A", "y", "tiles", "gather", "row_off", "status"}}
AHEAD_SELECT = {"p.tile_begin", "p.row_off"}                    # tc_vector
STATE = r"p\.(?:x|g|gi)\b\s*(?:\[|\+)"                          # persistent kernels


def _clean(text):
    return re.sub(r"__launch_bounds__\([^)]*\)", "", re.sub(r"//[^\n]*", "", text))


def _source(path):
    return _clean(open(path).read())


def _both_ways(text):
    """The text as it runs with `early` set and not set; itself where there is no such choice."""
    choice = re.compile(r"if \(early\) \{([^{}]*)\} else \{([^{}]*)\}")
    alone = re.compile(r"if \(early\) (pdl_wait\([^)]*\);)")
    if not choice.search(text) and not alone.search(text):
        return {"": text}
    return {"early": alone.sub(r"\1", choice.sub(r"\1", text)), "first": alone.sub("", choice.sub(r"\2", text))}


def _kernel_at(text, at):
    names = [m.group(1) for m in re.finditer(r"__global__\s+void\s+(\w+)\s*\(", text) if m.start() < at]
    return names[-1] if names else ""


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
        if name in AHEAD.get(_kernel_at(text, at), ()):
            return True
        if any(re.search(r"\b%s\b" % name, args) for args in re.findall(r"pdl_wait\(([^)]*)\)", text[:at])):
            return True
        # the definition before the load; behind it where the load stands in a lambda defined in front of a loop
        made = [m for m in re.finditer(r"\b%s\s*=(?!=)\s*([^;]*);" % name, text) if m.group(1) != "nullptr"]
        made = [m for m in made if m.start() < at][-1:] or made[:1]
        if not made:
            return False
        expression, at = made[0].group(1), made[0].start()
    return False


def _misplaced_loads(text):
    loads = [(m.start(), _call_argument(text, m.end())) for m in re.finditer(r"\b__ld(?:g|cs|cg)\(", text)]
    locals_ = [(m.start(), m.group(1)) for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+\w+\s*=\s*([^;]*);", text)]
    return [e for at, e in loads + locals_ if not _behind_wait(e, text, at)]


def _unwaited_arguments(text):
    found = []
    for m in re.finditer(r"__global__\s+void\s+(\w+)\s*\(([^{;]*?)\)\s*\{", text):
        pointers = {re.search(r"(\w+)\s*$", q).group(1) for q in re.sub(r"/\*.*?\*/", "", m.group(2)).split(",") if "*" in q}
        body = text[m.end():]
        body = body[:(re.search(r"__global__\s+void", body) or re.search(r"$(?![\s\S])", body)).start()]
        wait = re.search(r"pdl_wait\(([^)]*)\)", body)
        ahead = AHEAD.get(m.group(1), set())
        if not wait or not pointers <= set(re.findall(r"\w+", wait.group(1))) | ahead or "pdl_ptr(" in body[:wait.start()]:
            found.append(m.group(1))
        elif any(re.search(r"(?<![\w.])%s\s*(?:\[|\))" % q, body[:wait.start()]) for q in pointers - ahead):        # plain loads
            found.append(m.group(1))
    return found


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_read_only_loads_start_behind_the_wait(path):
    for way, text in _both_ways(_source(path)).items():
        assert _misplaced_loads(text) == [], way


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_pointer_arguments_go_through_the_wait(path):
    for way, text in _both_ways(_source(path)).items():
        assert _unwaited_arguments(text) == [], way


def _early_state(text):
    """Ways through a persistent kernel on which the state is read in front of the wait."""
    text = re.sub(r"if \(\(int\)cluster\.num_blocks\(\).*?\n    \}\n", "", text, flags=re.S)          # a way out
    found = []
    for local, plus in itertools.product((0, 1), (0, 1)):
        ways, keep, flags = [], [True], {"PK_LOCAL": local, "PK_PLUS": plus, "PK_EF": 0, "PK_FLOOR": 0}
        for line in text.split("\n"):
            if re.match(r"#ifndef\b", line):
                keep.append(True)
            elif re.match(r"#if\b", line):
                keep.append(bool(eval(line[3:].replace("&&", " and ").replace("!", " not "), {}, flags)))
            elif re.match(r"#else\b", line):
                keep[-1] = not keep[-1]
            elif re.match(r"#endif\b", line):
                keep.pop()
            elif all(keep):
                ways.append(line)
        one = "\n".join(ways)
        for first in (False, True) if not local else (False,):
            way = one.replace("if (WAIT_FIRST) pdl_wait();", "pdl_wait();" if first else "").replace("if (!WAIT_FIRST) pdl_wait();", "" if first else "pdl_wait();")
            state, wait = re.search(STATE, way), re.search(r"\bpdl_wait\(\)", way)
            if not wait or not state or state.start() < wait.start():
                found.append((local, first))
    return sorted(set(found))


PERSISTENT = [f for f in FILES if os.path.basename(f) in ("persistent_body.inc", "persistent_roles.inc")]


@pytest.mark.parametrize("path", PERSISTENT, ids=[os.path.basename(f) for f in PERSISTENT])
def test_persistent_kernels_read_the_state_behind_the_wait(path):
    assert _early_state(_source(path)) == []


def _early_select(text):
    """What tc_vector reads through its arguments in front of the wait."""
    body = text[text.index("void tc_vector("):]
    late = body.index("if (!STREAM) { if (!LATE) pdl_trigger(); pdl_wait(); }")
    return {m for m in re.findall(r"(p\.\w+)\s*\[", body[:late])} - AHEAD_SELECT


def test_selection_reads_ahead_only_the_tables():
    assert _early_select(_source(os.path.join(CSRC, "topk_cluster.cuh"))) == set()


def _without(name, line, by=""):
    text = _source(os.path.join(CSRC, name))
    assert text.count(line) == 1, line
    return text.replace(line, by)


def test_a_missing_wait_is_noticed():
    """The checks themselves, on sources with a wait taken out or a load moved."""
    early = _both_ways(_without("grad.cuh", "if (early) pdl_wait(x, partial, loss_partial);"))
    assert "grad_wide_kernel" in _unwaited_arguments(early["early"])
    early = _both_ways(_without("grad.cuh", "if (early) pdl_wait(x, partial, loss_partial);", "if (early) pdl_wait(partial, loss_partial);"))
    assert "grad_wide_kernel" in _unwaited_arguments(early["early"]) and "grad_wide_kernel" not in _unwaited_arguments(early["first"])
    first = _both_ways(_without("grad.cuh", "pdl_wait(A, y, x, tiles, partial, loss_partial, gather, row_off, status);\n        pdl_trigger();", "pdl_trigger();"))
    assert "grad_wide_kernel" in _unwaited_arguments(first["first"])
    moved = _without("grad.cuh", "const RowTile t = tiles[blockIdx.x];\n    const int chunks = ld >> 2, stages", "float4 xr0 = reinterpret_cast<const float4*>(x)[0];\n    const int chunks = ld >> 2, stages")
    assert "grad_wide_kernel" in _unwaited_arguments(_both_ways(moved)["early"])
    for name in ("persistent_body.inc", "persistent_roles.inc"):
        assert _early_state(_without(name, "    if (WAIT_FIRST) pdl_wait();\n")) == [(0, True)]
        assert (0, False) in _early_state(re.sub(r"(?m)^    if \(!WAIT_FIRST\) pdl_wait\(\);\n", "", _source(os.path.join(CSRC, name))))
        assert (1, False) in _early_state(_without(name, "        pdl_wait();\n        for (int j = tid;", "        for (int j = tid;"))
    assert _early_select(_without("topk_cluster.cuh", "if (LATE) tables();", "if (LATE) tables(); const float b0 = p.b[0];")) == {"p.b"}
