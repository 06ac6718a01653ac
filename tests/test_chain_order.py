"""Chained steps read populations only after the wait for the step before them.

A kernel launched as a programmatic dependent is resident while its input is still being written, so
its loads of populations must not go through the read-only path (.nc, __ldg) and must be ordered
behind griddepcontrol.wait: volatile statements with a memory clobber, issued after it. Read off the
sources here, since a build that breaks this may still give the right bits.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1202_6074_gb300", "csrc")


def text(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def body(src, start):
    """The braces' contents that open at or after position start."""
    i = src.index("{", start)
    depth, j = 0, i
    while True:
        depth += (src[j] == "{") - (src[j] == "}")
        if depth == 0:
            return src[i + 1:j]
        j += 1


def functions(src, pattern):
    return [body(src, m.end()) for m in re.finditer(pattern, src)]


def ordered(statement):
    return statement.startswith("asm volatile(") and '"memory"' in statement and ".nc" not in statement


def test_the_wait_and_the_loads_behind_it_are_ordered_statements():
    loads = functions(text("cm_core.cuh"), r"\bld_stream\(const [\w ]+\* p\) ")
    assert len(loads) == 5
    for f in loads:
        chained = re.search(r"if constexpr \(CHAINED\) (asm[^;]*\];[^;]*;)", f)
        assert chained and ordered(chained.group(1)), f
    for name, pattern in (("cm_core.cuh", r"\bvoid chain_wait\(\) "), ("cm_async.cuh", r"\bvoid copy_async16\([^)]*\) ")):
        (f,) = functions(text(name), pattern)
        assert len(re.findall(r"\basm\b", f)) == 1 and ordered(f.strip()), f


@pytest.mark.parametrize("name", ["cm_kernels.cuh", "cm_pair.cuh", "cm_async.cuh"])
def test_kernels_of_a_chain_read_populations_after_the_wait(name):
    src = text(name)
    kernels = [f for f in functions(src, r"__global__ void") if "chain_begin()" in f]
    assert len(kernels) == 1
    for f in kernels:
        assert f.count("chain_wait()") == 1
        before, after = f.split("chain_wait()")
        lambdas = [body(before, m.end()) for m in re.finditer(r"auto \w+ = \[&\]\([^)]*\)", before)]
        for b in lambdas:                     # defined before the wait, called after it
            before = before.replace(b, "")
        for read in ("gather", "stage(", "copy_async16", "load_force", "__ldg", "ld(", "ld2("):
            uses = [u for u in re.findall(r"[\w]*" + re.escape(read) + r"[^;]*", before) if not u.startswith("auto")]
            assert not uses, uses
        # nothing of the source state is read but by the gathers and the staged copies
        assert not re.search(r"__ldg\([^;]*\bsrc\b|\*\s*\(?src\b|\bsrc\[", f)


def test_the_pulls_of_chained_kernels_use_the_ordered_loads():
    pair = text("cm_pair.cuh")
    assert not re.search(r"::(template )?ld2?(<false>)?\(", pair)
    assert len(re.findall(r"::template ld2?<true>\(", pair)) >= 10
    one = functions(text("cm_core.cuh"), r"void gather_impl\(")[0]
    assert "constexpr bool CHAINED = PULL == kPullStored;" in one
    assert len(re.findall(r"Codec<S>::\S* ?ld2?\S*\(", one)) == len(re.findall(r"Codec<S>::template ld<CHAINED>\(", one)) == 2
    step = [f for f in functions(text("cm_kernels.cuh"), r"__global__ void") if "chain_begin()" in f][0]
    assert re.findall(r"\bgather<[^;]*", step) == ["gather<D, S, FT::WALLS, FT::BIG, kPullStored>(src, x, y, z, p, h)"]
