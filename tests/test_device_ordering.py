"""Sweeps launched as programmatic dependents become resident while the kernel
before them still writes the vectors they read.  What orders their reads is
griddepcontrol.wait, so a read of a vector must not be movable across it: the
compiler may move a non-volatile asm statement without a memory clobber, and
an .nc load (or one through a const __restrict__ pointer) tells it that the
data does not change while the kernel runs.  Read from the sources (no GPU
needed): only the matrix, which no kernel in flight writes, is read that way."""
import os
import re

import pytest

from paper_2111_09512_gb300 import _build

MATRIX_LOADS = {"ld_pair", "ld_one", "pair", "one"}  # values and columns of slices.cuh
FUNCTION = re.compile(r"__device__ __forceinline__ [\w\s]*?(\w+)\(")


def source(name):
    with open(os.path.join(_build.CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def waiting_units():
    return sorted(f for f in os.listdir(_build.CSRC)
                  if f.endswith((".cu", ".cuh")) and "grid_wait_prior();" in source(f))


def asm_loads(text):
    """(function, statement) of every inline load from global memory."""
    for m in re.finditer(r"\basm\b.*?\);", text, re.S):
        if re.search(r'"[^"]*\bld\.(relaxed\.\w+\.|acquire\.\w+\.)?global', m.group(0)):
            names = FUNCTION.findall(text, 0, m.start())
            yield (names[-1] if names else ""), m.group(0)


def test_vector_loads_stay_behind_the_wait():
    seen = set()
    for unit in ["sweep_ptx.cuh", *waiting_units()]:
        for function, statement in asm_loads(source(unit)):
            if function in MATRIX_LOADS:
                continue
            seen.add(function)
            assert re.match(r"asm\s+volatile", statement), (unit, function, statement)
            assert '"memory"' in statement and ".nc" not in statement, (unit, function, statement)
    assert {"ld_keep", "ld_cols"} <= seen


@pytest.mark.parametrize("unit", waiting_units())
def test_vectors_of_waiting_kernels_are_not_declared_constant(unit):
    text = source(unit)
    kernels = re.findall(r"__global__ void.*?\)\s*\{.*?\n\}\n", text, re.S)
    waiting = [k for k in kernels if "grid_wait_prior();" in k]
    assert waiting
    for k in waiting:
        head = k[:k.index("{")]
        for vector in ("c", "in"):
            assert not re.search(r"__restrict__\s+%s\b" % vector, head), head
