"""Kernels that start under programmatic dependent launch are up before the launch before them has
finished: CUDA's read-only path (__ldg, ld.global.nc, const __restrict__ parameters) is for memory that
nobody writes while a kernel is up, so such a kernel reads through plain loads only, after its wait.
Checked on the sources: the order of the loads that it allows is not something a run can show."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1111_0905_gb300" / "csrc"
WAIT = "wait_for_predecessor();"
READ_ONLY = re.compile(r"__ldg|\.nc\b|__restrict__|ld_here|Store<S>::ld\b|g_wall_fix|loc_ref<|[^_]pull<")


def _code(name):
    text = (CSRC / name).read_text()
    text = re.sub(r"//[^\n]*", "", text)
    return re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", text)


def _functions(code):
    """(name, signature and body) of the functions at namespace level."""
    for m in re.finditer(r"\b(\w+)\(([^;{}()]*(?:\([^()]*\)[^;{}()]*)*)\)\s*\{", code):
        depth, i = 1, m.end()
        while depth and i < len(code):
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        yield m.group(1), m.group(0) + code[m.end():i]


@pytest.mark.parametrize("name", ["lb_split.cuh", "lb_adjoint.cu"])
def test_dependent_kernels_read_through_plain_loads(name):
    functions = dict(_functions(_code(name)))
    kernels = [k for k, text in functions.items() if WAIT in text]
    assert kernels
    todo, seen = list(kernels), set()
    while todo:
        k = todo.pop()
        if k in seen:
            continue
        seen.add(k)
        found = READ_ONLY.search(functions[k])
        assert not found, (name, k, found.group(0))
        todo += [f for f in functions if f not in seen and re.search(rf"\b{f}\b", functions[k])]


def test_every_dependent_launch_waits_first():
    """Each kernel that follow() launches calls the wait, before any access through its arguments."""
    launched = set()
    for name in ("lb_launch.cuh", "lb_adjoint.cu"):
        launched |= set(re.findall(r"follow\(\s*(\w+_kernel)", _code(name)))
    bodies = dict(_functions(_code("lb_split.cuh"))) | dict(_functions(_code("lb_adjoint.cu")))
    assert launched
    for k in launched:
        head = bodies[k].split("{", 1)[1]
        assert WAIT in head, k
        assert not re.search(r"\bld_at\b|\bst_at\b|\b[AML]\w*\[|adj_pull|split_pull", head.split(WAIT)[0]), k
