"""Kernels that may be resident while an earlier kernel of the same call still writes (programmatic
dependent launch) must read what that kernel writes with ordinary loads: a read-only load promises
data that is constant for the kernel's lifetime, and may be moved above the wait.  No GPU needed: the
sources are looked through."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2406_17660_b200", "csrc")


def _kernels():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__", text):
            start = text.index("{", m.end())
            depth, at = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            head = re.sub(r"__launch_bounds__\([^)]*\)", "", text[m.end():start])
            yield f"{name}:{re.search(r'(\w+)\s*\(', head).group(1)}", text[m.end():at]


WAITING = [(k, body) for k, body in _kernels() if "grid_dep_wait()" in body]


def test_the_kernels_are_found():
    names = {k.split(":")[1] for k, _ in WAITING}
    assert {"project_tc_kernel", "gather_cols_kernel", "splitk_reduce_kernel", "splitk_rownorms_kernel",
            "norms_finalize_kernel", "select_kernel", "select_rank_kernel",
            "adam_apply_wide_kernel"} <= names


@pytest.mark.parametrize("kernel,body", WAITING, ids=[k for k, _ in WAITING])
def test_no_read_only_loads_after_a_wait(kernel, body):
    assert "__ldg" not in body and "__restrict__" not in body, kernel


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                yield name, re.sub(r"//[^\n]*", "", f.read())


ORDINARY = {k for _, text in _sources() for k in re.findall(r"(\w+)(?:<[^<>;]*>)?<<<", text)}
DEPENDENT = [(k, body) for k, body in _kernels() if k.split(":")[1] not in ORDINARY]
# pointers in the structs that kernels take: {struct: its pointer members}
STRUCTS = {s: set(re.findall(r"\*\s*(\w+)(?:\[\w+\])?[,;]", members) + re.findall(r"\*\s*\w+,\s*\*(\w+)", members))
           for _, text in _sources() for s, members in re.findall(r"struct (\w+) \{(.*?)\n\};", text, re.S)}


def _before_the_wait(body):
    """A kernel's parameters, and its text up to the first wait that every thread comes to, or None."""
    start = body.index("{")
    for m in re.finditer(r"(?:^|[;{}])\s*(grid_dep_wait\(\);)", body):
        before = body[start + 1:m.start(1)]
        if before.count("{") == before.count("}"):
            return body[:start], before
    return None


def test_the_ordinary_launches_are_found():
    assert ORDINARY == {"adam_vec4_kernel", "adam_scalar_kernel", "scatter_kernel", "scatter_cols_kernel",
                        "bounded_wait_kernel"}
    assert {"dY", "idx", "out", "rho", "status"} <= STRUCTS["TcParams"] and "W" in STRUCTS["UpdateGroup"]
    assert {"norms", "idx", "rho", "status"} <= STRUCTS["SelectArgs"]


@pytest.mark.parametrize("kernel,body", DEPENDENT, ids=[k for k, _ in DEPENDENT])
def test_every_dependent_kernel_waits_before_it_reads_or_writes(kernel, body):
    """What the wait makes visible is what the grids before it wrote; reads ahead of it, also of what the program's
    kernel before the call wrote, have no such promise."""
    found = _before_the_wait(body)
    assert found is not None, f"{kernel} has threads that do not wait"
    head, before = found
    before = re.sub(r"[\w.]+ [!=]= nullptr", "", before)              # whether there is one, not what it points at
    used = [p for p in re.findall(r"\*\s*(\w+)\s*[,)]", head) if re.search(rf"\b{p}\b", before)]
    for struct, param in re.findall(r"(\w+)\s*&?\s+(\w+)\s*[,)]", head):
        used += [f"{param}.{m}" for m in STRUCTS.get(struct, ()) if re.search(rf"\b{param}\.{m}\b", before)]
    assert not used, (kernel, used)


@pytest.mark.parametrize("name,text", list(_sources()), ids=[n for n, _ in _sources()])
def test_no_read_only_loads_but_in_ordinary_launches(name, text):
    """Device functions and inline assembly too."""
    if name in ("adam.cu", "scatter.cu"):           # launched the ordinary way
        return
    assert not re.search(r"__ldg|__restrict__|\.nc\b", text)
