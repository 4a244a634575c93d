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
