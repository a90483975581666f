"""Kernels launched as programmatic dependents, in the source: each waits, or
joins the kernel that it runs beside, before it touches memory or lets the next
one start, and one that joins also waits before it ends."""
import os
import re

import pytest

from paper_2003_11468_gb300 import build


def _sources():
    for name in sorted(os.listdir(build.CSRC)):
        if name.endswith(".cu"):
            with open(os.path.join(build.CSRC, name)) as f:
                yield re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _body(text, at):
    depth, start = 0, text.index("{", at)
    for k in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[start + 1:k]
    raise AssertionError("unbalanced braces")


def _kernels():
    for text in _sources():
        for m in re.finditer(r"__global__", text):
            head = text[m.end():text.index("{", m.end())]
            name = re.findall(r"\b(k_\w+)\s*\(", head)[0]
            plain = re.search(name + r"(<[^;{}]*?>)?<<<", text) is not None
            yield name, plain, _body(text, m.end())


KERNELS = {name: (plain, body) for name, plain, body in _kernels()}
DEPENDENT = sorted(name for name, (plain, _) in KERNELS.items() if not plain)


def test_kernels_are_found():
    assert {"k_scan", "k_link", "k_brick_sort", "k_dense_self", "k_dense_pairs", "k_finalize"} <= set(DEPENDENT)
    assert {n for n, (plain, _) in KERNELS.items() if plain} == {"k_bin_count", "k_bin_count_tile", "k_relink_check"}


@pytest.mark.parametrize("name", DEPENDENT)
def test_waits_before_it_reads(name):
    body = KERNELS[name][1]
    first = re.search(r"pdl_(wait|join)\(", body)
    assert first, name
    before = body[:first.start()]
    assert "pdl_trigger" not in before and "pdl_pass_on" not in before
    # declarations of shared memory and the choice between the two calls only
    before = re.sub(r"(extern )?__shared__[^;]*;", "", before)
    choice = re.fullmatch(r"\s*(if \((beside|kLo == 0)\)\s*\{?\s*)?", before)
    assert choice, before
    if choice.group(1):                       # a choice of the two calls, never of none
        assert re.match(r"[^;{}]*;[^{}]*?\}?\s*else\s*\{?\s*pdl_(wait|join)\(", body[first.start():])
    calls = re.findall(r"pdl_(wait|join)\(", body)
    if "join" in calls:                       # and completes after the kernel it ran beside
        assert calls[-1] == "wait" and re.search(r"(if \([^;{}]*\)\s*)?pdl_wait\(\);\s*$", body)
