"""Chained kernels read with ordinary loads (source check, no GPU).

A kernel started by launch_chained is resident while its predecessor still
writes the memory it will read, so that memory is not read-only for the
kernel's lifetime, which the non-coherent path (__ldg, `const T* __restrict__`
parameters) promises.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1010_4135_gb300", "csrc")
FILES = sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh")))
NON_COHERENT = re.compile(r"__ldg\s*\(|const\s+[\w<>:]+\s*\*\s*__restrict__|ld\.global\.nc")


def _functions(text):
    """(declaration, body) of every function at namespace level, comments removed."""
    text = re.sub(r"//[^\n]*", "", text)
    for head in re.finditer(r"__(?:global|device)__", text):
        brace = text.find("{", head.end())
        end = text.find(";", head.end())
        if brace < 0 or (0 <= end < brace):
            continue
        depth, k = 0, brace
        while True:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
            if depth == 0:
                break
        yield text[head.start():brace], text[brace:k]


def test_the_chained_kernels_are_found():
    names = {re.search(r"(\w+)\s*\($", decl[:decl.rindex("(") + 1] if "(" in decl else "").group(1)
             for n in FILES for decl, body in _functions(open(os.path.join(CSRC, n)).read())
             if "__global__" in decl and "chain_wait()" in body}
    assert {"fill_kernel", "step_fp64_kernel", "step_fp64_pairs_kernel", "step_pair_kernel",
            "step_pair_batch_kernel"} <= names


@pytest.mark.parametrize("name", FILES)
def test_no_non_coherent_loads_in_chained_kernels(name):
    funcs = list(_functions(open(os.path.join(CSRC, name)).read()))
    bodies = {}
    for decl, body in funcs:
        m = re.findall(r"(\w+)\s*\(", decl)
        if m:  # not an operator
            bodies.setdefault(m[-1], []).append((decl, body))
    todo = [(d, b) for d, b in funcs if "__global__" in d and "chain_wait()" in b]
    seen = set()
    while todo:  # the kernels and what they call in this file
        decl, body = todo.pop()
        assert not NON_COHERENT.search(decl + body), decl
        for callee in set(re.findall(r"(\w+)\s*(?:<[^;(){}]*>)?\s*\(", body)) & set(bodies) - seen:
            seen.add(callee)
            todo += bodies[callee]
