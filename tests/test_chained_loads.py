"""Chained kernels (chain_wait) may run while the kernel before them still
writes: the read-only load path, which wants data that nobody writes during the
kernel's lifetime, must not appear in them or in anything they call."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_05086_gb300", "csrc")
READ_ONLY = re.compile(r"\b__ldg\s*\(|\bld_row16\s*\(|ld\.global\.nc")


def functions(text):
    """Name -> body of every device function and kernel."""
    out = {}
    text = re.sub(r"//[^\n]*|__launch_bounds__\([^)]*\)", "", text)
    for m in re.finditer(r"__(?:device|global)__[^;{}]*?\b(\w+)\s*\([^;{}]*?\)\s*(?:const\s*)?\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        out[m.group(1)] = text[m.end():i]
    return out


def reached(fns, start):
    todo, seen = [start], set()
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        todo += [g for g in re.findall(r"\b(\w+)\s*(?:<[^;{}()]*>)?\s*\(", fns[f]) if g in fns]
    return seen


@pytest.mark.parametrize("source", ["learned.cu", "kernels.cu"])
def test_no_read_only_loads_in_chained_kernels(source):
    with open(os.path.join(CSRC, source)) as f:
        fns = functions(f.read())
    chained = [f for f, body in fns.items() if re.search(r"\bchain_wait\s*\(\)", body)]
    assert chained, "no chained kernel found"
    for kernel in chained:
        for f in sorted(reached(fns, kernel)):
            assert not READ_ONLY.search(fns[f]), f"{source}: {f}, reached from {kernel}"
