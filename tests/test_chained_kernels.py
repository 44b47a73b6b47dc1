"""Chained kernels (launch_chained in pt_common.cuh) by their source: the first statement of each waits for the
work before it, and no pointer that it or a function it calls takes is __restrict__ (a load through one could
move above the wait)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2207_08716_gb300", "csrc")


def _functions():
    """{(file, name): (signature, body)} of the device functions and kernels; overloads are concatenated."""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, f)).read(), flags=re.S)
        for m in re.finditer(r"__(?:global|device)__[^;{}]*?\b(\w+)\s*\(", re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)",
                                                                               lambda b: " " * len(b.group()), text)):
            at = text.index("(", m.end(1))
            level = 0
            for depth in range(at, len(text)):
                level += {"(": 1, ")": -1}.get(text[depth], 0)
                if level == 0:
                    break
            end = depth + 1
            if not re.match(r"\s*\{", text[end:]):
                continue                                       # a declaration
            i = text.index("{", end)
            level, j = 0, i
            for j in range(i, len(text)):
                level += {"{": 1, "}": -1}.get(text[j], 0)
                if level == 0:
                    break
            sig, body = out.get((f, m.group(1)), ("", ""))
            out[f, m.group(1)] = (sig + text[m.start():end], body + text[i + 1:j])
    return out


def _launched():
    names = set()
    for f in os.listdir(CSRC):
        names |= {(f, n) for n in re.findall(r"launch_chained\(\s*(k_\w+)", open(os.path.join(CSRC, f)).read())}
    return names


def test_chained_kernels_wait_first():
    fun = _functions()
    launched = _launched()
    assert len(launched) >= 25, launched
    for key in launched:
        assert key in fun, key
        assert re.match(r"\s*chain_begin\(\);", fun[key][1]), key
    for key, (sig, body) in fun.items():
        if "__global__" in sig and "chain_begin()" in body:
            assert key in launched, key


def test_nothing_a_chained_kernel_calls_takes_restricted_pointers():
    fun = _functions()
    by_name = {}
    for key in fun:
        by_name.setdefault(key[1], []).append(key)
    seen, todo = set(), list(_launched())
    while todo:
        key = todo.pop()
        if key in seen:
            continue
        seen.add(key)
        sig, body = fun[key]
        assert "__restrict__" not in sig + body, key
        for name in set(re.findall(r"\b(\w+)\s*(?:<[\w\s,:&*]*>)?\s*\(", body)):
            here = [k for k in by_name.get(name, ()) if k[0] == key[0]]
            todo += here or by_name.get(name, [])
    names = {k[1] for k in seen}
    assert {"lean_cell_level", "lean_face_point", "lean_picard_point", "stress_edges_point", "df_cell_level",
            "df_face_point", "corr_tile_run", "mix_perm_point", "quad_level", "mg_eq"} <= names, sorted(names)
