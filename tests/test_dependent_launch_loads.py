"""Kernels that start before the kernel in front of them has finished
(programmatic dependent launch: they call pdl_wait) read nothing through the
non-coherent path.  Such a load (ld.global.nc, __ldg, or one that the compiler
makes of a const __restrict__ pointer) is defined only for data that nobody
writes while the kernel runs, and the kernel in front is still writing then;
the compiler may also move it ahead of the wait.  No run shows this reliably,
so the sources are read: each such kernel and every function that it calls."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_06969_gb300", "csrc")
NON_COHERENT = re.compile(r"__ldg\b|ld\.global\.nc|\bconst\s+[\w:]+\s*\*\s*__restrict__")
NOT_CALLS = {"if", "for", "while", "switch", "return", "sizeof", "decltype", "static_assert"}


def functions(text):
    """[(name, signature + body)] of the function definitions in a source."""
    text = re.sub(r"/\*.*?\*/", " ", re.sub(r"//[^\n]*", "", text), flags=re.S)
    text = re.sub(r"^\s*#[^\n]*(\\\n[^\n]*)*", "", text, flags=re.M)
    out, start, k = [], 0, 0
    while k < len(text):
        c = text[k]
        if c == ";" or c == "}":
            start = k + 1
        elif c == "{":
            head = text[start:k]
            if "(" not in head or re.match(r"\s*(template\s*<[^{}]*>\s*)?(namespace|struct|class|enum|extern)\b", head):
                start = k + 1                        # its members are looked at by themselves
            else:
                depth, end = 1, k + 1
                while depth:
                    depth += {"{": 1, "}": -1}.get(text[end], 0)
                    end += 1
                plain = re.sub(r"__launch_bounds__\s*\([^()]*(\([^()]*\)[^()]*)*\)", "", head)
                name = re.search(r"([A-Za-z_]\w*)\s*\(", plain)
                if name:
                    out.append((name.group(1), head + text[k:end]))
                start, k = end, end - 1
        k += 1
    return out


def sources():
    defs = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            for name, body in functions(f.read()):
                defs.setdefault(name, []).append(body)
    return defs


def reached(defs, root):
    """root and the functions that it calls, directly or through others."""
    seen, todo = set(), [root]
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        for body in defs[name]:
            calls = set(re.findall(r"\b([A-Za-z_]\w*)\s*(?:<[^;(){}]*>)?\s*\(", body)) - NOT_CALLS
            todo += [c for c in calls if c in defs]
    return seen


def test_waiting_kernels_load_coherently():
    defs = sources()
    kernels = [n for n, bodies in defs.items() if any("pdl_wait()" in b and "__global__" in b for b in bodies)]
    # the reader finds kernels and what they call, through templates too
    assert {"kg_atom", "kg_finish", "kg_grad", "k_totals", "k_pack", "k_grad_partial"} <= set(kernels)
    assert {"group_sums", "group_pair", "pair_vector"} <= reached(defs, "kg_atom")
    assert "chunk_plan_block" in reached(defs, "k_pack")
    assert "load8_ro" in defs and any(NON_COHERENT.search(b) for b in defs["load8_ro"])
    bad = {(k, f) for k in kernels for f in reached(defs, k) if any(NON_COHERENT.search(b) for b in defs[f])}
    assert not bad, sorted(bad)
