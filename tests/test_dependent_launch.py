"""Kernels launched to start before their predecessor ends (those that begin with
dep_begin()) read nothing through the read-only data path: that path is specified for
memory that stays the same for a kernel's whole lifetime, and such a kernel is resident
while the one before it, of the same call or of the call before, still writes.  The
sources are read as text: no __ldg and no `const ... * __restrict__` in the kernels or in
the functions of their file that they reach."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_10783_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
SHARED = ("common.cuh", "jobs.cuh", "spline.cuh")


def _strip(text):
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _functions(text):
    """name -> list of (parameters, body) of every function defined in `text`."""
    out = {}
    for m in re.finditer(r"\b([A-Za-z_]\w*)\s*\(", text):
        depth, i = 1, m.end()
        while depth and i < len(text):
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        tail = re.match(r"\s*(const\s*)?\{", text[i:])
        if depth or not tail or m.group(1) in ("if", "for", "while", "switch", "__launch_bounds__"):
            continue
        depth, j = 1, i + tail.end()
        start = j
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        out.setdefault(m.group(1), []).append((text[m.end():i - 1], text[start:j - 1]))
    return out


def _reached(funcs, roots):
    seen, todo = set(), list(roots)
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        for _, body in funcs[f]:
            todo += [n for n in set(re.findall(r"\b([A-Za-z_]\w*)\s*(?:<[^;(){}]*>)?\s*\(", body)) if n in funcs]
    return seen


def _texts(f):
    return "".join(_strip(open(os.path.join(CSRC, n)).read()) for n in (f,) + SHARED)


@pytest.mark.parametrize("f", FILES)
def test_no_read_only_loads(f):
    funcs = _functions(_texts(f))
    roots = [n for n, defs in funcs.items() if n.startswith("k_") and any("dep_begin()" in b for _, b in defs)]
    for n in _reached(funcs, roots):
        for params, body in funcs[n]:
            assert body.find("__ldg") < 0, n
            assert not re.findall(r"const\s+\w+\s*\*\s*__restrict__", params + body), n


def test_kernels_found():
    """The reading above sees the kernels it is meant for."""
    found = {n for f in FILES for n, defs in _functions(_texts(f)).items()
             if n.startswith("k_") and any("dep_begin()" in b for _, b in defs)}
    assert {"k_mesh_stats", "k_sub_thresh_poly", "k_tile_label", "k_centroid_rows", "k_aperture", "k_reproject",
            "k_aff_sum2", "k_sub_conv", "k_chol_diag", "k_clean_pairs"} <= found
    funcs = _functions(_texts("detect.cu"))
    assert {"tile_label_fast", "tile_label_body"} <= _reached(funcs, ["k_tile_label"])


def test_dependent_kernels_wait():
    """Every kernel launched as a dependent one waits before anything else."""
    for f in FILES:
        text = _texts(f)
        funcs = _functions(text)
        names = set(re.findall(r"ipp_launch_dep\(\s*(?:\w[^?,]*\?\s*)?(k_\w+)", text))
        names |= set(re.findall(r"launch_resident<\s*(k_\w+)", text)) | set(re.findall(r":\s*(k_\w+)<\w+>,\s*dim3", text))
        for n in names:
            for _, body in funcs[n]:
                stmts = [s.strip() for s in body.split(";") if s.strip() and "__shared__" not in s]
                assert stmts[0] == "dep_begin()", n
