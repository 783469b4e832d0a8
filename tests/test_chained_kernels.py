"""Source rules of the kernels launched as programmatic dependents
(launch_chained): such a kernel is resident while its predecessor writes, so
it may read through the non-coherent path (__ldg, const __restrict__) only
what no kernel of a chain writes, no __restrict__ parameter may point to a
vector of the chain, and it waits before it touches one.  No run can show a
violation (whether a load moves before the wait is the compiler's choice), so
the sources are read."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_03632_gb300", "csrc")

# parameters that no chained kernel writes: matrices, indices, scalings, masks, the explicit loop's source
CONSTANT = {"row_ptr", "col", "val", "dinv", "d", "w", "mask", "pidx", "pval", "minv", "sigma", "rows", "idxT", "wT", "f"}
CONTROL = {"flag", "st"}  # the state block and its flag: read after the wait through plain or volatile loads


def sources():
    out = {}
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            out[name] = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
    return out


def closing(s, i, pair="()"):
    depth = 0
    for k in range(i, len(s)):
        depth += {pair[0]: 1, pair[1]: -1}.get(s[k], 0)
        if depth == 0:
            return k
    raise AssertionError("unbalanced")


def split_args(s):
    parts, depth, cur = [], 0, ""
    for c in s:
        depth += {"(": 1, "<": 1, "{": 1, ")": -1, ">": -1, "}": -1}.get(c, 0)
        if c == "," and depth == 0:
            parts.append(cur.strip())
            cur = ""
        else:
            cur += c
    return [p for p in parts + [cur.strip()] if p]


def chained_kernels():
    """(file, kernel, parameters, body) of every kernel that launch_chained is given."""
    src = sources()
    names = set()
    for text in src.values():
        for m in re.finditer(r"\blaunch_chained\(", text):
            args = split_args(text[m.end():closing(text, m.end() - 1)])
            k = re.match(r"(\w+)", args[1]).group(1)
            if k != "void":  # (the definition)
                names.add(k)
    out = []
    for k in sorted(names):
        for f, text in src.items():
            for m in re.finditer(r"__global__[^;{]*?\b%s\(" % k, text):
                e = closing(text, m.end() - 1)
                b = text.index("{", e)
                out.append((f, k, split_args(text[m.end():e]), text[b:closing(text, b, "{}")]))
    assert {k for _, k, _, _ in out} == names
    return out


KERNELS = chained_kernels()


def test_the_chains_are_found():
    assert len(KERNELS) >= 15


@pytest.mark.parametrize("file,kernel,params,body", KERNELS, ids=[k[1] for k in KERNELS])
def test_chained_kernel_reads_what_a_chain_writes_after_the_wait(file, kernel, params, body):
    for p in params:
        name = re.search(r"(\w+)$", p).group(1)
        if "__restrict__" in p:
            assert p.startswith("const") and name in CONSTANT, p
        elif p.startswith("const") and "*" in p:
            assert name in CONTROL, p
    for name in re.findall(r"__ldg\(\s*&?\s*(?:RB_AT\(\s*)?(?:\w+\.)?(\w+)", body):
        assert name in CONSTANT, f"__ldg of {name}"
    # the wait: in the kernel or in chained_rows, in every thread before any return
    head = re.split(r"\breturn;", body)[0]
    assert "pdl_wait()" in head or "chained_rows<" in body


@pytest.mark.parametrize("name", ["row_sum", "sum", "rows32", "rows32_ahead", "chained_rows", "row_dot64", "row_apply_df"])
def test_row_helpers_of_chained_kernels_take_live_vectors(name):
    found = 0
    for f, text in sources().items():
        if f not in ("mg.cu", "csr_rows.cuh", "krylov.cu"):
            continue
        for m in re.finditer(r"(?<![\w.])(?:T|void|double|df) %s\(" % name, text):
            params = split_args(text[m.end():closing(text, m.end() - 1)])
            if not any(re.search(r"\bcol$", p) for p in params):
                continue
            found += 1
            assert any(re.match(r"Live<\w+> x$", p) for p in params), params
    assert found
