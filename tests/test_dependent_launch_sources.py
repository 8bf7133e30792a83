"""Source check of the dependently launched kernels (no GPU).

A kernel that waits for its predecessor inside (pdl_wait) must not load what
the predecessor writes before the wait.  The wait is an asm statement with a
memory clobber; an array behind a __restrict__ argument may be taken to lie
outside of it.  So in a waiting kernel, and in the device functions that it
calls, __restrict__ is allowed on

- pointers to const data that no kernel of the iteration writes: the names in
  CONSTANT (operators, interpolation weights, index lists, diagonals), and
- arrays that the function writes and never reads.
"""
import os
import re

import pytest

from paper_2509_08109_gb300 import build

# A: operator planes; P: interpolation weights; rs: row sums; va, ci, so, rp:
# sliced-ELLPACK values, columns and offsets; map: coarse node numbers; dinv:
# reciprocal diagonals; w: lumped mass; targs: a batch's tables of pointers
CONSTANT = {"A", "P", "rs", "va", "ci", "so", "rp", "map", "dinv", "w", "targs"}

FUNC = re.compile(r"__(?P<kind>global|device)__\s+(?P<head>[^;{}]*?)\b(?P<name>\w+)\s*\((?P<args>[^{};]*)\)\s*(?:const\s*)?\{")


def _strip(text):
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "", text)


def _body(text, start):
    depth = 1
    for k in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[start:k]
    raise AssertionError("unbalanced braces")


def functions(text):
    """name -> list of (is_kernel, [arguments], body) of a source's device functions."""
    out = {}
    text = _strip(text)
    for m in FUNC.finditer(text):
        args = [a.strip() for a in re.sub(r"<[^<>]*>", "", m["args"]).split(",")]
        out.setdefault(m["name"], []).append((m["kind"] == "global", args, _body(text, m.end())))
    return out


def reads(name, body):
    """Whether the body does anything with the array but store to it (or see whether it is null)."""
    left = re.sub(rf"\*\s*reinterpret_cast<[^<>]*>\(\s*{name}\b[^;=]*?\)\s*=(?!=)", "", body)
    left = re.sub(rf"\b{name}\[(?:[^\[\]]|\[[^\[\]]*\])*\]\s*=(?!=)", "", left)
    left = re.sub(rf"\bif \({name}\)", "", left)
    # handed to restrict_node3d as its output (checked there)
    left = re.sub(rf"(restrict_node3d(?:<\w+>)?\([^;]*?), {name}\b", r"\1", left)
    return re.search(rf"\b{name}\b", left) is not None


def violations(text):
    fs = functions(text)
    todo = [n for n, v in fs.items() if any(k and "pdl_wait()" in b for k, _, b in v)]
    waiting, bad = set(), []
    while todo:
        n = todo.pop()
        if n in waiting:
            continue
        waiting.add(n)
        for is_kernel, args, body in fs[n]:
            if is_kernel and "pdl_wait()" not in body:
                continue
            todo += [c for c in set(re.findall(r"\b(\w+)\s*(?:<[^<>;]*>)?\(", body)) if c in fs and c not in waiting]
            for a in args:
                if "__restrict__" not in a:
                    continue
                name = re.findall(r"\w+", a)[-1]
                if re.match(r"const\b", a):
                    if name not in CONSTANT:
                        bad.append((n, name, "read"))
                elif reads(name, body):
                    bad.append((n, name, "read and written"))
    return waiting, bad


SOURCES = [s for s in build.sources() if "pdl_wait()" in open(s).read()]


def test_the_waiting_kernels_are_found():
    names = {os.path.basename(s) for s in SOURCES}
    assert {"krylov.cu", "aux2d.cu", "vcycle3d.cu", "fused2d.cu", "tail2d.cu"} <= names
    found = set().union(*(violations(open(s).read())[0] for s in SOURCES))
    assert {"k_update_xr32", "k_pspmv2d_strips", "k_jacobi", "sell_sum", "csr_row", "k_restrict3d"} <= found


@pytest.mark.parametrize("source", SOURCES, ids=os.path.basename)
def test_no_restrict_on_what_another_kernel_writes(source):
    assert violations(open(source).read())[1] == []


@pytest.mark.parametrize("line,bad", [
    ("const float* __restrict__ p, float* __restrict__ q) { pdl_wait(); q[0] = p[0]; }", [("k", "p", "read")]),
    ("const float* __restrict__ A, float* __restrict__ q) { pdl_wait(); q[0] += A[0]; }",
     [("k", "q", "read and written")]),
    ("const float* __restrict__ A, float* __restrict__ q) { pdl_wait(); q[A[0]] = A[1]; }", []),
    ("const float* __restrict__ p, float* q) { q[0] = p[0]; }", []),
])
def test_the_check_itself(line, bad):
    assert violations("__global__ void k(" + line)[1] == bad
