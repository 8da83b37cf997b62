"""Kernels that start under the end of the kernel before them (csrc/pdl.cuh) read what it wrote while they are already
running, so none of their reads may go by the read-only path or be moved up over the wait: no const __restrict__
parameter and no load intrinsic but those of the constant tables, in the kernels and in the device functions that
they call.  Checked on the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_19048_gb300", "csrc")
WAITS = re.compile(r"\bpdl_enter\(\)|griddepcontrol\.wait")
READ_ONLY = re.compile(r"const\s+[\w:]+\s*\*\s*__restrict__")
INTRINSIC = re.compile(r"__ld(?:ca|cg|cs|lu|cv)\(|__ldg\(&?(\w+)")


def _closing(s, i, pair):
    depth = 0
    for k in range(i, len(s)):
        depth += (s[k] == pair[0]) - (s[k] == pair[1])
        if depth == 0:
            return k
    raise ValueError(pair)


def _functions(s):
    """(qualifier, name, parameters, body) of every device function and kernel of a source text."""
    for m in re.finditer(r"__(global|device)__(?=[\s\w])", s):
        at = re.compile(r"([\w:]+)\s*\(").search(s, m.end())
        while at and at.group(1) in ("__launch_bounds__", "asm"):
            at = re.compile(r"([\w:]+)\s*\(").search(s, _closing(s, at.end() - 1, "()"))
        if not at or ";" in s[m.end():at.start()]:   # a variable
            continue
        end = _closing(s, at.end() - 1, "()")
        rest = s[end + 1:].lstrip()
        if not rest.startswith("{") and not rest.startswith("const"):
            continue
        b = s.index("{", end)
        yield m.group(1), at.group(1), s[at.end():end], s[b:_closing(s, b, "{}") + 1]


def _source(path):
    with open(path) as f:
        s = re.sub(r"//[^\n]*", "", f.read())
    return re.sub(r"__align__\(\d+\)", "", s)


HEADERS = [f for p in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) for f in _functions(_source(p))]
UNITS = {os.path.basename(p): list(_functions(_source(p))) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}
KERNELS = [(u, f) for u, fs in UNITS.items() for f in fs if f[0] == "global" and WAITS.search(f[3])]


def _table(pointer, body):
    """Whether a pointer is a constant table (g_...) or leads into one."""
    return pointer is not None and (pointer.startswith("g_") or
                                    re.search(r"\b%s\s*=[^;]*\bg_\w+" % pointer, body) is not None)


def faults(unit, kernel):
    helpers = {}
    for f in HEADERS + UNITS[unit]:
        if f[0] == "device":
            helpers.setdefault(f[1], []).append(f)
    seen, todo, found = set(), [kernel], []
    while todo:
        _, name, params, body = todo.pop()
        if READ_ONLY.search(params):
            found.append("%s: %s" % (name, READ_ONLY.search(params).group(0)))
        found += ["%s: %s" % (name, m.group(0)) for m in INTRINSIC.finditer(body) if not _table(m.group(1), body)]
        for callee in set(re.findall(r"(\w+)\s*(?:<[\w\s,:]*>)?\(", body)) & set(helpers) - seen:
            seen.add(callee)
            todo += helpers[callee]
    return found


def test_the_kernels_are_found():
    names = {k[1] for _, k in KERNELS}
    assert {"k_simulate", "k_gemm_bf16", "k_im2col", "k_colsum_finish", "k_gn_backward_s", "k_flow_density"} <= names
    assert len(KERNELS) >= 20


@pytest.mark.parametrize("unit,kernel", KERNELS, ids=[k[1] for _, k in KERNELS])
def test_reads_are_ordered_behind_the_wait(unit, kernel):
    assert faults(unit, kernel) == []


def test_a_read_only_parameter_is_found():
    unit, kernel = next((u, k) for u, k in KERNELS if k[1] == "k_im2col")
    planted = kernel[:2] + (kernel[2].replace("const __nv_bfloat16* x", "const __nv_bfloat16* __restrict__ x"), kernel[3])
    assert faults(unit, planted)
    assert faults(unit, kernel[:3] + (kernel[3].replace("pdl_enter();", "pdl_enter(); use(__ldca(x));"),))
