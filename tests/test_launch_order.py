"""Programmatic dependent launches: a kernel runs beside its predecessor until
griddepcontrol.wait, so nothing that an earlier launch of the solve writes may be
read before it, by the programmer or by the compiler (checked in the source, as a
load that moves ahead of the wait need not show in a run).

- Every const pointer parameter of such a kernel goes through rf_pdl_begin(), which
  takes the compiler's promise of constant data from it, except the operators, masks and
  inverses, which only a set-up writes; so do the vectors updated in place.
- Ahead of rf_pdl_begin() the kernel does not touch them.
- Neighbour values are loaded by volatile statements and not as read-only data.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_04763_gb300", "csrc")
SETUP_DATA = {"J", "md", "Jdf", "dmf", "dmc", "Ainv"}      # written by set-ups only
IN_PLACE = {"xf", "scal"}


def _read(f):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())


def _block(s, at):
    depth, i = 0, s.index("{", at)
    while True:
        depth += {"{": 1, "}": -1}.get(s[i], 0)
        i += 1
        if depth == 0:
            return i


def _functions():
    """(name, parameters, body) of every function that calls rf_pdl_begin() itself."""
    out = []
    for f in ("levelops.cu", "krylov.cu"):
        s = _read(f)
        for m in re.finditer(r"\b(k_\w+|\w+_body)\s*\(", s):
            close = m.end()
            depth = 1
            while depth:
                depth += {"(": 1, ")": -1}.get(s[close], 0)
                close += 1
            if s[close:close + 2] != " {":
                continue
            body = s[close:_block(s, close)]
            if "rf_pdl_begin(" in body:
                out.append((m.group(1), s[m.end():close - 1], body))
    return out


FUNCTIONS = _functions()


def test_kernels_were_found():
    names = {n for n, _, _ in FUNCTIONS}
    assert {"k_residual_small", "k_gs_pair_small64", "k_gs_pair", "k_bicg_xr", "restrict_planes_body"} <= names
    assert len(FUNCTIONS) > 35


@pytest.mark.parametrize("name,params,body", FUNCTIONS, ids=[f[0] for f in FUNCTIONS])
def test_data_of_earlier_launches_is_read_after_the_wait(name, params, body):
    before, after = body.split("rf_pdl_begin(", 1)
    passed = {t.strip() for t in after[:after.index(")")].split(",") if t.strip()}
    must = set()
    for p in params.split(","):
        m = re.search(r"\*\s*(?:__restrict__ )?(\w+)\s*$", p.strip())
        if not m:
            continue
        const = re.search(r"(^|\s)const (?!__grid_constant__)", " " + p) is not None
        if (const and m.group(1) not in SETUP_DATA) or m.group(1) in IN_PLACE:
            must.add(m.group(1))
        elif m.group(1) == "x" and name.startswith("k_gs") or name == "k_bicg_xr" and m.group(1) == "x":
            must.add("x")
    assert must <= passed, must - passed
    for v in passed:
        assert not re.search(r"\b%s\s*\[" % v, before), v


def test_neighbour_loads_stay_behind_the_wait():
    s = _read("levelops.cu")
    for fn in re.findall(r"\b(ld_keep|ld_written)\(const (?:float2|double2)\* p\) \{(.*?)\n\}", s, re.S):
        asm = [t for t in re.findall(r"asm[^;]*;", fn[1])]
        assert asm and all(t.startswith("asm volatile(\"ld.global.") and ".nc" not in t for t in asm), fn
    assert "__ldcg(" not in s
