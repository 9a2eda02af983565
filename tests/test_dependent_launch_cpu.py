"""Kernels that may start before their predecessor has finished (programmatic
dependent launch) read nothing ahead of the wait: read from the CUDA sources.

A kernel is launched that way when no <<<...>>> names it (or a function pointer taken
from it).  It has to call pdl_start before anything else, and every pointer parameter that it reads has to go through
pdl_start or pdl_behind: a load through the parameter itself may be scheduled ahead
of the wait, because the compiler may take the data of a const __restrict__
pointer as unchanged for the kernel's whole life.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1505_07865_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))

# parameters that a kernel only writes (or, ticket, changes by atomics)
WRITTEN = {
    "k_stokes": {"y"},
    "k_stokes_fx": {"y", "z"},
    "k_stokes_dots": {"w", "ticket"},
    "k_resid_restrict": {"fc"},
    "k_mg_tail": {"ug"},        # read through its copy ur
    "k_mg_cluster": {"ug"},
    "k_rb_first": {"fs", "us"},
    "k_rb_half": {"us", "unat"},
    "k_rb_restrict": {"fc"},
    "k_leg_down": {"uout", "fc"},
    "k_leg_up": {"uout"},
    "k_ps_div": {"qr", "q"},
    "k_ps_finish": {"z"},
    "k_spread_interp": {"out"},
    "k_mgs_block": {"pout", "hcol"},
    "k_mgs_norm": {"st", "vout", "out32", "grow", "H", "res_out", "out64"},
    "k_inner_combine": {"x", "means", "ticket"},
}


def _closing(s, i, pair):
    depth = 0
    while True:
        depth += {pair[0]: 1, pair[1]: -1}.get(s[i], 0)
        if depth == 0:
            return i
        i += 1


def _kernels(src):
    """name -> (pointer parameters, body) of every __global__ function"""
    out = {}
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\(.*?\)\s+)?(\w+)\(", src):
        a = m.end() - 1
        b = _closing(src, a, "()")
        params = [p.strip() for p in src[a + 1:b].split(",")]
        c = src.index("{", b)
        body = src[c + 1:_closing(src, c, "{}")]
        out[m.group(1)] = ([re.findall(r"\w+", p)[-1] for p in params if "*" in p], body)
    return out


def _stripped(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _dependent():
    for name in SOURCES:
        src = _stripped(name)
        for k, (ptrs, body) in _kernels(src).items():
            names = [k] + re.findall(r"\bauto\s*\*?\s*(\w+)\s*=[^;]*\b%s\b" % k, src)
            if not any(re.search(r"\b%s(?:<[^;<]*>)?\s*<<<" % n, src) for n in names):
                yield name, k, ptrs, body


CASES = list(_dependent())


def test_the_kernels_are_found():
    names = {k for _, k, _, _ in CASES}
    assert set(WRITTEN) <= names
    started = {k for f in SOURCES for k, (_, body) in _kernels(_stripped(f)).items() if "pdl_start(" in body}
    assert names >= started and len(started) >= 20


@pytest.mark.parametrize("src,name,ptrs,body", CASES, ids=[k for _, k, _, _ in CASES])
def test_reads_come_after_the_wait(src, name, ptrs, body):
    # ahead of pdl_start only copies of a pointer parameter
    head = body[:body.index("pdl_start(")]
    copies = dict(re.findall(r"const\s+\w+\s*\*\s*(\w+)\s*=\s*(\w+)\s*;", head))
    assert not re.sub(r"const\s+\w+\s*\*\s*\w+\s*=\s*\w+\s*;", "", head).strip(), head
    passed = set()
    for call in re.findall(r"\bpdl_(?:start|behind)\(([^)]*)\)", body):
        passed |= {p.strip() for p in call.split(",")}
    missing = set(ptrs) - passed - WRITTEN.get(name, set())
    assert not missing, f"{src}: {name} reads {sorted(missing)} past the wait's order"
    for copy, of in copies.items():
        assert copy in passed and of in ptrs
