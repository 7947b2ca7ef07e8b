"""Kernels launched over the end of the one before read memory that this one still writes when
they start: such data must not go through the read-only path (``__ldg`` or a restrict-qualified
pointer that the kernel never writes through), which is defined only for data that nothing
writes while the kernel lives.  Read from the sources: no GPU runs here.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_07499_gb300", "csrc")
FILES = ["hmg_fast.cu", "hmg_gen32_kernels.cuh", "hmg_fixed.cuh", "hmg_fixed_kernels.cuh", "hmg_kernels.cu"]
TABLES = ("tw", "twL", "twM", "twN", "tab", "g.tw32", "g.twf", "g.rcp")   # written once, before any kernel


def _source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def _functions(src):
    """(name, parameters, body) of every device function and kernel."""
    for m in re.finditer(r"__(?:global|device)__[^;{}]*?\b(\w+)\(", src):
        def match(i, pair):
            depth = 0
            while True:
                depth += (src[i] == pair[0]) - (src[i] == pair[1])
                i += 1
                if depth == 0:
                    return i
        if m.group(1).startswith("__"):   # __launch_bounds__( ... ) name(
            end = match(m.end() - 1, "()")
            n = re.match(r"\s*(\w+)\(", src[end:])
            if not n:
                continue
            name, p0 = n.group(1), end + n.end() - 1
        else:
            name, p0 = m.group(1), m.end() - 1
        p1 = match(p0, "()")
        b0 = src.find("{", p1)
        if src[p1:b0].strip(" \n") not in ("", "const"):
            continue
        yield name, src[p0 + 1:p1 - 1], src[b0:match(b0, "{}")]


def test_parser_sees_the_kernels():
    early = {n for f in FILES for n, _, b in _functions(_source(f)) if "grid_begin()" in b}
    assert {"k_fy", "k_fz3", "k_fzs", "k_px_round_p", "k_gx_round", "k_gz", "k_fxx_col", "k_fxx_z", "k_reduce", "k_yxy"} <= early


@pytest.mark.parametrize("name", FILES)
def test_early_kernels_read_by_plain_loads(name):
    for fn, params, body in _functions(_source(name)):
        for p in params.split(","):
            m = re.search(r"const\b.*\*\s*__restrict__\s*(\w+)", p)
            if m and ("grid_begin()" in body or not fn.startswith("k_")):
                assert m.group(1) in TABLES, f"{name}: {fn}({p.strip()})"
        for m in re.finditer(r"__ldg\(&([\w.]+)", body):
            assert m.group(1) in TABLES, f"{name}: {fn}: {m.group(0)}"


@pytest.mark.parametrize("kernel", ["k_fz3", "k_fzs"])
def test_spectrum_of_an_equilibrium_test_is_not_restrict(kernel):
    # their Z_EQ form only reads the spectrum, const or not
    params = {n: p for n, p, _ in _functions(_source("hmg_fast.cu"))}[kernel]
    assert "float2* spec" in params
