"""Kernels that may start before the one in front of them has finished (no GPU needed).

Such a kernel waits in its first statement (dep_begin).  What the kernel in front writes
must not be declared constant for the whole kernel, or the compiler may read it before
the wait, or past the coherent cache.  The sources are read for that: every pointer of
such a kernel but those of tables written when a run is bound goes through dep_begin,
none that is only read is __restrict__, and no load asks for the non-coherent path but of a
table.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_11052_gb300", "csrc")
# written at bind, which synchronises
TABLES = {"tab", "ktab", "desc", "p0", "g0", "c0", "tile_inst", "node_pos"}
# places that kernels write (and read, if at all, through the same pointer)
WRITTEN = {"out", "mode", "part", "fpart", "x", "v", "lrho2", "E_hat", "E8", "E4", "rho"}


def _sources():
    return {os.path.basename(f): open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def _kernels():
    """name -> (parameters, body) of the kernels of the library."""
    found = {}
    for text in _sources().values():
        text = re.sub(r"//[^\n]*", "", text)
        for m in re.finditer(r"__global__ void[^;{]*?\b(k_\w+)\s*\(([^{;]*?)\)\s*\{", text, re.S):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            params = [" ".join(p.split()) for p in m.group(2).split(",")]
            found[m.group(1)] = (params, text[m.end():end])
    return found


KERNELS = _kernels()
DEPENDENT = sorted(k for k, (_, body) in KERNELS.items() if "dep_begin(" in body)


def test_every_kernel_that_may_start_early_waits():
    launched = set()
    for text in _sources().values():
        launched |= set(re.findall(r"launch_dep\(\s*(k_\w+)", text))
    assert launched and launched <= set(DEPENDENT) | {"kern"}
    assert "k_b_push_deposit" in DEPENDENT      # launched through a name of its own


@pytest.mark.parametrize("name", DEPENDENT)
def test_nothing_that_a_kernel_in_front_writes_is_constant(name):
    params, body = KERNELS[name]
    first = body.strip().split(";")[0]
    call = re.fullmatch(r"dep_begin\(([\w, ]*)\)", first)
    assert call, "the first statement is the wait"
    handed = {a.strip() for a in call.group(1).split(",")} - {""}
    pointers = {re.search(r"(\w+)$", p).group(1): p for p in params if "*" in p}
    assert set(pointers) - TABLES == handed
    for arg, decl in pointers.items():
        if "__restrict__" in decl and arg not in TABLES:
            assert "const " not in decl and arg in WRITTEN, decl


def test_only_tables_are_read_past_the_coherent_cache():
    for name, text in _sources().items():
        text = re.sub(r"//[^\n]*", "", text)
        assert "ld.global.nc" not in text, name
        for m in re.finditer(r"__ldg\(\s*(\w+)", text):
            assert m.group(1) in TABLES, (name, m.group(0))
