"""Kernels that are launched before their predecessor has finished (programmatic
dependent launch) read what it writes with ordinary loads only: a read-only
load promises data that does not change during the grid's life, and nothing
need keep it behind the wait.  Checked in the sources, since a reordering
would show by chance."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1904_06881_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def _functions(text):
    """(header, body) of every function definition at namespace scope."""
    for m in re.finditer(r"^(?:template[^\n]*\n)?(?:__global__|__device__|static|inline)[^;{}]*\)\s*\{", text, re.M):
        depth, k = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(0), text[m.end():k]


def test_read_only_loads_are_of_flags_and_tables():
    early = 0
    for name in ("tlb_device.cuh", "tlb_kernels.cuh", "tlb_step.cuh"):
        text = _source(name)
        for head, body in _functions(text):
            waits = "pdl_wait()" in body
            early += waits
            if "__global__" in head and not waits:
                continue                       # a plain launch: its predecessors are done
            assert "const void *__restrict__" not in head, head
            for q in re.findall(r"const\s+(?:float2?|__half)\s*\*\s*__restrict__\s*(\w+)", head):
                assert q == "c", (name, head)  # a tile in shared memory
            for arg in re.findall(r"__ldg\(([^;]*)", body):
                assert re.match(r"(?:e\.)?(?:type|wall_tiles) \+", arg), (name, arg)
    assert early == 4                          # step and moments, one lattice and a table
    # structs' members are in no function's header
    gio = _source("tlb_kernels.cuh")
    for arg in re.findall(r"__ldg\(([^;]*)", gio[gio.index("struct GIO<float>"):gio.index("struct Tile;")]):
        raise AssertionError(arg)
