"""Ordering in the hand-written kernels, read from their source: what a build may reorder shows
on a GPU only as a rare wrong result, so the statements that forbid it are checked as text."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2310_15183_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
# instructions that order, publish or wait for memory accesses of other instructions
ORDERING = re.compile(r"fence\.|mbarrier\.|cp\.async|cp\.reduce|red\.|bar\.|barrier\.|"
                      r"tcgen05\.(alloc|dealloc|relinquish|commit|fence|wait|st|cp)")


def _code(path):
    """The file without comments."""
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _asm_statements(path):
    text = _code(path)
    for m in re.finditer(r"\basm\b", text):
        depth, i = 0, text.index("(", m.start())
        for j in range(i, len(text)):
            depth += {"(": 1, ")": -1}.get(text[j], 0)
            if depth == 0:
                yield text[m.start():j + 1]
                break


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_ordering_instructions_hold_memory_accesses(path):
    """Each such statement is volatile and clobbers memory: a compiler may otherwise move an
    ordinary shared-memory store of an operand past the fence its reader relies on."""
    for s in _asm_statements(path):
        if ORDERING.search(s):
            assert re.match(r"asm\s+volatile", s) and '"memory"' in s, s


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_tensor_memory_loads_wait_in_their_own_statement(path):
    """tcgen05.ld returns before its registers hold the data; a wait in a statement of its own
    says nothing about those registers to the compiler."""
    for s in _asm_statements(path):
        if "tcgen05.ld" in s:
            assert s.find("tcgen05.wait::ld") > s.find("tcgen05.ld."), s


def _kernels(text):
    """Bodies of the __global__ functions."""
    for m in re.finditer(r"__global__", text):
        i = text.index("{", text.index(")\n{", m.start()))
        depth = 0
        for j in range(i, len(text)):
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            if depth == 0:
                yield text[i:j + 1]
                break


def _enclosing(body, pos):
    """Heads (the text since the statement before) of the blocks around a position."""
    stack = []
    for j in range(pos):
        if body[j] == "{":
            stack.append(body[max(body.rfind(c, 0, j) for c in ";{}") + 1:j])
        elif body[j] == "}":
            stack.pop()
    return stack


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_a_bounded_wait_has_one_outcome_per_warp(path):
    """A wait that may run out is taken by one lane, by the warp as one (mbar_wait_warp), or its
    outcome is joined over the CTA (__syncthreads_and): lanes that left a loop on their own would
    be missed by the next warp-wide instruction of the others, which then waits without a limit."""
    for body in _kernels(_code(path)):
        if "__syncthreads_and" in body:
            continue
        for m in re.finditer(r"mbar_wait\(", body):
            assert any("lane == 0" in head for head in _enclosing(body, m.start())), \
                body[m.start() - 80:m.start() + 80]
