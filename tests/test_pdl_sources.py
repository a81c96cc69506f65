"""Kernels that start before their predecessor has ended, read as source: each
one that launch_pdl launches waits for its operands, and no matrix it reads or
writes is __restrict__ (the compiler could then move accesses before the wait;
no run shows whether it did)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1909_01554_gb300", "csrc")


def matching(text, at, opening, closing):
    """The index behind the bracket that closes the one at `at`."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == opening) - (text[i] == closing)
        if depth == 0:
            return i + 1
    raise AssertionError("unbalanced")


def kernels(text):
    """(name, parameters, body) of every __global__ function of a source."""
    for found in re.finditer(r"__global__ void (?:__launch_bounds__)?", text):
        at = found.end()
        if found.group().endswith("__"):
            at = matching(text, at, "(", ")")
        name = re.compile(r"\s*(\w+)\(").match(text, at)
        end = matching(text, name.end() - 1, "(", ")")
        body = text.index("{", end)
        yield name.group(1), text[name.end():end - 1], text[body:matching(text, body, "{", "}")]


SOURCES = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read()) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}
WAITING = [(f, *k) for f, text in SOURCES.items() for k in kernels(text) if "wait_for_operands()" in k[2]]


def test_every_kernel_launched_early_waits():
    early = {name for text in SOURCES.values() for call in re.findall(r"launch_pdl\(([^;]*);", text)
             for name in re.findall(r"\w+_kernel\b", call)}
    early |= {"direct_kernel", "tc_fp4_kernel"}  # with launch attributes of their own
    assert len(early) >= 10 and early == {k[1] for k in WAITING}


@pytest.mark.parametrize("source,name,parameters,body", WAITING, ids=[f"{k[0]}:{k[1]}" for k in WAITING])
def test_no_matrix_is_restrict(source, name, parameters, body):
    # (tables written before the stream's last kernel started, of structs and 32-bit or signed numbers, may be)
    assert not re.search(r"\buint64_t\s*\*\s*__restrict__", parameters)
