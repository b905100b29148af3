"""Compiler ordering around the asynchronous steps of the device code, on the
sources (no GPU needed).

An inline-assembly statement without a "memory" clobber does not order the
plain loads and stores around it: the compiler may move an operand store past
the proxy fence that publishes it, or a read of the tensor-memory address
ahead of the barrier behind its allocation.  So every statement that
synchronises, allocates, copies asynchronously or issues tensor-core work
names "memory", and a tcgen05.ld stands in one statement with the wait that
makes its registers valid (a clobber orders memory, not registers)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2103_16073_gb300", "csrc")
ORDERS = re.compile(r"tcgen05\.|mbarrier\.|fence\.|barrier\.cluster|cp\.async")


def statements(text):
    """The inline-assembly statements of a source, parenthesis to parenthesis."""
    out = []
    for m in re.finditer(r"\basm\s+volatile\s*\(|\basm\s*\(", text):
        depth, i, quoted = 1, m.end(), False
        while depth:
            c = text[i]
            if c == '"' and text[i - 1] != "\\":
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            i += 1
        out.append(text[m.start():i])
    return out


FILES = sorted(p for p in glob.glob(os.path.join(CSRC, "*.cu*")) if "asm" in open(p).read())


def test_statements_are_found():
    assert statements('asm volatile("a.b [%0];" ::"r"(f(x)) : "memory"); g();') == [
        'asm volatile("a.b [%0];" ::"r"(f(x)) : "memory")']
    assert sum(len(statements(open(p).read())) for p in FILES) > 20


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_asynchronous_statements_order_memory(path):
    for s in statements(open(path).read()):
        if ORDERS.search(s):
            assert '"memory"' in s and "volatile" in s, s
        if "tcgen05.ld" in s:
            assert "tcgen05.wait::ld" in s, s


def test_bulk_copies_stay_within_a_cta():
    """The kernels also run with one rank per GPU, where a copy goes to the
    CTA that issues it: the plain form, without a mask of further CTAs."""
    plain = re.compile(r"cp\.async\.bulk\.shared::cluster\.global\.mbarrier::complete_tx::bytes \[%0\], \[%1\], %2, \[%3\];")
    copies = [s for p in FILES for s in statements(open(p).read()) if "cp.async.bulk" in s]
    assert copies and all(plain.search(s) for s in copies)
