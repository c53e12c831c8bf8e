"""Kernels of a chain of dependent launches are resident before their
predecessor's writes are visible (chain_wait in pa_internal.cuh), so what they read
is not read-only for their lifetime: no read-only load and no __restrict__ on it.
Only kernels that are launched alone may use them."""
from __future__ import annotations

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2006_00561_gb300", "csrc")
ALONE = ("k_gather", "k_philox_rate", "k_intops")  # plain launches
HINTS = re.compile(r"__ldg\s*\(|__restrict__|ld\.global\.nc|__ldca\s*\(")


def code(name: str) -> str:
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def without_kernel(text: str, kernel: str) -> str:
    """`text` without the definition of `kernel`, arguments and body."""
    at = re.search(r"\b%s\s*\([^;{]*\{" % kernel, text)
    if not at:
        return text
    depth, end = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
    return text[: at.start()] + text[end:]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_chained_kernels_read_without_read_only_hints(name):
    text = code(name)
    for kernel in ALONE:
        assert not re.search(r"launch_chained\([^;]*\b%s\b" % kernel, text)
        text = without_kernel(text, kernel)
    lines = [line.strip() for line in text.splitlines() if HINTS.search(line)]
    assert not lines, lines


def test_the_scan_sees_a_hint():
    assert HINTS.search("v = __ldg(p + i);") and HINTS.search("const uint4* __restrict__ p")
    body = "__global__ void k_gather(RunDev d) { if (a) { b = __ldg(p); } } int after;"
    assert "after" in without_kernel(body, "k_gather") and not HINTS.search(
        without_kernel(body, "k_gather"))
