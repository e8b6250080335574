"""Kernel attributes belong to a device: a launcher that asks for more than 48 KB
of dynamic shared memory once a process would fail on the second device a
program uses (and return a first error for ever).  Every launcher asks again on
each call (0.19 us); here: none keeps the answer in a static."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_03013_gb300", "csrc")


def test_no_launcher_sets_a_kernel_attribute_once_a_process():
    calls = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"cudaFuncSetAttribute", text):
            calls += 1
            statement = re.split(r"[;{}]", text[:m.start()])[-1]
            assert not re.search(r"\bstatic\b|call_once", statement), (name, statement.strip())
    assert calls >= 10
