"""The functions that remember which devices know a kernel's attributes have
internal linkage (csrc): the statics of inline functions and templates are one
object for all libraries of a process, while every library registers kernels of
its own, so that the second library would find the work of the first and launch
without the attribute."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2208_06191_gb300", "csrc")


def test_attribute_state_has_internal_linkage():
    found = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"static PerDevice<bool> \w+;", text):
            found += 1
            # the line that opens the enclosing function
            head = [ln for ln in text[:m.start()].split("\n") if re.match(r"\S.*\(", ln)][-1]
            assert not head.startswith("inline"), (name, head)
    assert found >= 4
