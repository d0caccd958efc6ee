"""Simulation state is read through coherent loads.

A step's kernel may be resident while the one before it still writes the state it is
about to read (programmatic dependent launch).  Loads of the read-only path
(ld.global.nc, __ldg, const __restrict__ pointers to state) and asm loads that are not
volatile may be moved above the wait for that kernel, where a list entry would not be
written yet.  Whether a compiler does so cannot be tested by running it, so the sources
are looked at.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1410_3464_gb300", "csrc")


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", ["device.cuh", "step.cuh", "interface.cuh"])
def test_state_is_read_through_coherent_loads(name):
    src = code(name)
    assert ".nc." not in src
    # constant for the life of a handle: the rates of a batch member's parameters
    assert set(re.findall(r"__ldg\(([^()]*)\)", src)) <= {"&v"}
    # ... its descriptors and the work list
    const = re.findall(r"const (\w+(?:<\w+>)?)\* __restrict__ \w+", src)
    assert set(const) <= {"DevInst", "Work"}, const
    for load in re.findall(r"asm (\w*)\s*\(\"ld\.global", src) + re.findall(r"asm(\()\"ld\.global", src):
        assert load == "volatile"
    for wait in re.findall(r"asm ([^;]*griddepcontrol\.wait;[^;]*);", src):
        assert wait.startswith("volatile") and '"memory"' in wait
