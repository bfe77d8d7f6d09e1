"""Sweeps may run beside the end of the sweep that writes their source array, so they load
populations with ordinary (coherent) loads: read from the source, since what a non-coherent
load would return is not defined and so not to be observed."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0811_4593_gb300", "csrc")
NON_COHERENT = re.compile(r"__ldg\s*\(|\.nc\b|Storage<\w+>::load\s*\(")


def _functions(names):
    """The code (comments excluded) of each function of ``names`` in the kernel headers."""
    found = {}
    for f in ("kernels.cuh", "resident.cuh"):
        with open(os.path.join(CSRC, f), encoding="utf-8") as fh:
            text = re.sub(r"//[^\n]*|/\*.*?\*/", "", fh.read(), flags=re.S)
        for m in re.finditer(r"\b(\w+)\s*\(", text):
            if m.group(1) not in names:
                continue
            head = re.compile(r"[^;{}]*\{").match(text, m.start())
            if not head:  # a call or a declaration
                continue
            at, depth = head.end(), 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            found.setdefault(m.group(1), []).append(text[head.end():at])
    return found


# what loads populations in the sweeps, and the sweeps themselves
NAMES = ("load_pop", "ld_half_l2", "ld_half2_l2", "load_pair", "sweep_node", "sweep_block", "update_node",
         "sweep_kernel", "sweep_pair_kernel", "sweep_rows_kernel", "resident_kernel", "grid_steps_kernel")


@pytest.mark.parametrize("name", NAMES)
def test_population_loads_of_sweeps_are_coherent(name):
    bodies = _functions({name}).get(name)
    assert bodies, f"{name} is not there any more"
    for body in bodies:
        assert not NON_COHERENT.search(body), NON_COHERENT.search(body).group(0)
