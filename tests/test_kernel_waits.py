"""Kernels that start while their predecessor drains (griddepcontrol) must not
read its data through read-only loads: for a const __restrict__ pointer the
compiler may move them above the wait.  Every kernel that waits takes such
pointers only for the tables made once when a run is created."""

import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1604_08159_gb300" / "csrc"
TABLES = {"tw", "sigma", "dsym", "inv"}
KERNEL = re.compile(r"__global__\s+void\s*(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(([^{]*?)\)\s*\{")


def waiting_kernels():
    for f in sorted(CSRC.glob("*.cu*")):
        s = f.read_text()
        for m in KERNEL.finditer(s):
            end, depth = m.end(), 1
            while depth:
                depth += {"{": 1, "}": -1}.get(s[end], 0)
                end += 1
            if "pdl_wait" in s[m.end():end]:
                yield f.name, m.group(1), m.group(2)


def test_no_read_only_pointers_to_a_predecessors_data():
    found = list(waiting_kernels())
    assert len(found) > 40
    bad = [(file, kernel, p.strip()) for file, kernel, params in found
           for p in params.split(",")
           if re.search(r"\bconst\b.*__restrict__", p, re.S) and p.split()[-1] not in TABLES]
    assert not bad, bad
