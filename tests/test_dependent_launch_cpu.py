"""What the kernels that are launched while their predecessor still runs
(dependent_launch.cuh) may read through the read-only data path: the operator's
tables alone.  States and traces are written by the kernel before, so they take
ordinary loads after the wait; a read-only load may be moved above it."""
import os
import re

import pytest

from tests.libutil import ROOT

CSRC = os.path.join(ROOT, "paper_2505_15771_gb300", "csrc")
# files with dependent kernels and the device functions they call
FILES = ["stage.cu", "stage_kernels.cuh", "stage_team.cuh"]
# operator tables: members of DevOps (directly or by arithmetic), pointers into them
TABLES = {"op", "A.op", "OpData", "WideData", "ci", "co", "scal", "M0", "cd", "nbt", "bet", "src", "p", "NC", "SOLID",
          "reinterpret_cast"}
TABLE_PARAMS = {"ri", "rd"}


def text(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def arguments(src, opening):
    """The text inside the parenthesis at src[opening]."""
    depth = 0
    for i in range(opening, len(src)):
        depth += {"(": 1, ")": -1}.get(src[i], 0)
        if depth == 0:
            return src[opening + 1:i]
    raise AssertionError("unbalanced parentheses")


@pytest.mark.parametrize("name", FILES)
def test_read_only_loads_are_of_operator_tables(name):
    src = text(name)
    for m in re.finditer(r"\b__ldg\(", src):
        arg = arguments(src, m.end() - 1)
        first = re.match(r"[\s(]*((?:A\.)?\w+)", arg).group(1)
        assert first in TABLES, arg


def test_dependent_kernels_take_no_restrict_pointer_to_written_data():
    src = {f: text(f) for f in FILES}
    kernels = {m for f in FILES for m in re.findall(r"launch_dependent\((\w+)<", src[f])}
    assert kernels == {"stage_kernel", "team_kernel", "grad_stage_kernel", "record_kernel"}
    for k in kernels:
        found = [(f, m) for f in FILES for m in re.finditer(r"__global__[^;{]*?\b%s\(" % k, src[f])]
        assert len(found) == 1, k
        f, m = found[0]
        params = arguments(src[f], m.end() - 1)
        restrict = {p.split("=")[0].split()[-1].lstrip("*") for p in params.split(",") if "__restrict__" in p}
        assert restrict <= TABLE_PARAMS, (k, restrict)
        body = src[f][m.end():]
        assert "wait_for_predecessor" in body or k == "team_kernel"


@pytest.mark.parametrize("name,count", [("stage.cu", 1), ("sdirk.cu", 1)])
def test_ticket_counters_are_fenced_on_both_sides(name, count):
    """The last block to take a ticket overwrites (the device clock) or reads
    (the partial sums) what the others read or wrote before theirs: without a
    fence on each side of the ticket a block's access may pass it."""
    src = text(name)
    tickets = list(re.finditer(r"atomicAdd\([^,]*ticket", src))
    assert len(tickets) == count
    for m in tickets:
        kernel = src[src.rindex("__global__", 0, m.start()):]
        at = m.start() - (len(src) - len(kernel))
        before = re.split(r"clock->step|A\.partial", kernel[:at])[-1]
        after = re.split(r"clock->step|A\.partial", kernel[at:])[0]
        assert "__threadfence()" in before and "__threadfence()" in after
