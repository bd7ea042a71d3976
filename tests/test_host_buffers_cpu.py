"""The buffers that hho_erk_run_host keeps with an operator (host_buffers.h) stay
consistent when an allocation fails, tried on the host with an allocator that
fails on demand."""
import os
import subprocess

import pytest

from tests.libutil import ROOT

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <set>

#include "host_buffers.h"

static std::set<double*> live;
static int countdown;   // the allocation that fails
static bool memset_ok;
static bool made;   // a buffer is new
static int grow(hho_ops* o, int64_t size) {
    return grow_host_buffers(
        o, size,
        [](size_t n) -> double* {
            if (--countdown == 0) return nullptr;
            double* p = (double*)malloc(sizeof(double) * n);
            live.insert(p);
            return p;
        },
        [](double* p) {
            if (!live.erase(p)) abort();   // freed twice, or never allocated
            free(p);
        },
        [](double* p, size_t) { return live.count(p) && memset_ok; }, &made);
}
static bool ready(const hho_ops& o, int64_t size) {
    return live.count(o.d_host_state) && live.count(o.d_host_canon) && live.count(o.d_host_work) &&
           o.host_work_size >= size && live.size() == 3;
}
static bool consistent(const hho_ops& o) {
    for (double* p : {o.d_host_state, o.d_host_canon, o.d_host_work})
        if (p && !live.count(p)) return false;
    return o.host_work_size == 0 || (o.d_host_work && o.d_host_state && o.d_host_canon);
}

int main(int argc, char** argv) {
    const int first = atoi(argv[1]), fail = atoi(argv[2]);   // work size of the first call; which allocation fails
    memset_ok = fail != 4;
    countdown = fail == 4 ? 0 : fail;
    hho_ops o;
    o.n_state = 7;
    o.n_canonical = 5;
    if (first) {   // a good call before
        const bool m = memset_ok;
        const int c = countdown;
        countdown = 0, memset_ok = true;
        if (grow(&o, first) != HHO_OK || !ready(o, first)) return 1;
        countdown = c, memset_ok = m;
    }
    const int rc = grow(&o, 40);
    if (rc == HHO_OK || !consistent(o)) return 2;
    countdown = 0, memset_ok = true;
    if (grow(&o, 30) != HHO_OK || !ready(o, 30)) return 3;   // a smaller tableau afterwards
    if (grow(&o, 40) != HHO_OK || !ready(o, 40)) return 4;
    const double* w = o.d_host_work;
    if (!made || grow(&o, 20) != HHO_OK || o.d_host_work != w || made) return 5;
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_buffers")
    (d / "main.cpp").write_text(PROGRAM)
    exe = str(d / "main")
    csrc = os.path.join(ROOT, "paper_2505_15771_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I" + csrc, "-I" + os.path.join(ROOT, "include"), str(d / "main.cpp"), "-o", exe],
                   check=True)
    return exe


# fresh operators: state, canonical vector, work, clearing; then one with a smaller work buffer: work, clearing
@pytest.mark.parametrize("first,fail", [(0, 1), (0, 2), (0, 3), (0, 4), (16, 1), (16, 4)])
def test_a_failed_allocation_leaves_whole_buffers(program, first, fail):
    assert subprocess.run([program, str(first), str(fail)]).returncode == 0
