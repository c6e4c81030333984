"""Host-side decisions of a step (csrc/npfem_plan.h) on the CPU: the header is compiled into a
small program that answers one query per line."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1903_06479_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "npfem_plan.h"
using namespace npfem;
static std::vector<PlanGroup> groups()
{
    int k = 0;
    std::vector<PlanGroup> g;
    if (scanf("%d", &k) != 1) return g;
    for (int q = 0; q < k; ++q) {
        int n, window, clusters;
        long long cells;
        if (scanf("%d %d %lld %d", &n, &window, &cells, &clusters) != 4) return g;
        g.push_back({n, (n + 3) & ~3, window, cells, clusters != 0});
    }
    return g;
}
int main()
{
    char what[32];
    while (scanf("%31s", what) == 1) {
        if (!strcmp(what, "carry")) {
            const CarryPlan c = plan_carry(groups());
            printf("%lld", c.total);
            for (size_t q = 0; q < c.rec.size(); ++q) printf(" %d %lld %lld", c.window[q], c.off[q], c.rec[q]);
            printf("\n");
        }
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "plan.cpp", d / "plan"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def ask(line):
        return subprocess.run([str(exe)], input=line + "\n", capture_output=True, text=True, check=True).stdout.split()
    return ask


def _record(n, m):
    """Elements of one cell's record: header, m x m products, 2 m vectors."""
    return 4 + ((m * m + 3) & ~3) + 6 * m * ((n + 3) & ~3)


# groups (vertices, own window, cells, takes the cluster kernel) and the window each group's launch
# takes: a cluster group its own, the others that of the first SIMT group with cells
@pytest.mark.parametrize("groups,windows", [
    ([(642, 5, 3, 0)], [5]),
    ([(642, 2, 7, 1), (258, 8, 9, 1)], [2, 8]),                       # clusters: a larger window second
    ([(642, 2, 7, 1), (2562, 8, 3, 0)], [2, 8]),                      # clusters, then SIMT
    ([(642, 3, 0, 0), (258, 8, 5, 0), (66, 1, 4, 0)], [8, 8, 8]),     # the first group has no cells
    ([(642, 8, 2, 0), (258, 1, 5, 0)], [8, 8]),
    ([(642, 0, 2, 1), (1026, 0, 5, 0)], [0, 0]),
])
def test_carried_records_lie_in_the_buffer(plan, groups, windows):
    line = "carry %d " % len(groups) + " ".join("%d %d %d %d" % g for g in groups)
    out = [int(q) for q in plan(line)]
    total, rows = out[0], [out[1 + 3 * q:4 + 3 * q] for q in range(len(groups))]
    end = 0
    for (n, _, cells, _), (window, off, rec), want in zip(groups, rows, windows):
        if cells:
            assert window == want
        assert rec == _record(n, window) and off == end
        end += rec * cells
    assert total == end


def test_launches_take_the_planned_records():
    """No launch sizes a record by itself: the buffer and every launch share one plan."""
    src = open(os.path.join(CSRC, "npfem_api.cu")).read()
    assert "carry_rec_elems" not in src and src.count("plan_carry(") == 1
