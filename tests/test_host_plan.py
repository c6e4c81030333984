"""Host-side decisions of a step (csrc/npfem_plan.h) on the CPU: the header is compiled into a
small program that answers one query per line."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1903_06479_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
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
        } else if (!strcmp(what, "threads")) {
            int n, fp64, dense, damped, eval;
            long long cells;
            if (scanf("%d %d %d %d %lld %d", &n, &fp64, &dense, &damped, &cells, &eval) != 6) return 1;
            const SimtMesh m = {n, fp64 != 0, dense != 0, damped != 0};
            printf("%d\n", eval ? eval_threads(m, cells, 152) : simt_threads(m, cells, 152));
        } else if (!strcmp(what, "dense")) {
            int fp64, fp32, damped, n;
            long long cells;
            if (scanf("%d %d %d %d %lld", &fp64, &fp32, &damped, &n, &cells) != 5) return 1;
            printf("%d\n", (int)applies_dense(fp64 != 0, fp32 != 0, damped != 0, n, cells));
        } else if (!strcmp(what, "buffers")) {
            // one handle's buffer: "n<bytes>" needs room, "c<bytes>" the same inside a capture of the
            // library, "u<bytes>" inside another one, "g" a graph was made, "d" one is destroyed;
            // prints the buffers in use, freed and set aside in order
            struct Mem {
                int next = 1, settled = 0;
                std::vector<long> freed;
                int settle() { ++settled; return 0; }
                void release(void* p) { freed.push_back((long)p); }
                int acquire(void** p, size_t) { *p = (void*)(long)next++; return 0; }
            } mem;
            Captures c;
            GrowBuf b;
            char op[64];
            while (scanf("%63s", op) == 1 && strcmp(op, "end")) {
                const size_t need = strtoull(op + 1, nullptr, 10);
                if (op[0] == 'g') ++c.graphs;
                if (op[0] == 'd')
                    for (void* p : c.end_graph()) mem.release(p);
                if (op[0] == 'n' || op[0] == 'c' || op[0] == 'u') {
                    c.own = op[0] == 'c';
                    if (grow(&b, need, &c, mem)) return 1;
                    if (op[0] != 'n') c.see(&b);
                    c.own = false;
                }
            }
            printf("%ld |", (long)b.p);
            for (long p : mem.freed) printf(" %ld", p);
            printf(" |");
            for (void* p : c.kept) printf(" %ld", (long)p);
            printf(" | %d\n", mem.settled);
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


# buffers are numbered as they are made: the one in use | freed | set aside | waits before a free
@pytest.mark.parametrize("ops,want", [
    ("n8 n4 n8", "1 | | | 0"),
    ("n8 n16", "2 | 1 | | 1"),                          # no capture: freed once nothing uses it
    ("n8 g c8 n16", "2 | | 1 | 0"),                     # a live graph holds the first
    ("n8 g c8 n16 n32", "3 | 2 | 1 | 1"),               # the second was never captured
    ("n8 g c8 n16 g c16 n32", "3 | | 1 2 | 0"),
    ("n8 g c8 n16 d", "2 | 1 | | 0"),                   # its graph is gone
    ("n8 g c8 n16 g c16 n32 d", "3 | | 1 2 | 0"),       # one of two graphs is left
    ("n8 g c8 n16 g c16 n32 d d", "3 | 1 2 | | 0"),
    ("n8 g c8 d n16", "2 | 1 | | 1"),                   # captured by a graph that no longer lives
    ("n8 u8 n16 g d", "2 | | 1 | 0"),                   # somebody else's capture: until the handle goes
])
def test_buffers_of_live_graphs_are_not_freed(plan, ops, want):
    assert " ".join(plan("buffers " + ops + " end")) == want


# vertices, FP64, dense inverse, damped, cells, evaluation on 152 SMs: the edges of the rule
@pytest.mark.parametrize("mesh,want", [
    ((642, 0, 1, 0, 152, 0), 512), ((642, 0, 1, 0, 153, 0), 256), ((642, 0, 1, 0, 304, 0), 256),
    ((642, 0, 1, 0, 305, 0), 512), ((642, 0, 1, 0, 456, 0), 512), ((642, 0, 1, 0, 457, 0), 256),
    ((642, 0, 1, 0, 620, 0), 256), ((642, 0, 1, 0, 16384, 0), 256), ((642, 0, 1, 1, 620, 0), 512),
    ((642, 0, 1, 1, 1000, 0), 512), ((642, 0, 1, 1, 1400, 0), 256),
    ((1026, 0, 0, 0, 304, 0), 256), ((1026, 0, 0, 0, 400, 0), 512), ((1026, 0, 0, 0, 700, 0), 512),
    ((1026, 0, 0, 0, 930, 0), 256), ((2562, 0, 0, 0, 400, 0), 512),
    ((258, 0, 1, 0, 152, 0), 512), ((258, 0, 1, 0, 304, 0), 256), ((258, 0, 1, 0, 305, 0), 128),
    ((258, 0, 1, 1, 400, 0), 128), ((384, 0, 1, 0, 400, 0), 128), ((385, 0, 1, 0, 400, 0), 512),
    ((1026, 0, 0, 0, 304, 1), 512), ((642, 0, 1, 0, 304, 1), 256), ((258, 0, 1, 0, 400, 1), 128),
    ((320, 1, 0, 0, 1, 0), 128), ((321, 1, 0, 0, 152, 0), 512), ((642, 1, 0, 0, 153, 0), 128), ((1026, 1, 0, 0, 9, 1), 512),
])
def test_block_sizes(plan, mesh, want):
    assert int(plan("threads %d %d %d %d %d %d" % mesh)[0]) == want


# FP64, FP32, damped, vertices, cells of the launch (BF16 and TF32 handles are neither FP64 nor FP32)
@pytest.mark.parametrize("case,want", [
    ((0, 1, 0, 700, 1), 1), ((0, 1, 0, 700, 16384), 1), ((0, 0, 0, 700, 16384), 1), ((0, 1, 1, 642, 1), 1),
    ((0, 1, 0, 701, 8), 1), ((0, 1, 0, 701, 9), 0), ((0, 1, 0, 1100, 8), 1), ((0, 1, 0, 1101, 1), 0),
    ((0, 0, 0, 701, 1), 0), ((0, 1, 1, 701, 1), 0), ((1, 0, 0, 66, 1), 0),
])
def test_dense_inverse_by_mesh(plan, case, want):
    assert int(plan("dense %d %d %d %d %d" % case)[0]) == want
