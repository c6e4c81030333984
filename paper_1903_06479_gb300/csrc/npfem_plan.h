// Host-side decisions of a step that need no CUDA call: what the groups of a call take from
// which handle, where their carried pairs lie, and when a buffer may be freed.
#pragma once

#include <cstddef>
#include <mutex>
#include <vector>

#ifdef __CUDACC__
#define NPFEM_HD __host__ __device__
#else
#define NPFEM_HD
#endif

namespace npfem {

constexpr int kMaxGroups = 8;  // meshes per npfem_step launch

// Carried L-BFGS pairs of one cell, in elements of the state type: the solver's history
// ring as the last solve left it: [0] the pair count, [1] the ring head, [2] that
// solve's iterations, from [4] the inner products s_i^T y_j by ring slot (m x m, padded
// to a multiple of 4), then the s vectors of ring slots 0..m-1 and the y vectors
// ([3][n_pad] each).  The pairs are used while that solve took at most kCarryMaxIters
// iterations.
constexpr int kCarryMaxIters = 3;
NPFEM_HD inline long long carry_head_elems(int m) { return 4 + (((long long)m * m + 3) & ~3LL); }
NPFEM_HD inline long long carry_rec_elems(int n_pad, int m) { return carry_head_elems(m) + 2LL * m * 3 * n_pad; }

// Meshes whose FP32 cells apply the dense inverse; finer ones (and FP64) apply the sparse
// factor.  A matter of the mesh, so that a cell's arithmetic does not depend on the other
// groups of its call: the two differ in the order of their sums.  At 642 vertices the inverse is
// 1.65 MB from L2 in 48.5 K cycles, the factor 0.47 MB in eleven steps in 41 K, and a population
// takes the same time with either (1520 cells 1869 / 1726 us, 3001 cells of 258 2.38 / 2.99 ms);
// at 1026 vertices (37 cells, four steps) 2.65 / 2.24 ms.
//
// One exception: launches of at most kDenseFewCells cells of an FP32 handle keep the dense
// inverse up to kDenseFewVerts vertices, and its time (1026 x 1, four steps, 2418 us; the
// factor 2095).  Another order of the sums moves velocities by about 6e-8 um/us.  Among many
// cells that is 3e-6 of the fastest; one slow cell's velocities moved by 1e-4 of their size
// (1026 x 1 at a low shear rate, where either order is 2e-3 from FP64), and a few cells may all
// be slow.  Eight cells drawn from the shear rates of 10 to 1000 / s are all below 100 / s once in
// 10^8.  BF16 and TF32 handles, whose contractions were never these, take the factor.
constexpr int kDenseVerts = 700, kDenseFewVerts = 1100, kDenseFewCells = 8;

// Do the cells of a mesh of n vertices apply the dense inverse in a SIMT launch of `cells`?
// (fp64, fp32: the handle's precision is NPFEM_PREC_FP64, NPFEM_PREC_FP32.)
inline bool applies_dense(bool fp64, bool fp32, bool damped, int n, long long cells)
{
    if (fp64 || n > kDenseFewVerts) return false;
    return n <= kDenseVerts || (fp32 && !damped && cells <= kDenseFewCells);
}

// Block size of a SIMT group: a mesh's evaluation keeps about n / 32 warps busy and most of
// its phases are latency-bound, so when every SM has several cells to solve, two blocks of
// 256 threads or four of 128 per SM overlap each other's phases (vectors that then do not
// fit in shared memory go to global memory, L2).  Measured, FP32, three steps of 3040
// cells, 512 / 256 / 128 threads: 66 vertices 296 / 161 / 107 us, 258: 1087 / 688 / 557,
// 362: 1223 / 830 / 804; 1520 cells: 642: 2048 / 1726 / 1901, 1026: 5235 / 4758 / 6816;
// 400 cells of 2562: 7677 / 12086.  With at most a cell per SM a cell's own latency counts:
// 40 cells of 66 vertices 33 / 30 / 31 us, 162: 64 / 66 / 79, 258: 68 / 78 / 105.  FP64 is
// bound by the FP64 pipe; four blocks hide its latencies best at every size (160 cells of
// 66 vertices 972 / 705 / 573 us, 258: 5321 / 4846 / 4666).
//
// Cells come in rounds of one per resident block, and a pair of cells on an SM takes 1.65
// (dense inverse), 1.75 (sparse factor) or 1.8 (damped) times one cell's time, so an odd
// number of rounds of single cells can be the shorter: 512 / 256 threads, two steps, 642 x
// 310 1260 / 1318 us, 642 x 456 1267 / 1451, 1026 x 400 3230 / 3810, 1026 x 700 5354 / 5683;
// but 642 x 304 866 / 773, 642 x 620 2067 / 2021, 1026 x 608 4331 / 4017, 1026 x 930 7342 /
// 7248.
struct SimtMesh {
    int n;
    bool fp64, dense, damped;
};

inline int simt_threads(const SimtMesh& m, long long cells, long long sms)
{
    if (m.fp64) return cells > sms || m.n <= 320 ? 128 : 512;
    if (m.n <= 384 && cells > 2 * sms) return 128;
    if (m.n > 1200 || cells <= sms) return 512;
    const double pair = m.damped ? 1.8 : (m.dense ? 1.65 : 1.75);
    const long long singles = (cells + sms - 1) / sms, pairs = (cells + 2 * sms - 1) / (2 * sms);
    return m.n > 384 && (double)singles < pair * (double)pairs ? 512 : 256;
}

// The same for an evaluation of the objective, which applies no inverse: finer meshes gain
// nothing from smaller blocks, whose vectors spill (evaluations of 1026 x 160, 400 and 600
// cells, 512 / 256 threads: 78 / 78, 113 / 138, 147 / 146 us; 786: 69 / 63, 98 / 110, 126 / 114;
// 642: 54 / 48, 77 / 78, 98 / 84).
inline int eval_threads(const SimtMesh& m, long long cells, long long sms)
{
    return !m.fp64 && m.n > kDenseVerts ? 512 : simt_threads(m, cells, sms);
}

// One group of a call: its mesh, its own handle's L-BFGS window, and whether its cells go to
// the tensor-core cluster kernel (with its own handle's options).
struct PlanGroup {
    int n, n_pad, window;
    long long cells;
    bool clusters;
};

// The first group with cells for the SIMT launches, whose handle's options they take (-1: none).
inline int simt_lead(const std::vector<PlanGroup>& groups)
{
    for (size_t g = 0; g < groups.size(); ++g)
        if (groups[g].cells > 0 && !groups[g].clusters) return (int)g;
    return -1;
}

// Where every group's carried pairs lie in the call's buffer, in elements: its first record and
// the size of one, by the window of the options its launch takes.  The buffer is sized and
// the launches are set up by this alone (handles of one call may differ in their window).
struct CarryPlan {
    std::vector<int> window;
    std::vector<long long> off, rec;
    long long total = 0;
};

inline CarryPlan plan_carry(const std::vector<PlanGroup>& groups)
{
    CarryPlan c;
    const int lead = simt_lead(groups);
    for (const PlanGroup& g : groups) {
        c.window.push_back(g.clusters || lead < 0 ? g.window : groups[lead].window);
        c.rec.push_back(carry_rec_elems(g.n_pad, c.window.back()));
        c.off.push_back(c.total);
        c.total += c.rec.back() * g.cells;
    }
    return c;
}

// A device buffer that grows on demand.  A captured graph's kernels keep its address, so what a
// capture has seen is not freed when a larger buffer takes its place (its old address stays
// good for the graph's replays): it is set aside until the last graph on the handle is gone,
// or, when a capture that is not the library's own saw it, until the handle is.
struct GrowBuf {
    void* p = nullptr;
    size_t bytes = 0;
    unsigned seen = 0;  // Captures::epoch of the last capture that saw it (0: none)
};

// Shared by a handle and its graphs (either may go first).
struct Captures {
    std::mutex mu;
    std::vector<void*> kept;  // superseded buffers that a graph may still use
    unsigned epoch = 1;
    int graphs = 0;           // live graphs of the library over the handle
    bool own = false;         // a graph of the library is being captured
    bool foreign = false;     // some other capture saw a buffer: its graph's end is not known

    void see(GrowBuf* b)
    {
        std::lock_guard<std::mutex> lk(mu);
        b->seen = epoch;
        if (!own) foreign = true;
    }

    // The graph is gone: what the caller may free now.
    std::vector<void*> end_graph()
    {
        std::lock_guard<std::mutex> lk(mu);
        std::vector<void*> out;
        if (graphs > 0) --graphs;
        if (graphs == 0 && !foreign) {
            out.swap(kept);
            ++epoch;
        }
        return out;
    }
};

// Makes room for `need` bytes (contents are lost when it grows).  mem: settle() waits until
// nothing queued uses the buffer any more, release(p), acquire(&p, bytes); both that can
// fail return nonzero.
template <typename Mem>
int grow(GrowBuf* b, size_t need, Captures* c, Mem&& mem)
{
    if (need <= b->bytes) return 0;
    if (b->p) {
        std::unique_lock<std::mutex> lk(c->mu);
        if (b->seen == c->epoch) {
            c->kept.push_back(b->p);
        } else {
            lk.unlock();
            if (int e = mem.settle()) return e;
            mem.release(b->p);
        }
        *b = GrowBuf();
    }
    if (int e = mem.acquire(&b->p, need)) {
        b->p = nullptr;
        return e;
    }
    b->bytes = need;
    return 0;
}

}  // namespace npfem
