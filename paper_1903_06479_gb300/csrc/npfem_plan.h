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
// factor.  A matter of the mesh alone, so that a cell's arithmetic does not depend on the
// other cells of its call: the two differ in the order of their sums.  At 642 vertices the
// inverse is 1.65 MB from L2 in 48.5 K cycles, the factor 0.47 MB in eleven steps in 41 K, and
// a population takes the same time with either (1520 cells 1869 / 1726 us, 3001 cells of 258
// 2.38 / 2.99 ms); above, the factor wins at every count (FP32, dense / sparse: DENSEFIGS).
constexpr int kDenseVerts = 700;

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
