// Host-side, once-per-topology sparse factorisation of H~ in FP64 (not on the timed
// path): nested dissection of the mesh and a block LDL^T over its separator tree, laid
// out for solve_sparse() in npfem_cell.cuh.
//
// H~ couples a vertex with its two-ring, so a closed surface mesh splits by short rings
// of vertices (separators): 642 vertices need 92 K factor entries against 412 K of the
// dense inverse, 2562 vertices 0.5 M against 6.6 M.  For a node k of the tree with
// vertices S and boundary B (the ancestors' vertices its subtree touches), eliminating
// the subtree leaves the frontal matrix F; with D = F_SS^-1 and W = D F_SB,
//   forward:  t_S = q_S - sum over descendants d of W_d^T t_d   (deepest level first)
//   backward: x_S = D t_S - W x_B                               (root first)
// Both are written as rows of groups of four consecutive positions (zero-filled): a lane
// reads one group (16 bytes in FP32) at a time.  The rows of a step (a level of one
// sweep) are cut into slices of one warp, stored in the order the lanes read them.
#include <math.h>

#include <algorithm>
#include <numeric>
#include <string>

#include "npfem_internal.h"

namespace npfem {
namespace {

struct Node {
    std::vector<int> S, B;      // vertices of the node; boundary vertices by position
    std::vector<int> child;
    int depth = 0, pos = 0;     // first position of S
    std::vector<double> D, W;   // [s][s], [s][b]
    std::vector<double> U;      // [b][b] update for the parent (released once used)
};

struct Tree {
    const HostTopo& H;
    const double* X;            // rest positions [n][3]
    int leaf;
    std::vector<Node> nodes;    // post-order: children before their parent
    std::vector<int> mark;

    Tree(const HostTopo& h, const double* x, int leaf_) : H(h), X(x), leaf(leaf_), mark(h.n, 0) {}

    // Splits idx by a plane: left part, separator (the right's vertices adjacent to the
    // left), rest of the right.  Returns a cost (estimated factor work).
    double split(const std::vector<int>& order, size_t h, bool flip, std::vector<int>* sep, std::vector<int>* a,
                 std::vector<int>* b)
    {
        a->clear();
        b->clear();
        sep->clear();
        const size_t m = order.size();
        for (size_t q = 0; q < m; ++q) mark[order[q]] = ((q < h) != flip) ? 1 : 2;
        for (int v : order) {
            if (mark[v] == 1) {
                a->push_back(v);
                continue;
            }
            bool touch = false;
            for (int p = H.L_ptr[v]; p < H.L_ptr[v + 1] && !touch; ++p) touch = mark[H.L_idx[p]] == 1;
            (touch ? sep : b)->push_back(v);
        }
        for (int v : order) mark[v] = 0;
        const double s = (double)sep->size(), big = (double)std::max(a->size(), b->size());
        return 0.5 * s * s + 0.6 * big * sqrt(big);
    }

    // The best plane cut of idx: separator (along the cut) and the two sides.
    void cut(const std::vector<int>& idx, std::vector<int>* S, std::vector<int>* side_a, std::vector<int>* side_b)
    {
        // planes normal to the axes and some diagonals, at three positions each, either
        // side giving the separator
        static const double dirs[7][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {1, 1, 0}, {1, -1, 0}, {1, 1, 1}, {1, -1, 1}};
        static const double frac[3] = {0.5, 0.45, 0.55};
        std::vector<int> order(idx), sep, a, b, bs;
        double best = -1.0;
        int bdir = 0;
        for (int d = 0; d < 7; ++d) {
            std::vector<std::pair<double, int>> key;
            for (int v : idx) key.push_back({X[3 * v] * dirs[d][0] + X[3 * v + 1] * dirs[d][1] + X[3 * v + 2] * dirs[d][2], v});
            std::sort(key.begin(), key.end());
            for (size_t q = 0; q < key.size(); ++q) order[q] = key[q].second;
            for (double f : frac) {
                const size_t h = std::max<size_t>(1, (size_t)(f * order.size()));
                for (int flip = 0; flip < 2; ++flip) {
                    const double c = split(order, h, flip != 0, &sep, &a, &b);
                    if (best < 0.0 || c < best) {
                        best = c;
                        bdir = d;
                        bs.swap(sep);
                        side_a->swap(a);
                        side_b->swap(b);
                    }
                }
            }
        }
        // separator vertices along the cut (by angle about the mesh's centre in the
        // cutting plane), so that what a subtree touches of it is nearly consecutive
        double u[3], w[3];
        const double* dn = dirs[bdir];
        const int ax = fabs(dn[0]) <= fabs(dn[1]) && fabs(dn[0]) <= fabs(dn[2]) ? 0 : (fabs(dn[1]) <= fabs(dn[2]) ? 1 : 2);
        const double e[3] = {ax == 0 ? 1.0 : 0.0, ax == 1 ? 1.0 : 0.0, ax == 2 ? 1.0 : 0.0};
        for (int c = 0; c < 3; ++c) u[c] = dn[(c + 1) % 3] * e[(c + 2) % 3] - dn[(c + 2) % 3] * e[(c + 1) % 3];
        for (int c = 0; c < 3; ++c) w[c] = dn[(c + 1) % 3] * u[(c + 2) % 3] - dn[(c + 2) % 3] * u[(c + 1) % 3];
        const double nu = sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), nw = sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
        std::vector<std::pair<double, int>> ang;
        for (int v : bs) {
            double pu = 0.0, pw = 0.0;
            for (int c = 0; c < 3; ++c) {
                pu += X[3 * v + c] * u[c] / nu;
                pw += X[3 * v + c] * w[c] / nw;
            }
            ang.push_back({atan2(pw, pu), v});
        }
        std::sort(ang.begin(), ang.end());
        for (auto& q : ang) S->push_back(q.second);
    }

    int build(std::vector<int> idx, int depth)
    {
        Node nd;
        nd.depth = depth;
        if ((int)idx.size() <= leaf) {
            nd.S = std::move(idx);
        } else {
            std::vector<int> a, b;
            cut(idx, &nd.S, &a, &b);
            if (!a.empty()) nd.child.push_back(build(std::move(a), depth + 1));
            if (!b.empty()) nd.child.push_back(build(std::move(b), depth + 1));
        }
        nodes.push_back(std::move(nd));
        return (int)nodes.size() - 1;
    }
};

// In-place inverse of a symmetric positive definite matrix (symmetric sweeps on the lower
// triangle, then mirrored); false when a pivot is not positive.
bool invert_spd(std::vector<double>& A, int n)
{
    std::vector<double> c(n);
    for (int k = 0; k < n; ++k) {
        const double piv = A[(size_t)k * n + k];
        if (!(piv > 0.0)) return false;
        const double p = 1.0 / piv;
        for (int i = 0; i < n; ++i) c[i] = i >= k ? A[(size_t)i * n + k] : A[(size_t)k * n + i];
        for (int i = 0; i < n; ++i) {
            double* Ai = &A[(size_t)i * n];
            const double f = c[i] * p;
            for (int j = 0; j <= i; ++j) Ai[j] -= f * c[j];
        }
        for (int i = k + 1; i < n; ++i) A[(size_t)i * n + k] = c[i] * p;
        for (int j = 0; j < k; ++j) A[(size_t)k * n + j] = c[j] * p;
        A[(size_t)k * n + k] = -p;
    }
    for (int i = 0; i < n; ++i)
        for (int j = 0; j <= i; ++j) {
            A[(size_t)i * n + j] = -A[(size_t)i * n + j];
            A[(size_t)j * n + i] = A[(size_t)i * n + j];
        }
    return true;
}

}  // namespace

int build_sparse_factor(const HostTopo& H, const double* rest, double mass_scale, double l_scale, SparseHost* out,
                        SparseHost* out_cluster, std::string* err)
{
    const int n = H.n;
    Tree T(H, rest, kSparseLeaf);
    std::vector<int> all(n);
    std::iota(all.begin(), all.end(), 0);
    T.build(std::move(all), 0);
    std::vector<Node>& N = T.nodes;

    SparseHost* o = out;
    // positions (every node's vertices padded to a multiple of four)
    std::vector<int> pos(n, -1), owner(n, -1);
    o->perm.clear();
    int depth = 0;
    for (size_t k = 0; k < N.size(); ++k) {
        N[k].pos = (int)o->perm.size();
        for (int v : N[k].S) {
            pos[v] = (int)o->perm.size();
            owner[v] = (int)k;
            o->perm.push_back(v);
        }
        while (o->perm.size() & 3) o->perm.push_back(-1);
        depth = std::max(depth, N[k].depth);
    }
    o->npos = (int)o->perm.size();
    if (2 * (long long)o->npos > 4 * 65535LL) {
        *err = "mesh too large for the sparse factor's 16-bit groups";
        return NPFEM_ERR_INVALID_ARG;
    }

    // boundaries and numeric factorisation, children first
    std::vector<int> loc(n, -1);
    for (size_t k = 0; k < N.size(); ++k) {
        Node& nd = N[k];
        const int s = (int)nd.S.size();
        std::vector<int> bset;
        for (int v : nd.S)
            for (int p = H.L_ptr[v]; p < H.L_ptr[v + 1]; ++p)
                if (pos[H.L_idx[p]] >= nd.pos + s) bset.push_back(H.L_idx[p]);
        for (int c : nd.child)
            for (int v : N[c].B)
                if (owner[v] != (int)k) bset.push_back(v);
        std::sort(bset.begin(), bset.end(), [&](int p, int q) { return pos[p] < pos[q]; });
        bset.erase(std::unique(bset.begin(), bset.end()), bset.end());
        nd.B = bset;
        const int b = (int)bset.size(), m = s + b;
        for (int q = 0; q < s; ++q) loc[nd.S[q]] = q;
        for (int q = 0; q < b; ++q) loc[bset[q]] = s + q;
        std::vector<double> F((size_t)m * m, 0.0);
        for (int q = 0; q < s; ++q) {
            const int v = nd.S[q];
            F[(size_t)q * m + q] += mass_scale * H.mass[v];
            for (int p = H.L_ptr[v]; p < H.L_ptr[v + 1]; ++p) {
                const int w = H.L_idx[p];
                if (pos[w] < nd.pos) continue;  // eliminated below
                const int r = loc[w];
                const double val = l_scale * H.L_val[p];
                F[(size_t)q * m + r] += val;
                if (r >= s) F[(size_t)r * m + q] += val;
            }
        }
        for (int c : nd.child) {
            const int bc = (int)N[c].B.size();
            for (int i = 0; i < bc; ++i)
                for (int j = 0; j < bc; ++j)
                    F[(size_t)loc[N[c].B[i]] * m + loc[N[c].B[j]]] += N[c].U[(size_t)i * bc + j];
            std::vector<double>().swap(N[c].U);
        }
        nd.D.assign((size_t)s * s, 0.0);
        for (int i = 0; i < s; ++i)
            for (int j = 0; j < s; ++j) nd.D[(size_t)i * s + j] = F[(size_t)i * m + j];
        if (!invert_spd(nd.D, s)) {
            *err = "H~ is not positive definite";
            return NPFEM_ERR_NOT_SPD;
        }
        nd.W.assign((size_t)s * b, 0.0);
        for (int i = 0; i < s; ++i)
            for (int r = 0; r < s; ++r) {
                const double d = nd.D[(size_t)i * s + r];
                const double* Fr = &F[(size_t)r * m + s];
                double* Wi = nd.W.data() + (size_t)i * b;
                for (int j = 0; j < b; ++j) Wi[j] += d * Fr[j];
            }
        nd.U.assign((size_t)b * b, 0.0);
        for (int i = 0; i < b; ++i) {
            // symmetric: the lower triangle, mirrored
            double* Ui = nd.U.data() + (size_t)i * b;
            for (int j = 0; j <= i; ++j) Ui[j] = F[(size_t)(s + i) * m + s + j];
            for (int r = 0; r < s; ++r) {
                const double f = F[(size_t)r * m + s + i];
                const double* Wr = nd.W.data() + (size_t)r * b;
                for (int j = 0; j <= i; ++j) Ui[j] -= f * Wr[j];
            }
            for (int j = 0; j < i; ++j) nd.U[(size_t)j * b + i] = Ui[j];
        }
        for (int v : nd.S) loc[v] = -1;
        for (int v : bset) loc[v] = -1;
    }

    // rows by step: forward levels deepest first (the leaves need none), backward root first
    std::vector<std::vector<std::pair<int, int>>> below(n);  // (node, column of W) per boundary vertex
    for (size_t k = 0; k < N.size(); ++k)
        for (size_t j = 0; j < N[k].B.size(); ++j) below[N[k].B[j]].push_back({(int)k, (int)j});
    // for the schedules [sched0, sched1)
    auto lay_out = [&](SparseHost* o, int warps, int sched0, int sched1) {
    o->rows.clear();
    o->idx.clear();
    o->val.clear();
    o->slices.clear();
    o->step_begin.assign(1, 0);
    struct Row {
        int pos, forward;
        std::vector<int> groups;
        std::vector<double> val;
    };
    std::vector<Row> step;
    std::vector<double> dense(2 * (size_t)o->npos, 0.0);
    std::vector<char> used(o->npos / 2, 0);
    std::vector<int> groups;
    auto put = [&](int at, double v) {
        dense[at] = v;
        if (!used[at >> 2]) {
            used[at >> 2] = 1;
            groups.push_back(at >> 2);
        }
    };
    auto emit = [&](int p, int forward) {
        Row r;
        r.pos = p;
        r.forward = forward;
        std::sort(groups.begin(), groups.end());
        for (int g : groups) {
            for (int q = 0; q < 4; ++q) {
                r.val.push_back(dense[4 * (size_t)g + q]);
                dense[4 * (size_t)g + q] = 0.0;
            }
            used[g] = 0;
        }
        r.groups.swap(groups);
        step.push_back(std::move(r));
    };
    // a step's rows in slices of one warp: 32 / 2^lg rows of 2^lg lanes each, padded to the
    // slice's longest row
    auto close = [&]() {
        if (step.empty()) return;
        size_t share = 1;
        auto lg_of = [&](const Row& r) {
            int lg = 0;
            while (lg < 5 && (share << lg) < r.groups.size()) ++lg;
            return lg;
        };
        // the smallest share of groups per lane that gives every warp at most one slice
        for (; share < (size_t)kSparseMaxIters; ++share) {
            int cnt[6] = {0, 0, 0, 0, 0, 0}, slices = 0;
            for (const Row& r : step) ++cnt[lg_of(r)];
            for (int lg = 0; lg < 6; ++lg) slices += ((cnt[lg] << lg) + 31) >> 5;
            if (slices <= warps) break;
        }
        std::stable_sort(step.begin(), step.end(), [&](const Row& p, const Row& q) {
            const int lp = lg_of(p), lq = lg_of(q);
            return lp != lq ? lp > lq : p.groups.size() > q.groups.size();
        });
        for (size_t r = 0; r < step.size();) {
            const int lg = lg_of(step[r]), per = 32 >> lg;
            size_t e = r;
            int iters = 0;
            while (e < step.size() && (int)(e - r) < per && lg_of(step[e]) == lg) {
                iters = std::max(iters, (int)((step[e].groups.size() + (1u << lg) - 1) >> lg));
                ++e;
            }
            SparseHost::Slice sl;
            sl.base = (int)(o->idx.size() / 32);
            sl.iters = iters;
            sl.lg = lg;
            sl.row = (int)(o->rows.size() / 2);
            o->idx.resize(o->idx.size() + 32 * (size_t)iters, 0);
            o->val.resize(o->val.size() + 128 * (size_t)iters, 0.0);
            for (int q = 0; q < per; ++q) {
                if (r + q >= e) {
                    o->rows.push_back(-1);
                    o->rows.push_back(0);
                    continue;
                }
                const Row& w = step[r + q];
                o->rows.push_back(w.pos);
                o->rows.push_back(w.forward ? -1 : o->perm[w.pos]);
                for (size_t g = 0; g < w.groups.size(); ++g) {
                    const size_t at = ((size_t)sl.base + (g >> lg)) * 32 + ((size_t)q << lg) + (g & ((1u << lg) - 1));
                    o->idx[at] = (unsigned short)w.groups[g];
                    for (int k = 0; k < 4; ++k) o->val[4 * at + k] = w.val[4 * g + k];
                }
            }
            o->slices.push_back(sl);
            r = e;
        }
        o->step_begin.push_back((int)o->slices.size());
        step.clear();
    };
    for (int l = depth - 1; l >= 0; --l) {
        for (size_t k = 0; k < N.size(); ++k) {
            if (N[k].depth != l || N[k].child.empty()) continue;
            for (int v : N[k].S) {
                if (below[v].empty()) continue;
                for (auto& d : below[v]) {
                    const Node& c = N[d.first];
                    for (size_t r = 0; r < c.S.size(); ++r) put(c.pos + (int)r, -c.W[r * c.B.size() + d.second]);
                }
                emit(pos[v], 1);
            }
        }
        close();
    }
    for (int l = 0; l <= depth; ++l) {
        for (size_t k = 0; k < N.size(); ++k) {
            if (N[k].depth != l) continue;
            const Node& c = N[k];
            const int s = (int)c.S.size(), b = (int)c.B.size();
            for (int i = 0; i < s; ++i) {
                for (int j = 0; j < s; ++j) put(c.pos + j, c.D[(size_t)i * s + j]);
                for (int j = 0; j < b; ++j) put(o->npos + pos[c.B[j]], -c.W[(size_t)i * b + j]);
                emit(c.pos + i, 0);
            }
        }
        close();
    }

    // schedules: the warps take a step's slices in turn; the last of a step ends in a barrier
    for (int v = sched0; v < sched1; ++v) {
        const int nw = sparse_sched_warps(v);
        std::vector<int>& sc = o->sched[v];
        sc.clear();
        for (size_t st = 0; st + 1 < o->step_begin.size(); ++st) {
            const int b = o->step_begin[st], e = o->step_begin[st + 1];
            for (int q = b; q < e; q += nw)
                for (int w = 0; w < nw; ++w) {
                    SparseHost::Slice sl = {0, 0, 0, 0};
                    if (q + w < e) sl = o->slices[q + w];
                    sc.push_back(sl.base);
                    sc.push_back(sl.iters);
                    sc.push_back(sl.lg | (q + nw >= e ? 256 : 0));
                    sc.push_back(sl.row);
                }
        }
    }
    };
    lay_out(out, kSparseWarps, 0, 3);
    if (out_cluster) {
        out_cluster->npos = out->npos;
        out_cluster->perm = out->perm;
        lay_out(out_cluster, kSparseWarpsCluster, 1, kSparseScheds);
    }
    return 0;
}

}  // namespace npfem
