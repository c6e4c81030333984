// C ABI of libnpfem.so (declared in include/npfem.h): handle set-up, placement of the
// per-cell solver vectors in shared or global memory, and the launches.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "npfem_internal.h"

using namespace npfem;

namespace {

thread_local std::string g_last_error;

int fail(int code, const std::string& msg)
{
    g_last_error = msg;
    return code;
}

}  // namespace

int npfem::set_error(int code, const std::string& msg) { return fail(code, msg); }

namespace npfem {
std::atomic<unsigned long long> g_launches{0};
void count_launch(unsigned long long k) { g_launches.fetch_add(k); }
}  // namespace npfem

namespace {

#define NPFEM_CUDA(call)                                                                               \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess)                                                                         \
            return fail(e_ == cudaErrorMemoryAllocation ? NPFEM_ERR_OOM : NPFEM_ERR_CUDA,              \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                           \
    } while (0)

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev)
    {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard()
    {
        int cur = -1;
        cudaGetDevice(&cur);
        if (prev >= 0 && cur != prev) cudaSetDevice(prev);
    }
};

}  // namespace


namespace {

template <typename X, typename S>
int upload(npfem_handle* h, const std::vector<S>& src, const X** out)
{
    int err = 0;
    std::vector<X> tmp(src.size());
    for (size_t i = 0; i < src.size(); ++i) tmp[i] = (X)src[i];
    X* d = h->alloc<X>(std::max<size_t>(tmp.size(), 1), &err);
    if (!d) return err;
    if (!tmp.empty()) NPFEM_CUDA(cudaMemcpy(d, tmp.data(), tmp.size() * sizeof(X), cudaMemcpyHostToDevice));
    *out = d;
    return 0;
}

template <typename T>
int upload_sparse(npfem_handle* h, const SparseHost& F, SparseDev<T>* sp)
{
    int rc;
    const int* drow = nullptr;
    if ((rc = upload(h, F.perm, &sp->perm))) return rc;
    if ((rc = upload(h, F.rows, &drow))) return rc;
    if ((rc = upload(h, F.idx, &sp->idx))) return rc;
    if ((rc = upload(h, F.val, &sp->val))) return rc;
    sp->row = reinterpret_cast<const int2*>(drow);
    sp->npos = F.npos;
    for (int v = 0; v < kSparseScheds; ++v) {
        sp->sched[v] = nullptr;
        sp->entries[v] = 0;
        if (F.sched[v].empty()) continue;
        const int* ds = nullptr;
        if ((rc = upload(h, F.sched[v], &ds))) return rc;
        sp->sched[v] = reinterpret_cast<const int4*>(ds);
        sp->entries[v] = (int)F.sched[v].size() / (4 * sparse_sched_warps(v));
    }
    return 0;
}

// The factors of H~ and, with damping, M~; empty where the cells apply dense inverses.
struct Factors {
    SparseHost system, cluster, mass;
};

template <typename T>
int fill_topo(npfem_handle* h, TopoDev<T>* tp, const Factors& F)
{
    const HostTopo& H = h->host;
    int rc;
    std::vector<unsigned short> tri4(4 * (size_t)H.nt, 0);
    for (int t = 0; t < H.nt; ++t)
        for (int a = 0; a < 3; ++a) tri4[4 * t + a] = (unsigned short)H.tri[3 * t + a];
    const unsigned short* dtri = nullptr;
    if ((rc = upload(h, tri4, &dtri))) return rc;
    tp->tri = reinterpret_cast<const ushort4*>(dtri);
    if ((rc = upload(h, H.dminv, &tp->dminv))) return rc;
    if ((rc = upload(h, H.W, &tp->W))) return rc;
    if ((rc = upload(h, H.mass, &tp->mass))) return rc;
    std::vector<double> inv_m(H.n);
    for (int i = 0; i < H.n; ++i) inv_m[i] = 1.0 / H.mass[i];
    if ((rc = upload(h, inv_m, &tp->inv_mass))) return rc;
    if ((rc = upload(h, H.bend_w, &tp->bend_w))) return rc;
    if ((rc = upload(h, H.dg_norm, &tp->dg_norm))) return rc;
    if ((rc = upload(h, H.csum, &tp->csum))) return rc;
    if ((rc = upload(h, H.nsign, &tp->nsign))) return rc;
    if ((rc = upload(h, H.ring_ptr, &tp->ring_ptr))) return rc;
    std::vector<unsigned short> ridx(H.ring_idx.begin(), H.ring_idx.end());
    if ((rc = upload(h, ridx, &tp->ring_idx))) return rc;
    if ((rc = upload(h, H.ring_c, &tp->ring_c))) return rc;
    if ((rc = upload(h, H.ring_ct, &tp->ring_ct))) return rc;
    if ((rc = upload(h, H.rest_c, &tp->rest_c))) return rc;
    tp->mlp = nullptr;
    tp->tmlp = nullptr;
    if ((rc = upload(h, H.inc_ptr, &tp->inc_ptr))) return rc;
    std::vector<unsigned> incu(H.inc_idx.begin(), H.inc_idx.end());
    if ((rc = upload(h, incu, &tp->inc_idx))) return rc;
    // Fixed-width tables: each vertex's one-ring in cyclic order r_0 .. r_{v-1} (v <= 8)
    // so that triangle (i, r_q, r_{q+1 mod v}) is incident triangle q of vertex i, in
    // the mesh's orientation.  Needs every one-ring to be one cycle of at most 8.
    std::vector<std::vector<int>> cyc(H.n);
    bool ok8 = true;
    {
        std::vector<std::vector<std::pair<int, int>>> nxt(H.n);  // (j, k) for triangles (i, j, k)
        for (int t = 0; t < H.nt; ++t)
            for (int a = 0; a < 3; ++a)
                nxt[H.tri[3 * t + a]].push_back({H.tri[3 * t + (a + 1) % 3], H.tri[3 * t + (a + 2) % 3]});
        for (int i = 0; i < H.n && ok8; ++i) {
            const int v = (int)nxt[i].size();
            if (v > 8 || v != H.ring_ptr[i + 1] - H.ring_ptr[i]) {
                ok8 = false;
                break;
            }
            int j = nxt[i][0].first;
            for (int q = 0; q < v; ++q) {
                cyc[i].push_back(j);
                int k = -1;
                for (const auto& e : nxt[i])
                    if (e.first == j) k = e.second;
                if (k < 0) {
                    ok8 = false;
                    break;
                }
                j = k;
            }
            if (ok8 && j != nxt[i][0].first) ok8 = false;
            if (ok8) {
                std::vector<int> sc(cyc[i]);
                std::sort(sc.begin(), sc.end());
                ok8 = std::adjacent_find(sc.begin(), sc.end()) == sc.end();
            }
        }
    }
    tp->k8 = ok8 ? 1 : 0;
    tp->ring8_idx = nullptr;
    tp->ring8_c = tp->ring8_ct = nullptr;
    if (tp->k8) {
        std::vector<unsigned short> r8(8 * (size_t)H.n);
        std::vector<double> c8(8 * (size_t)H.n, 0.0), ct8(8 * (size_t)H.n, 0.0);
        for (int i = 0; i < H.n; ++i) {
            for (int q = 0; q < 8; ++q) r8[8 * i + q] = (unsigned short)i;
            for (int q = 0; q < (int)cyc[i].size(); ++q) {
                const int j = cyc[i][q];
                r8[8 * i + q] = (unsigned short)j;
                for (int p = H.ring_ptr[i]; p < H.ring_ptr[i + 1]; ++p)
                    if (H.ring_idx[p] == j) {
                        c8[8 * i + q] = H.ring_c[p];
                        ct8[8 * i + q] = H.ring_ct[p];
                    }
            }
        }
        // slot of each triangle corner in its vertex's cyclic ring, packed 3 bits per
        // corner into the fourth component of the triangle's index record
        for (int t = 0; t < H.nt; ++t) {
            unsigned packed = 0;
            for (int a = 0; a < 3; ++a) {
                const int i = H.tri[3 * t + a], j = H.tri[3 * t + (a + 1) % 3];
                int slot = 0;
                while (cyc[i][slot] != j) ++slot;
                packed |= (unsigned)slot << (3 * a);
            }
            tri4[4 * t + 3] = (unsigned short)packed;
        }
        NPFEM_CUDA(cudaMemcpy(const_cast<unsigned short*>(dtri), tri4.data(), tri4.size() * sizeof(unsigned short),
                              cudaMemcpyHostToDevice));
        if ((rc = upload(h, r8, &tp->ring8_idx))) return rc;
        if ((rc = upload(h, c8, &tp->ring8_c))) return rc;
        if ((rc = upload(h, ct8, &tp->ring8_ct))) return rc;
    }
    tp->n = H.n;
    tp->nt = H.nt;
    tp->n_pad = h->n_pad;
    tp->nnz = (int)H.ring_idx.size();
    tp->l_ptr = nullptr;
    tp->l_idx = nullptr;
    tp->l_val = nullptr;
    tp->beta_h = (T)(h->mat.beta_D / h->dt);
    if (h->mat.beta_D > 0.0) {
        if ((rc = upload(h, H.L_ptr, &tp->l_ptr))) return rc;
        std::vector<unsigned short> lidx(H.L_idx.begin(), H.L_idx.end());
        if ((rc = upload(h, lidx, &tp->l_idx))) return rc;
        if ((rc = upload(h, H.L_val, &tp->l_val))) return rc;
    }
    tp->ainv_lp = nullptr;
    tp->h_ptr = nullptr;
    tp->h_idx = nullptr;
    tp->h_val = nullptr;
    if (F.system.npos && (rc = upload_sparse(h, F.system, &tp->sp))) return rc;
    if (F.cluster.npos && (rc = upload_sparse(h, F.cluster, &tp->spc))) return rc;
    if (F.mass.npos && (rc = upload_sparse(h, F.mass, &tp->spm))) return rc;
    tp->C = (T)h->mat.C;
    tp->B = (T)h->mat.B;
    tp->Dsk = (T)h->mat.D;
    tp->kvol = (T)h->mat.k_vol;
    tp->h = (T)h->dt;
    tp->inv_h2 = (T)(1.0 / (h->dt * h->dt));
    tp->inertia_scale = (T)(1.0 + h->dt * h->mat.alpha_D);
    tp->kappa = (T)h->mat.kappa;
    tp->lbar = (T)H.lbar;
    tp->inv_lbar = (T)(1.0 / H.lbar);
    tp->V0 = H.V0;
    tp->V0hi = (T)H.V0;
    tp->V0lo = (T)(H.V0 - (double)tp->V0hi);
    return 0;
}

int check_opts(const npfem_opts* o)
{
    if (o->precision < NPFEM_PREC_FP64 || o->precision > NPFEM_PREC_BF16)
        return fail(NPFEM_ERR_INVALID_ARG, "opts.precision must be one of NPFEM_PREC_*");
    if (o->lbfgs_m < 0 || o->lbfgs_m > kMaxHistory)
        return fail(NPFEM_ERR_INVALID_ARG, "opts.lbfgs_m must be in 0..8");
    if (o->max_iter < 0 || o->max_halvings < 0 || o->max_halvings > 60)
        return fail(NPFEM_ERR_INVALID_ARG, "opts.max_iter must be >= 0 and max_halvings in 0..60");
    if (!(o->tol >= 0.0) || !(o->c1 > 0.0 && o->c1 < 1.0) || !(o->c2 > o->c1 && o->c2 < 1.0) ||
        !(o->armijo_noise >= 0.0))
        return fail(NPFEM_ERR_INVALID_ARG, "opts: need tol >= 0, 0 < c1 < c2 < 1, armijo_noise >= 0");
    if (o->refine < 0 || o->refine > 1) return fail(NPFEM_ERR_INVALID_ARG, "opts.refine must be 0 or 1");
    if (o->fill_idle_sms < 0 || o->fill_idle_sms > 1)
        return fail(NPFEM_ERR_INVALID_ARG, "opts.fill_idle_sms must be 0 or 1");
    if (o->warm_history < 0 || o->warm_history > 2)
        return fail(NPFEM_ERR_INVALID_ARG, "opts.warm_history must be 0, 1 or 2");
    return 0;
}

// What the block-size rule (npfem_plan.h) asks about a mesh.
SimtMesh simt_mesh(const npfem_handle* h)
{
    return {h->n, h->precision == NPFEM_PREC_FP64, h->n <= kDenseVerts, h->mat.beta_D > 0.0};
}

// Collision planes of a call (those installed on its first handle), from the first vertex of
// the launch's x on.
struct Planes {
    const float* at = nullptr;
    double w = 0.0;
};

// One SIMT launch.  Options, counters and scratch are those of `lead` (the first handle of the
// call's SIMT groups; the launch's own first one if null).
template <typename T>
int run_cells(npfem_handle* const* meshes, int n_groups, const int32_t* cells, T* x, T* v, const T* f, const T* y,
              T* grad_out, double* parts, npfem_cell_stats* stats, int mode, cudaStream_t stream,
              const T* u0 = nullptr, const long long* state_offs = nullptr, const long long* stats_offs = nullptr,
              int threads = 0, const T* hist_in = nullptr, T* hist_out = nullptr, long long pos_stride = 0,
              unsigned int* defer = nullptr, int hist_ext = 0, T* carry = nullptr,
              const long long* carry_offs = nullptr, const long long* carry_recs = nullptr, Planes col = Planes(),
              npfem_handle* lead = nullptr)
{
    npfem_handle* h0 = lead ? lead : meshes[0];
    LaunchArgs<T> a;
    memset(&a, 0, sizeof(a));
    long long total = 0, state = 0, slot = 0, all = 0;
    for (int gi = 0; gi < n_groups; ++gi) all += cells[gi];
    int smem_max = 0;
    // an evaluation (one group) chooses for itself
    if (threads <= 0) threads = eval_threads(simt_mesh(h0), cells[0], h0->sm_count);
    // 512 / threads blocks share an SM's shared memory (1 KB of it per block is the system's)
    const int budget = (threads < 512 ? h0->smem_sm / (512 / threads) : h0->smem_optin) - kFixedSmem - 1024;
    for (int gi = 0; gi < n_groups; ++gi) {
        npfem_handle* h = meshes[gi];
        GroupDesc<T>& g = a.g[gi];
        g.topo = *reinterpret_cast<const TopoDev<T>*>(sizeof(T) == 4 ? (const void*)&h->tf : (const void*)&h->td);
        if (!h->applies_dense(all)) g.topo.ainv = nullptr;
        g.cell_begin = total;
        g.state_off = state_offs ? state_offs[gi] : state;
        g.stats_off = stats_offs ? stats_offs[gi] : total;
        g.cells = cells[gi];
        g.carry_rec = carry_recs ? carry_recs[gi] : 0;
        g.carry_off = carry_offs ? carry_offs[gi] : 0;
        long long sb = 0;
        // (an evaluation solves nothing: no room for the solve's vectors)
        place_vectors(&g, h->n, h->n_pad, h->nt, mode == 1 ? 0 : h->npos(), h0->opts.lbfgs_m, budget, &sb);
        slot = std::max(slot, sb);
        smem_max = std::max(smem_max, g.smem_bytes);
        total += cells[gi];
        state += 3LL * h->n * cells[gi];
    }
    if (total == 0) return 0;
    a.n_groups = n_groups;
    a.total_cells = total;
    a.x = x;
    a.v = v;
    a.f = f;
    a.y = y;
    a.grad_out = grad_out;
    a.parts = parts;
    a.stats = stats;
    a.work = h0->work;
    set_solver_params(&a.p, h0->opts);
    a.p.mode = mode;
    a.u0 = u0;
    a.hist_in = hist_in;
    a.hist_out = hist_out;
    a.pos_stride = sizeof(T) == 4 && hist_out ? pos_stride : 0;
    a.hist_ext = sizeof(T) == 4 && hist_out ? hist_ext : 0;
    a.carry = mode == 0 && hist_out ? carry : nullptr;
    a.defer = defer;
    a.col = reinterpret_cast<const float4*>(col.at);
    a.col_w = (T)col.w;

    const int smem = kFixedSmem + smem_max;
    int per_sm = 1;
    NPFEM_CUDA(cells_per_sm<T>(a, threads, smem, h0->smem_optin, &per_sm));
    per_sm = std::max(per_sm, 1);
    long long grid = std::min<long long>(total, (long long)h0->sm_count * per_sm);
    a.slot_bytes = slot;
    if (slot > 0) {
        NPFEM_CUDA(h0->reserve(&h0->scratch, (size_t)slot * (size_t)grid, stream));
        a.scratch = static_cast<char*>(h0->scratch.p);
    }
    NPFEM_CUDA(launch_cells<T>(a, (int)grid, threads, smem, stream));
    return 0;
}

// Few FP64 cells: one launch of clusters of 8, 4 or 2 blocks per cell, the largest size at which
// every cell's cluster is resident at once.  *done says whether the launch was made (not
// with beta_D > 0, one-rings past the fixed width or meshes too large).
int run_cells_cluster(npfem_handle* const* meshes, int n_groups, const int32_t* cells, double* x, double* v, const double* f,
                      npfem_cell_stats* stats, cudaStream_t stream, const long long* state_offs, const long long* stats_offs,
                      const double* hist_in, double* hist_out, double* carry, const long long* carry_offs,
                      const long long* carry_recs, Planes col, npfem_handle* h0, bool* done)
{
    *done = false;
    long long total = 0;
    for (int gi = 0; gi < n_groups; ++gi) {
        const npfem_handle* h = meshes[gi];
        if (!h->td.k8 || h->mat.beta_D > 0.0 || h->n < 32 || h->n > 4096) return 0;
        total += cells[gi];
    }
    if (total == 0 || 2 * total > h0->sm_count) return 0;
    for (int lg = 3; lg >= 1; --lg) {
        const int C = 1 << lg;
        if (C * total > h0->sm_count) continue;
        LaunchArgs<double> a;
        memset(&a, 0, sizeof(a));
        long long at = 0, slot = 0;
        int smem_max = 0, nt_max = 0;
        bool fits = true;
        for (int gi = 0; gi < n_groups; ++gi) {
            npfem_handle* h = meshes[gi];
            GroupDesc<double>& g = a.g[gi];
            g.topo = h->td;
            g.cell_begin = at;
            g.state_off = state_offs[gi];
            g.stats_off = stats_offs[gi];
            g.cells = cells[gi];
            g.carry_rec = carry_recs[gi];
            g.carry_off = carry_offs[gi];
            long long sb = 0;
            fits = place_vectors_cluster(&g, h->n_pad, h->npos(), h0->opts.lbfgs_m, C,
                                         h0->smem_optin - kFixedSmem - 1024, &sb) && fits;
            slot = std::max(slot, sb);
            smem_max = std::max(smem_max, g.smem_bytes);
            nt_max = std::max(nt_max, h->nt);
            at += cells[gi];
        }
        if (!fits) continue;
        // a thread per two to four triangles of a block's share: every further warp runs the
        // reductions' FP64 shuffles and merges without data
        int block = 128;
        while (block < 512 && 4 * block < nt_max / C) block *= 2;
        const int smem = kFixedSmem + smem_max;
        const int key = smem + (block << 20);
        if (h0->cl_smem[lg] != key) {
            NPFEM_CUDA(query_cells_cl(C, block, smem, h0->smem_optin, &h0->cl_max[lg]));
            h0->cl_smem[lg] = key;
        }
        if (h0->cl_max[lg] < total) continue;
        a.n_groups = n_groups;
        a.total_cells = total;
        a.x = x;
        a.v = v;
        a.f = f;
        a.stats = stats;
        a.work = h0->work;
        set_solver_params(&a.p, h0->opts);
        a.p.cluster = C;
        a.hist_in = hist_in;
        a.hist_out = hist_out;
        a.carry = hist_out ? carry : nullptr;
        a.col = reinterpret_cast<const float4*>(col.at);
        a.col_w = col.w;
        a.slot_bytes = slot;
        if (slot > 0) {
            NPFEM_CUDA(h0->reserve(&h0->scratch, (size_t)slot * (size_t)(C * total), stream));
            a.scratch = static_cast<char*>(h0->scratch.p);
        }
        NPFEM_CUDA(launch_cells_cl(a, C, (int)total, block, smem, stream));
        *done = true;
        return 0;
    }
    return 0;
}

// One tensor-core launch for one mesh group (BF16, n <= kTcMaxVerts).
int run_cells_tc(npfem_handle* h, int cells, float* x, float* v, const float* f, npfem_cell_stats* stats,
                 cudaStream_t stream, const float* u0, const float* hist_in, float* hist_out, long long pos_stride,
                 unsigned int* only, Planes col, int hist_ext, float* carry, long long carry_rec)
{
    if (cells == 0) return 0;
    LaunchArgs<float> a;
    memset(&a, 0, sizeof(a));
    a.hist_ext = hist_out ? hist_ext : 0;
    a.carry = hist_out ? carry : nullptr;
    a.col = reinterpret_cast<const float4*>(col.at);
    a.col_w = (float)col.w;
    a.u0 = u0;
    a.hist_in = hist_in;
    a.hist_out = hist_out;
    a.pos_stride = hist_out ? pos_stride : 0;
    a.only = only;
    a.need = only ? only + 1 : nullptr;
    GroupDesc<float>& g = a.g[0];
    g.topo = h->tf;
    g.cell_begin = 0;
    g.state_off = 0;
    g.cells = cells;
    g.carry_rec = carry_rec;
    g.carry_off = 0;
    const int cluster = h->tf.rb;
    const int ncol = cluster * 3 > 16 ? 32 : 16;
    const int bbytes = (ncol * h->tf.kpad * 2 + 127) & ~127;
    const int budget = h->smem_optin - kFixedSmem - 1024 - bbytes;
    long long slot = 0;
    place_vectors(&g, h->n, h->n_pad, h->nt, h->npos(), h->opts.lbfgs_m, budget, &slot, bbytes, true);
    if (g.loc[V_GC] < 0) return fail(NPFEM_ERR_INVALID_ARG, "mesh too large for the tensor-core path's shared memory");
    a.n_groups = 1;
    a.total_cells = cells;
    a.x = x;
    a.v = v;
    a.f = f;
    a.stats = stats;
    a.work = h->work;
    set_solver_params(&a.p, h->opts);
    a.p.mode = 0;
    a.p.cluster = cluster;
    a.p.refine = h->opts.refine;
    // one block per SM: a second block on the SM would wait in the tensor-memory
    // allocation while its cluster waits for it
    int smem = kFixedSmem + g.smem_bytes;
    smem = std::max(smem, h->smem_optin / 2 + 4096);
    if (h->tc_smem != smem) {
        NPFEM_CUDA(query_cells_tc(cluster, h->mat.beta_D > 0.0, kTcThreads, smem, h->smem_optin,
                                  &h->tc_max_clusters));
        h->tc_smem = smem;
    }
    const int max_clusters = h->tc_max_clusters;
    const long long want = std::min<long long>((cells + cluster - 1) / cluster, max_clusters);
    const int grid = (int)(want * cluster);

    // SMs the clusters leave idle (clusters stay within a GPC) run the SIMT kernel on
    // the same work counter: each cell goes to whichever kind of block asks first
    LaunchArgs<float> b;
    long long slot_b = 0;
    int smem_b = 0;
    int helper = h->sm_count - grid;
    if (cells <= grid || h->opts.fill_idle_sms == 0) helper = 0;
    if (helper > 0) {
        b = a;
        place_vectors(&b.g[0], h->n, h->n_pad, h->nt, h->npos(), h->opts.lbfgs_m, h->smem_optin - kFixedSmem - 1024, &slot_b);
        b.p.cluster = 0;
        b.p.refine = 0;
        // more than half of an SM's shared memory, so that no block shares an SM with a cluster's
        smem_b = std::max(kFixedSmem + b.g[0].smem_bytes, h->smem_optin / 2 + 4096);
    }
    a.total_blocks = grid + helper;
    a.slot_bytes = slot;
    const size_t need = (size_t)slot * (size_t)grid + (size_t)slot_b * (size_t)helper;
    if (need > 0) {
        NPFEM_CUDA(h->reserve(&h->scratch, need, stream));
        a.scratch = slot > 0 ? static_cast<char*>(h->scratch.p) : nullptr;
    }
    if (helper > 0) {
        b.total_blocks = a.total_blocks;
        b.claim_top = 1;
        b.reserve = grid;  // about one cell per cluster block: the helper's cells take longer
        b.slot_bytes = slot_b;
        b.scratch = slot_b > 0 ? static_cast<char*>(h->scratch.p) + (size_t)slot * (size_t)grid : nullptr;
        if (!h->side_stream) {
            NPFEM_CUDA(cudaStreamCreateWithFlags(&h->side_stream, cudaStreamNonBlocking));
            NPFEM_CUDA(cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
            NPFEM_CUDA(cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming));
        }
        NPFEM_CUDA(cudaEventRecord(h->ev_fork, stream));
    }
    NPFEM_CUDA(launch_cells_tc(a, cluster, kTcThreads, smem, grid, stream));
    if (helper > 0) {
        cudaError_t e = cudaStreamWaitEvent(h->side_stream, h->ev_fork, 0);
        if (e == cudaSuccess) e = allow_cells_smem<float>(b, kTcThreads, h->smem_optin);
        if (e == cudaSuccess) e = launch_cells<float>(b, helper, kTcThreads, smem_b, h->side_stream);
        if (e != cudaSuccess) {
            // the clusters alone cannot reset the shared counters: clear them behind
            // the launch so that the next step starts clean, and report the failure
            cudaMemsetAsync(h->work, 0, 2 * sizeof(unsigned), stream);
            cudaMemsetAsync(h->work + 3, 0, sizeof(unsigned), stream);
            return fail(NPFEM_ERR_CUDA, std::string("idle-SM launch: ") + cudaGetErrorString(e));
        }
        NPFEM_CUDA(cudaEventRecord(h->ev_join, h->side_stream));
        NPFEM_CUDA(cudaStreamWaitEvent(stream, h->ev_join, 0));
    }
    return 0;
}

// The solver launches of one step: one cluster launch per group that takes the
// tensor-core kernel (BF16, mesh of at most kTcMaxVerts vertices, not tuned away), and
// one persistent SIMT launch per block size over the other groups.
int step_groups(npfem_handle* const* meshes, int n_groups, const int32_t* cells_per_group, void* x, void* v,
                const void* f_ext, cudaStream_t s, npfem_cell_stats* stats, const float* u0, const void* hist_in,
                void* hist_out, long long pos_stride, int hist_ext, void* carry, const CarryPlan& kept)
{
    const int prec = meshes[0]->precision;
    const npfem_handle* first = meshes[0];  // its collision planes hold for the whole call
    std::vector<long long> soff(n_groups), coff(n_groups);
    const std::vector<long long>&koff = kept.off, &krec = kept.rec;
    long long st = 0, ct = 0;
    for (int g = 0; g < n_groups; ++g) {
        soff[g] = st;
        coff[g] = ct;
        st += 3LL * meshes[g]->n * cells_per_group[g];
        ct += cells_per_group[g];
    }
    std::vector<char> done(n_groups, 0);
    for (int g = 0; g < n_groups; ++g) {
        if (cells_per_group[g] == 0) {
            done[g] = 1;
            continue;
        }
        if (prec == NPFEM_PREC_BF16 && meshes[g]->takes_clusters()) {
            npfem_handle* hg = meshes[g];
            int32_t cg = cells_per_group[g];
            float* xg = (float*)x + soff[g];
            float* vg = (float*)v + soff[g];
            const float* fg = (const float*)f_ext + soff[g];
            npfem_cell_stats* sg = stats ? stats + coff[g] : nullptr;
            const float* hin = hist_in ? (const float*)hist_in + soff[g] : nullptr;
            float* hout = hist_out ? (float*)hist_out + soff[g] : nullptr;
            float* kg = carry ? (float*)carry + koff[g] : nullptr;
            Planes colg;
            if (first->col_planes) colg = {first->col_planes + 4 * (soff[g] / 3), first->col_w};
            unsigned int* only = nullptr;
            const size_t listed = sizeof(unsigned int) * ((size_t)cg + 3);
            if (hout) {
                // allocated with the history (first call of a trajectory), so that the
                // steps that use it allocate nothing (they may be captured in a graph)
                const bool fresh = listed > hg->defer.bytes;
                NPFEM_CUDA(hg->reserve(&hg->defer, listed, s));
                if (fresh) NPFEM_CUDA(cudaMemsetAsync(hg->defer.p, 0, 3 * sizeof(unsigned int), s));
            }
            if (hin && listed <= hg->defer.bytes) {
                unsigned int* defer = static_cast<unsigned int*>(hg->defer.p);
                // along a trajectory many cells are accepted at the first iterate: a SIMT
                // launch on every SM (the clusters' idle SMs included) evaluates each cell
                // there and finishes those, and the cluster kernel takes only the rest
                // (one block of 512 threads per SM: its vectors fit in shared memory, so a
                // trajectory's first pass does not grow the handle's scratch)
                NPFEM_CUDA(cudaMemcpyAsync(defer + 2, defer + 1, sizeof(unsigned int), cudaMemcpyDeviceToDevice, s));
                NPFEM_CUDA(cudaMemsetAsync(defer, 0, 2 * sizeof(unsigned int), s));
                int rc = run_cells<float>(&hg, 1, &cg, xg, vg, fg, nullptr, nullptr, nullptr, sg, 0, s,
                                          u0 ? u0 + soff[g] : nullptr, nullptr, nullptr, 512, hin, hout, pos_stride,
                                          defer, hist_ext, kg, nullptr, &krec[g], colg);
                if (rc) return rc;
                only = defer;
            }
            int rc = run_cells_tc(hg, cg, xg, vg, fg, sg, s, u0 ? u0 + soff[g] : nullptr, hin, hout, pos_stride, only,
                                  colg, hist_ext, kg, krec[g]);
            if (rc) return rc;
            done[g] = 1;
        }
    }
    // the other groups: with at most a cell per SM in all one launch, else each at its own
    // block size, groups of one size together.  A group with at most a cell per SM beside a
    // larger population of meshes at least as fine joins that launch (alone it would take
    // the time of a cell on an empty GPU).
    const long long sms = meshes[0]->sm_count;
    long long left = 0;
    npfem_handle* lead = nullptr;
    for (int g = n_groups - 1; g >= 0; --g)
        if (!done[g]) {
            left += cells_per_group[g];
            lead = meshes[g];  // in the end that of simt_lead()
        }
    std::vector<int> shape(n_groups, 512);
    std::vector<char> dense(n_groups, 0), joined(n_groups, 0);
    if (left > sms) {
        for (int g = 0; g < n_groups; ++g) {
            int as = g;
            for (int m = 0; m < n_groups && cells_per_group[g] <= sms; ++m)
                if (!done[m] && cells_per_group[m] > sms && meshes[m]->n >= meshes[g]->n) as = m;
            shape[g] = simt_threads(simt_mesh(meshes[as]), cells_per_group[as], sms);
            dense[g] = meshes[as]->applies_dense(left);
            if (as != g) joined[g] = 1;
        }
        // Launches follow one another, so a group that leaves SMs idle costs its own latency
        // (about n) where one launch of 512-thread blocks would fill those SMs with the other
        // cells; that launch takes longest-cell or total work, the separate ones gain 1.9 from
        // four blocks per SM and 1.2 from two.  642 x 100 + 258 x 200, two steps: 467 us in one
        // launch, 589 in two.
        if (prec != NPFEM_PREC_FP64) {
            double apart = 0, sum = 0, longest = 0;
            for (int g = 0; g < n_groups; ++g) {
                if (done[g]) continue;
                const double n = meshes[g]->n, w = n * cells_per_group[g] / sms;
                sum += w;
                longest = std::max(longest, n);
                // two sparse solves on an SM take 1.8 of one (1026 x 200 + 642 x 200: 2828 us apart,
                // 2565 in one launch; 642 x 300 + 1026 x 300: 2893 and 3518)
                const bool two = shape[g] == 256 && !dense[g];
                const double per_sm = shape[g] == 128 ? 1.9 : (two ? 1.1 : (shape[g] == 256 ? 1.2 : 1.0));
                apart += joined[g] ? w / per_sm : std::max(two ? 1.8 * n : n, w / per_sm);
            }
            if (n_groups > 1 && std::max(longest, sum) < apart) {
                std::fill(shape.begin(), shape.end(), 512);
                std::fill(dense.begin(), dense.end(), 0);
            }
        }
    } else if (n_groups == 1) {
        shape[0] = simt_threads(simt_mesh(meshes[0]), left, sms);
    }
    for (int g0 = 0; g0 < n_groups; ++g0) {
        if (done[g0]) continue;
        const int threads = shape[g0];
        std::vector<npfem_handle*> hs;
        std::vector<int32_t> cs;
        std::vector<long long> so, co, ko, kr;
        for (int g = g0; g < n_groups; ++g) {
            if (done[g] || shape[g] != threads || dense[g] != dense[g0]) continue;
            hs.push_back(meshes[g]);
            cs.push_back(cells_per_group[g]);
            so.push_back(soff[g]);
            co.push_back(coff[g]);
            ko.push_back(koff[g]);
            kr.push_back(krec[g]);
            done[g] = 1;
        }
        int rc;
        Planes col;
        if (first->col_planes) col = {first->col_planes, first->col_w};
        bool clustered = false;
        if (prec == NPFEM_PREC_FP64) {
            rc = run_cells_cluster(hs.data(), (int)hs.size(), cs.data(), (double*)x, (double*)v, (const double*)f_ext,
                                   stats, s, so.data(), co.data(), (const double*)hist_in, (double*)hist_out,
                                   (double*)carry, ko.data(), kr.data(), col, lead, &clustered);
            if (rc) return rc;
        }
        if (clustered) continue;
        for (npfem_handle* h : hs) h->simt_block = threads;
        if (prec == NPFEM_PREC_FP64)
            rc = run_cells<double>(hs.data(), (int)hs.size(), cs.data(), (double*)x, (double*)v, (const double*)f_ext,
                                   nullptr, nullptr, nullptr, stats, 0, s, nullptr, so.data(), co.data(), threads,
                                   (const double*)hist_in, (double*)hist_out, 0, nullptr, 0, (double*)carry,
                                   ko.data(), kr.data(), col, lead);
        else
            rc = run_cells<float>(hs.data(), (int)hs.size(), cs.data(), (float*)x, (float*)v, (const float*)f_ext,
                                  nullptr, nullptr, nullptr, stats, 0, s, u0, so.data(), co.data(), threads,
                                  (const float*)hist_in, (float*)hist_out, pos_stride, nullptr, hist_ext,
                                  (float*)carry, ko.data(), kr.data(), col, lead);
        if (rc) return rc;
    }
    return 0;
}

// Learned first increments of every group with a warm start, into meshes[0]'s
// buffer at the groups' state offsets (a separate launch: in the cluster kernel a
// block computing them would hold up its whole cluster).  Null when no group has one.
int precompute_warm_start(npfem_handle* const* meshes, int n_groups, const int32_t* cells, const float* x,
                          const float* v, const float* f, cudaStream_t s, const float** u0)
{
    *u0 = nullptr;
    bool any = false;
    size_t total = 0;
    for (int g = 0; g < n_groups; ++g) {
        any = any || (meshes[g]->tf.ws_mode && meshes[g]->tf.mlp && cells[g] > 0);
        total += (size_t)3 * meshes[g]->n * cells[g];
    }
    if (!any) return 0;
    npfem_handle* h0 = meshes[0];
    NPFEM_CUDA(h0->reserve(&h0->ws_u, total * sizeof(float), s));
    float* u = static_cast<float*>(h0->ws_u.p);
    size_t off = 0;
    for (int g = 0; g < n_groups; ++g) {
        if (meshes[g]->tf.ws_mode && meshes[g]->tf.mlp && cells[g] > 0)
            NPFEM_CUDA(launch_ws_increments(meshes[g], cells[g], x + off, v + off, f + off, u + off, false, s));
        off += (size_t)3 * meshes[g]->n * cells[g];
    }
    *u0 = u;
    return 0;
}

// First increments of every group along a trajectory with a temporal network, into
// meshes[0]'s buffer at the groups' state offsets (one launch per group).
int precompute_temporal(npfem_handle* const* meshes, int n_groups, const int32_t* cells, const float* x,
                        const float* v, const float* f, const float* hist, long long pos_stride, cudaStream_t s,
                        const float** u0)
{
    npfem_handle* h0 = meshes[0];
    size_t total = 0;
    for (int g = 0; g < n_groups; ++g) total += (size_t)3 * meshes[g]->n * cells[g];
    NPFEM_CUDA(h0->reserve(&h0->ws_u, total * sizeof(float), s));
    float* u = static_cast<float*>(h0->ws_u.p);
    size_t off = 0;
    const float* c1 = hist;                  // c_{n-1}
    const float* c2 = hist + 3 * pos_stride;  // c_{n-2}
    const float* fp = hist + 4 * pos_stride;  // F_{n-1}
    for (int g = 0; g < n_groups; ++g) {
        if (cells[g] > 0)
            NPFEM_CUDA(launch_ws_temporal(meshes[g], cells[g], x + off, v + off, f + off, fp + off, c1 + off, c2 + off,
                                          nullptr, nullptr, nullptr, nullptr, u + off, 3LL * meshes[g]->n, s));
        off += (size_t)3 * meshes[g]->n * cells[g];
    }
    *u0 = u;
    return 0;
}

int validate_group(npfem_handle* const* meshes, int n_groups, const int32_t* cells)
{
    if (!meshes || n_groups < 1 || n_groups > kMaxGroups || !cells)
        return fail(NPFEM_ERR_INVALID_ARG, "need 1..8 mesh handles and a cells_per_group array");
    for (int g = 0; g < n_groups; ++g) {
        if (!meshes[g]) return fail(NPFEM_ERR_INVALID_ARG, "null mesh handle");
        if (cells[g] < 0) return fail(NPFEM_ERR_INVALID_ARG, "negative cell count");
        if (meshes[g]->device != meshes[0]->device || meshes[g]->precision != meshes[0]->precision ||
            meshes[g]->dt != meshes[0]->dt)
            return fail(NPFEM_ERR_INVALID_ARG, "all handles of one call must share device, precision and dt");
    }
    return 0;
}

}  // namespace

extern "C" {

void npfem_default_opts(npfem_opts* o)
{
    if (!o) return;
    o->precision = NPFEM_PREC_FP32;
    o->lbfgs_m = 5;
    o->max_iter = 50;
    o->tol = 1e-6;
    o->c1 = 1e-4;
    o->c2 = 0.9;
    o->max_halvings = 30;
    o->fixed_alpha = 0;
    o->equal_mass = 0;
    o->armijo_noise = 4.0;
    o->refine = 0;
    o->fill_idle_sms = 1;
    o->warm_history = 2;
}

const char* npfem_last_error(void) { return g_last_error.c_str(); }

unsigned long long npfem_launch_count(void) { return npfem::g_launches.load(); }

int npfem_kernel_timing(npfem_handle* h, int capacity)
{
    if (!h || capacity < 0) return fail(NPFEM_ERR_INVALID_ARG, "npfem_kernel_timing: bad argument");
    DeviceGuard guard(h->device);
    std::lock_guard<std::mutex> lk(h->mu);
    NPFEM_CUDA(cudaDeviceSynchronize());
    for (cudaEvent_t e : h->tev) cudaEventDestroy(e);
    h->tev.clear();
    h->tev_used = 0;
    for (int q = 0; q < 2 * capacity; ++q) {
        cudaEvent_t e;
        NPFEM_CUDA(cudaEventCreate(&e));
        h->tev.push_back(e);
    }
    return 0;
}

int npfem_get_tuning(const npfem_handle* h, int* use_tc, int* threads, int* fill_idle_sms)
{
    if (!h || !use_tc || !threads || !fill_idle_sms) return fail(NPFEM_ERR_INVALID_ARG, "npfem_get_tuning: null argument");
    *use_tc = h->takes_clusters();
    *threads = h->simt_block;
    *fill_idle_sms = h->opts.fill_idle_sms;
    return 0;
}

int npfem_autotune(npfem_handle* const* meshes, int n_groups, const int32_t* cells_per_group, const void* x,
                   const void* v, const void* f_ext, double dt, int trial_steps, float* trial_ms)
{
    if (int rc = validate_group(meshes, n_groups, cells_per_group)) return rc;
    if (!x || !v || !f_ext || trial_steps < 1) return fail(NPFEM_ERR_INVALID_ARG, "npfem_autotune: bad argument");
    DeviceGuard guard(meshes[0]->device);
    NPFEM_CUDA(cudaDeviceSynchronize());
    const int prec = meshes[0]->precision;
    const size_t es = prec == NPFEM_PREC_FP64 ? 8 : 4;
    struct Shape {
        int use_tc, fill, slot;
    };
    if (trial_ms)
        for (int q = 0; q < 5 * n_groups; ++q) trial_ms[q] = -1.f;
    cudaStream_t s = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    NPFEM_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    NPFEM_CUDA(cudaEventCreate(&e0));
    NPFEM_CUDA(cudaEventCreate(&e1));
    int rc = 0;
    size_t off = 0;
    for (int g = 0; g < n_groups && !rc; ++g) {
        npfem_handle* h = meshes[g];
        const int cells = cells_per_group[g];
        const size_t bytes = (size_t)3 * h->n * cells * es;
        if (cells == 0) continue;
        std::vector<Shape> cand;
        cand.push_back({0, h->opts.fill_idle_sms, 0});
        if (h->fits_clusters()) {
            cand.push_back({1, 1, 2});
            cand.push_back({1, 0, 3});
        }
        void *tx = nullptr, *tv = nullptr;
        cudaError_t ce = cudaMalloc(&tx, bytes);
        if (ce == cudaSuccess) ce = cudaMalloc(&tv, bytes);
        if (ce != cudaSuccess) {
            rc = fail(ce == cudaErrorMemoryAllocation ? NPFEM_ERR_OOM : NPFEM_ERR_CUDA, "npfem_autotune: trial buffers");
        }
        float best = 1e30f;
        Shape pick = {h->use_tc, h->opts.fill_idle_sms, -1};
        const int hist_opt = h->opts.warm_history;
        for (const Shape& c : cand) {
            if (rc) break;
            h->use_tc = c.use_tc;
            h->opts.fill_idle_sms = c.fill;
            const char* xs = static_cast<const char*>(x) + off;
            const char* vs = static_cast<const char*>(v) + off;
            const void* fs = static_cast<const char*>(f_ext) + off;
            // one untimed step, then trial_steps back to back (as in a time loop)
            float total = 0.f;
            npfem_handle* one[1] = {h};
            h->hist_sig.clear();  // each candidate's untimed step starts without history
            NPFEM_CUDA(cudaMemcpyAsync(tx, xs, bytes, cudaMemcpyDeviceToDevice, s));
            NPFEM_CUDA(cudaMemcpyAsync(tv, vs, bytes, cudaMemcpyDeviceToDevice, s));
            rc = npfem_step(one, 1, &cells, tx, tv, fs, dt, s, nullptr);
            if (!rc) NPFEM_CUDA(cudaEventRecord(e0, s));
            for (int k = 0; k < trial_steps && !rc; ++k) rc = npfem_step(one, 1, &cells, tx, tv, fs, dt, s, nullptr);
            if (!rc) {
                NPFEM_CUDA(cudaEventRecord(e1, s));
                NPFEM_CUDA(cudaEventSynchronize(e1));
                NPFEM_CUDA(cudaEventElapsedTime(&total, e0, e1));
            }
            if (!rc && trial_ms) trial_ms[5 * g + c.slot] = total / trial_steps;
            if (!rc && total < best) {
                best = total;
                pick = c;
            }
        }
        h->use_tc = pick.use_tc;
        h->opts.fill_idle_sms = pick.fill;
        h->opts.warm_history = hist_opt;
        h->hist_sig.clear();
        if (tx) cudaFree(tx);
        if (tv) cudaFree(tv);
        off += bytes;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamDestroy(s);
    return rc;
}

int npfem_kernel_time_last(npfem_handle* h, float* ms)
{
    if (!h || !ms) return fail(NPFEM_ERR_INVALID_ARG, "npfem_kernel_time_last: bad argument");
    DeviceGuard guard(h->device);
    std::lock_guard<std::mutex> lk(h->mu);
    if (h->tev_used < 2) return fail(NPFEM_ERR_INVALID_ARG, "npfem_kernel_time_last: nothing recorded");
    NPFEM_CUDA(cudaEventSynchronize(h->tev[1]));
    NPFEM_CUDA(cudaEventElapsedTime(ms, h->tev[0], h->tev[1]));
    return 0;
}

int npfem_kernel_times(npfem_handle* h, float* ms_out, int max, int* count)
{
    if (!h || !count || max < 0 || (max > 0 && !ms_out)) return fail(NPFEM_ERR_INVALID_ARG, "npfem_kernel_times: bad argument");
    DeviceGuard guard(h->device);
    std::lock_guard<std::mutex> lk(h->mu);
    int k = 0;
    for (int q = 0; q + 1 < h->tev_used && k < max; q += 2, ++k) {
        NPFEM_CUDA(cudaEventSynchronize(h->tev[q + 1]));
        NPFEM_CUDA(cudaEventElapsedTime(&ms_out[k], h->tev[q], h->tev[q + 1]));
    }
    *count = k;
    h->tev_used = 0;
    return 0;
}

int npfem_create(const npfem_mesh* mesh, const npfem_material* mat, const npfem_opts* opts, double dt, int device,
                 npfem_handle** out)
{
    g_last_error.clear();
    if (!mesh || !mat || !opts || !out || !mesh->tris || !mesh->rest_xyz)
        return fail(NPFEM_ERR_INVALID_ARG, "null argument");
    *out = nullptr;
    if (!(dt > 0.0) || !isfinite(dt)) return fail(NPFEM_ERR_INVALID_ARG, "dt must be positive");
    if (int rc = check_opts(opts)) return rc;
    if (!(mat->density > 0.0) || mat->kappa < 0.0 || mat->kappa > 1.0 || mat->C < 0 || mat->B < 0 || mat->D < 0 ||
        mat->k_bend < 0 || mat->k_vol < 0 || mat->k_mat_hess < 0 || mat->alpha_D < 0 || !(mat->beta_D >= 0.0))
        return fail(NPFEM_ERR_INVALID_ARG, "material: need density > 0, kappa in [0,1], non-negative moduli");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev)
        return fail(NPFEM_ERR_INVALID_ARG, "no such CUDA device");
    DeviceGuard guard(device);

    npfem_handle* h = new npfem_handle();
    h->device = device;
    h->precision = opts->precision;
    h->dt = dt;
    h->opts = *opts;
    h->mat = *mat;
    std::string err;
    int rc = build_host_topo(mesh, mat, opts->equal_mass, &h->host, &err);
    if (rc) {
        delete h;
        return fail(rc, err);
    }
    h->n = h->host.n;
    h->nt = h->host.nt;
    h->n_pad = (h->n + 3) & ~3;
    for (int c = 0; c < 3; ++c) {
        const auto mm = std::minmax_element(h->host.rest_c.begin() + (size_t)c * h->n, h->host.rest_c.begin() + (size_t)(c + 1) * h->n);
        h->rest_extent += (*mm.second - *mm.first) * (*mm.second - *mm.first) / 3.0;
    }
    h->rest_extent = sqrt(h->rest_extent);
    cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, device);
    cudaDeviceGetAttribute(&h->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    cudaDeviceGetAttribute(&h->smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);

    auto bail = [&](int code) {
        h->release();
        delete h;
        return code;
    };
    const int n = h->n, np = h->n_pad;
    int e = 0;
    // dense H~ = M~/h^2 + L in FP64, inverted on the GPU.  Rayleigh damping
    // C = alpha_D M + beta_D L (Sec. 2.1.4) gives M~ = (1 + h alpha_D) M + h beta_D L, so
    // H~ = (1 + h alpha_D)/h^2 M + (1 + beta_D/h) L
    std::vector<double> H((size_t)n * n, 0.0);
    const double ms = (1.0 + dt * mat->alpha_D) / (dt * dt);
    const double lscale = 1.0 + mat->beta_D / dt;
    for (int i = 0; i < n; ++i) {
        H[(size_t)i * n + i] += ms * h->host.mass[i];
        for (int q = h->host.L_ptr[i]; q < h->host.L_ptr[i + 1]; ++q)
            H[(size_t)i * n + h->host.L_idx[q]] += lscale * h->host.L_val[q];
    }
    h->ainv64 = h->alloc<double>((size_t)n * n, &e);
    double* prow = h->alloc<double>(2 * (size_t)n, &e);
    int* flag = h->alloc<int>(4, &e);
    h->work = h->alloc<unsigned int>(4, &e);
    if (e) return bail(e);
    if (cudaMemset(h->work, 0, 4 * sizeof(unsigned)) != cudaSuccess) return bail(fail(NPFEM_ERR_CUDA, "memset failed"));
    // one inversion on the GPU, in place; done() waits for it
    auto invert = [&](double* dA, const std::vector<double>& A, const char* what) -> int {
        if (cudaMemcpy(dA, A.data(), A.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemset(flag, 0, 4 * sizeof(int)) != cudaSuccess)
            return fail(NPFEM_ERR_CUDA, std::string("upload of ") + what + " failed");
        const cudaError_t ce = invert_spd_fp64(dA, n, prow, flag, 0);
        if (ce != cudaSuccess) return fail(NPFEM_ERR_CUDA, std::string("inversion of ") + what + ": " + cudaGetErrorString(ce));
        return 0;
    };
    auto done = [&](const char* what) -> int {
        int hflag = 0;
        if (cudaMemcpy(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
            return fail(NPFEM_ERR_CUDA, std::string("inversion of ") + what + " failed");
        if (hflag == 2) return fail(NPFEM_ERR_TIMEOUT, std::string("inversion of ") + what + ": a grid barrier gave up");
        if (hflag) return fail(NPFEM_ERR_NOT_SPD, std::string(what) + " is not positive definite");
        return 0;
    };
    // the dense inverse (also for npfem_get_inverse), while the host forms the sparse factors
    // of a mesh whose cells apply those; beta_D > 0: M~ is not diagonal, the first guess
    // applies M~^-1 the same way (Eq. preOptimizationNewton)
    const bool damped = mat->beta_D > 0.0, dense = h->precision != NPFEM_PREC_FP64 && n <= kDenseVerts;
    const bool few = h->applies_dense(1);  // dense at least in launches of few cells
    if ((rc = invert(h->ainv64, H, "H~"))) return bail(rc);
    Factors factors;
    int frc = 0;
    if (!dense) {
        frc = build_sparse_factor(h->host, mesh->rest_xyz, ms, lscale, &factors.system,
                                  opts->precision == NPFEM_PREC_FP64 ? &factors.cluster : nullptr, &err);
        if (!frc && damped && !h->fits_clusters())
            frc = build_sparse_factor(h->host, mesh->rest_xyz, 1.0 + dt * mat->alpha_D, dt * mat->beta_D, &factors.mass,
                                      nullptr, &err);
        if (frc == NPFEM_ERR_NOT_SPD && factors.mass.npos) err = "M~ is not positive definite";
    }
    if ((rc = done("H~"))) return bail(rc);
    if (frc) return bail(fail(frc, err));
    float *a32 = nullptr, *m32 = nullptr;
    if (few) {
        a32 = h->alloc<float>((size_t)np * np, &e);
        if (e) return bail(e);
    }
    if (symmetrise(h->ainv64, n, np, a32, 0) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)
        return bail(fail(NPFEM_ERR_CUDA, "symmetrising A^-1 failed"));
    const bool dense_mass = damped && (dense || h->fits_clusters());
    if (dense_mass) {
        std::vector<double> Mt((size_t)n * n, 0.0);
        for (int i = 0; i < n; ++i) {
            Mt[(size_t)i * n + i] += (1.0 + dt * mat->alpha_D) * h->host.mass[i];
            for (int q = h->host.L_ptr[i]; q < h->host.L_ptr[i + 1]; ++q)
                Mt[(size_t)i * n + h->host.L_idx[q]] += dt * mat->beta_D * h->host.L_val[q];
        }
        m32 = h->alloc<float>((size_t)np * np, &e);
        double* m64 = h->alloc<double>((size_t)n * n, &e);
        if (e) return bail(e);
        if ((rc = invert(m64, Mt, "M~")) || (rc = done("M~"))) return bail(rc);
        if (symmetrise(m64, n, np, m32, 0) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)
            return bail(fail(NPFEM_ERR_CUDA, "symmetrising M~^-1 failed"));
    }
    rc = h->precision == NPFEM_PREC_FP64 ? fill_topo<double>(h, &h->td, factors) : fill_topo<float>(h, &h->tf, factors);
    if (rc) return bail(rc);
    h->tf.ainv = a32;
    h->tf.minv = m32;
    h->tf.dense_p = dense_parts(n);
    if (h->precision == NPFEM_PREC_BF16 && n <= kTcMaxVerts) {
        // tensor-core path: BF16 A^-1 in 128-row blocks with K padded to 16, and L for
        // the refinement residual
        const int kpad = (n + 15) & ~15, rb = (n + 127) / 128;
        void* abf = h->alloc<unsigned short>((size_t)rb * 128 * kpad, &e);
        if (e) return bail(e);
        if (publish_inverse_bf16_blocked(h->ainv64, n, rb * 128, kpad, abf, 0) != cudaSuccess ||
            cudaDeviceSynchronize() != cudaSuccess)
            return bail(fail(NPFEM_ERR_CUDA, "publishing the BF16 A^-1 failed"));
        h->tf.ainv_lp = abf;
        h->tf.kpad = kpad;
        h->tf.rb = rb;
        // the refinement residual q - H~ r needs H~ = ms M + (1 + beta_D/h) L
        std::vector<float> lval(h->host.L_val.size());
        for (size_t q = 0; q < lval.size(); ++q) lval[q] = (float)(lscale * h->host.L_val[q]);
        std::vector<unsigned short> lidx(h->host.L_idx.begin(), h->host.L_idx.end());
        if ((rc = upload(h, h->host.L_ptr, &h->tf.h_ptr))) return bail(rc);
        if ((rc = upload(h, lidx, &h->tf.h_idx))) return bail(rc);
        if ((rc = upload(h, lval, &h->tf.h_val))) return bail(rc);
    }
    *out = h;
    return 0;
}

int npfem_destroy(npfem_handle* h)
{
    if (!h) return fail(NPFEM_ERR_INVALID_ARG, "null handle");
    {
        DeviceGuard guard(h->device);
        cudaDeviceSynchronize();
        h->release();
    }
    delete h;
    return 0;
}

int npfem_step(npfem_handle* const* meshes, int n_groups, const int32_t* cells_per_group, void* x, void* v,
               const void* f_ext, double dt, void* stream, npfem_cell_stats* stats)
{
    if (int rc = validate_group(meshes, n_groups, cells_per_group)) return rc;
    if (!x || !v || !f_ext) return fail(NPFEM_ERR_INVALID_ARG, "null state pointer");
    if (dt != meshes[0]->dt) return fail(NPFEM_ERR_INVALID_ARG, "dt differs from the handle's dt");
    // the limit of the TF32 precision, whatever its cells run on
    for (int g = 0; g < n_groups; ++g)
        if (meshes[g]->precision == NPFEM_PREC_TF32 && cells_per_group[g] > 0 && meshes[g]->n > kTf32MaxVerts)
            return fail(NPFEM_ERR_INVALID_ARG, "npfem_step: TF32 handles of at most 4096 vertices");
    DeviceGuard guard(meshes[0]->device);
    std::lock_guard<std::mutex> lk(meshes[0]->mu);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    npfem_handle* h0 = meshes[0];
    // temporal warm start: read the last step's corrections when this call steps the
    // same groups and cell counts, and write this step's
    const void* hist_in = nullptr;
    void* hist_out = nullptr;
    long long pos_stride = 0;
    int hist_ext = 0;
    void* carry = nullptr;
    std::vector<PlanGroup> groups;
    for (int g = 0; g < n_groups; ++g)
        groups.push_back({meshes[g]->n, meshes[g]->n_pad, meshes[g]->opts.lbfgs_m, cells_per_group[g],
                          meshes[g]->takes_clusters()});
    const CarryPlan kept = plan_carry(groups);
    if (h0->opts.warm_history) {
        std::vector<long long> sig;
        size_t elems = 0;
        for (int g = 0; g < n_groups; ++g) {
            sig.push_back(reinterpret_cast<long long>(meshes[g]));
            sig.push_back(cells_per_group[g]);
            sig.push_back(kept.window[g]);
            elems += (size_t)3 * meshes[g]->n * cells_per_group[g];
            if (meshes[g]->precision != NPFEM_PREC_FP64 && meshes[g]->tf.tmlp) hist_ext = 1;
        }
        sig.push_back(hist_ext);
        // FP64: the corrections; FP32: the corrections, then the positions' rounding
        // residues, then the FP32 positions they belong to (compensated positions); with a
        // temporal network also the previous correction and the last force
        const bool f32 = h0->precision != NPFEM_PREC_FP64;
        pos_stride = f32 ? (long long)elems : 0;
        const size_t bytes = elems * (f32 ? (hist_ext ? 5 : 3) * 4 : 8);
        if (bytes > h0->hist.bytes) h0->hist_sig.clear();
        NPFEM_CUDA(h0->reserve(&h0->hist, bytes, s));
        if (h0->opts.warm_history == 2 && bytes > 0) {
            // carried L-BFGS pairs: one record per cell, valid together with the corrections
            const size_t kb = (size_t)kept.total * (f32 ? 4 : 8);
            if (kb > h0->carry.bytes) h0->hist_sig.clear();
            NPFEM_CUDA(h0->reserve(&h0->carry, kb, s));
            carry = h0->carry.p;
        }
        if (bytes > 0) {
            if (sig == h0->hist_sig) hist_in = h0->hist.p;
            hist_out = h0->hist.p;
            h0->hist_sig = sig;
        }
    }
    const float* u0 = nullptr;
    if (meshes[0]->precision != NPFEM_PREC_FP64 && !hist_in) {
        if (int rc = precompute_warm_start(meshes, n_groups, cells_per_group, (const float*)x, (const float*)v,
                                           (const float*)f_ext, s, &u0))
            return rc;
    } else if (hist_in && hist_ext) {
        // along a trajectory with a temporal network: u = u_y + c_{n-1} + R MLP(features)
        // for every group (u_y + c_{n-1} where a group has no network)
        if (int rc = precompute_temporal(meshes, n_groups, cells_per_group, (const float*)x, (const float*)v,
                                         (const float*)f_ext, (const float*)hist_in, pos_stride, s, &u0))
            return rc;
    }
    const bool timed = h0->tev_used + 2 <= (int)h0->tev.size();
    unsigned rec_flags = cudaEventRecordDefault;
    if (timed) {
        // inside a stream capture the pair must become event-record nodes of the graph
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        NPFEM_CUDA(cudaStreamIsCapturing(s, &cap));
        if (cap == cudaStreamCaptureStatusActive) rec_flags = cudaEventRecordExternal;
        NPFEM_CUDA(cudaEventRecordWithFlags(h0->tev[h0->tev_used], s, rec_flags));
    }
    int rc = step_groups(meshes, n_groups, cells_per_group, x, v, f_ext, s, stats, u0, hist_in, hist_out, pos_stride,
                         hist_ext, carry, kept);
    if (rc) h0->hist_sig.clear();
    if (!rc && timed) {
        NPFEM_CUDA(cudaEventRecordWithFlags(h0->tev[h0->tev_used + 1], s, rec_flags));
        h0->tev_used += 2;
    }
    return rc;
}

// The device address of a pinned host buffer mapped into the current device's address
// space (cudaHostAlloc, or cudaHostRegister with mapping), or null for any other pointer.
static void* mapped_host(void* p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();  // not a pointer the runtime knows: clear the error, copy instead
        return nullptr;
    }
    return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
}

int npfem_step_host(npfem_handle* h, int n_cells, void* x_host, void* v_host, const void* f_host, double dt,
                    void* stream, npfem_cell_stats* stats_host)
{
    if (!h || n_cells < 0 || !x_host || !v_host || !f_host) return fail(NPFEM_ERR_INVALID_ARG, "null argument");
    if (dt != h->dt) return fail(NPFEM_ERR_INVALID_ARG, "dt differs from the handle's dt");
    DeviceGuard guard(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t es = h->precision == NPFEM_PREC_FP64 ? 8 : 4;
    const size_t bytes = (size_t)n_cells * 3 * h->n * es;
    {
        std::lock_guard<std::mutex> lk(h->mu);
        if ((size_t)n_cells > h->host_cells) {
            NPFEM_CUDA(cudaStreamSynchronize(s));
            if (h->hx) cudaFree(h->hx);
            if (h->hv) cudaFree(h->hv);
            if (h->hf) cudaFree(h->hf);
            if (h->hstats) cudaFree(h->hstats);
            h->hx = h->hv = h->hf = nullptr;
            h->hstats = nullptr;
            h->host_cells = 0;
            NPFEM_CUDA(cudaMalloc(&h->hx, bytes));
            NPFEM_CUDA(cudaMalloc(&h->hv, bytes));
            NPFEM_CUDA(cudaMalloc(&h->hf, bytes));
            NPFEM_CUDA(cudaMalloc(&h->hstats, sizeof(npfem_cell_stats) * (size_t)std::max(n_cells, 1)));
            h->host_cells = (size_t)n_cells;
        }
    }
    if (n_cells == 0) return 0;
    int32_t cells = n_cells;
    npfem_handle* hs[1] = {h};
    // a synchronous step starts on an idle GPU, where the idle-SM blocks can be placed
    // before the clusters and cost cluster slots (measured: slower), so it runs without
    const int fill = h->opts.fill_idle_sms;
    h->opts.fill_idle_sms = 0;
    // pinned host buffers mapped into the device's address space are stepped in place:
    // the solver's loads at the start of a cell and its stores at the end move x, v and
    // F_ext over the host link while other cells compute, instead of copies before and
    // after the step
    void* xd = mapped_host(x_host);
    void* vd = mapped_host(v_host);
    void* fd = mapped_host(const_cast<void*>(f_host));
    void* sd = stats_host ? mapped_host(stats_host) : nullptr;
    if (xd && vd && fd && (!stats_host || sd)) {
        int rc = npfem_step(hs, 1, &cells, xd, vd, fd, dt, stream, static_cast<npfem_cell_stats*>(sd));
        h->opts.fill_idle_sms = fill;
        if (rc) return rc;
        NPFEM_CUDA(cudaStreamSynchronize(s));
        return 0;
    }
    cudaError_t e = cudaMemcpyAsync(h->hx, x_host, bytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h->hv, v_host, bytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h->hf, f_host, bytes, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) {
        h->opts.fill_idle_sms = fill;
        return fail(NPFEM_ERR_CUDA, std::string("npfem_step_host copies in: ") + cudaGetErrorString(e));
    }
    int rc = npfem_step(hs, 1, &cells, h->hx, h->hv, h->hf, dt, stream, stats_host ? h->hstats : nullptr);
    h->opts.fill_idle_sms = fill;
    if (rc) return rc;
    NPFEM_CUDA(cudaMemcpyAsync(x_host, h->hx, bytes, cudaMemcpyDeviceToHost, s));
    NPFEM_CUDA(cudaMemcpyAsync(v_host, h->hv, bytes, cudaMemcpyDeviceToHost, s));
    if (stats_host)
        NPFEM_CUDA(cudaMemcpyAsync(stats_host, h->hstats, sizeof(npfem_cell_stats) * n_cells, cudaMemcpyDeviceToHost, s));
    NPFEM_CUDA(cudaStreamSynchronize(s));
    return 0;
}

int npfem_eval(npfem_handle* h, int n_cells, const void* x, const void* y, void* grad, double* parts, void* stream)
{
    if (!h || n_cells < 0 || !x || !y || !grad || !parts) return fail(NPFEM_ERR_INVALID_ARG, "null argument");
    DeviceGuard guard(h->device);
    std::lock_guard<std::mutex> lk(h->mu);
    npfem_handle* hs[1] = {h};
    int32_t cells = n_cells;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (h->precision == NPFEM_PREC_FP64)
        return run_cells<double>(hs, 1, &cells, (double*)x, nullptr, nullptr, (const double*)y, (double*)grad, parts,
                                 nullptr, 1, s);
    return run_cells<float>(hs, 1, &cells, (float*)x, nullptr, nullptr, (const float*)y, (float*)grad, parts, nullptr,
                            1, s);
}

int npfem_ws_guess(npfem_handle* h, int n_cells, const float* x, const float* v, const float* f, float* x1, void* stream)
{
    if (!h || n_cells < 0 || !x || !v || !f || !x1) return fail(NPFEM_ERR_INVALID_ARG, "npfem_ws_guess: null argument");
    if (h->precision == NPFEM_PREC_FP64) return fail(NPFEM_ERR_INVALID_ARG, "npfem_ws_guess: FP32 state handles only");
    DeviceGuard guard(h->device);
    std::lock_guard<std::mutex> lk(h->mu);
    if (!h->tf.ws_mode || !h->tf.mlp) return fail(NPFEM_ERR_INVALID_ARG, "npfem_ws_guess: no warm start installed");
    if (n_cells == 0) return 0;
    NPFEM_CUDA(launch_ws_increments(h, n_cells, x, v, f, x1, true, static_cast<cudaStream_t>(stream)));
    return 0;
}

int npfem_check_device(npfem_handle* h)
{
    if (!h) return fail(NPFEM_ERR_INVALID_ARG, "null handle");
    DeviceGuard guard(h->device);
    NPFEM_CUDA(cudaDeviceSynchronize());
    unsigned flag = 0;
    NPFEM_CUDA(cudaMemcpy(&flag, h->work + 2, sizeof(unsigned), cudaMemcpyDeviceToHost));
    if (flag) {
        NPFEM_CUDA(cudaMemset(h->work + 2, 0, sizeof(unsigned)));
        return fail(NPFEM_ERR_TIMEOUT, "a bounded device wait gave up in a previous step (tensor-core MMA completion)");
    }
    return 0;
}

int npfem_flag_wait_timeout(npfem_handle* h)
{
    if (!h) return fail(NPFEM_ERR_INVALID_ARG, "null handle");
    DeviceGuard guard(h->device);
    NPFEM_CUDA(cudaDeviceSynchronize());
    const unsigned one = 1u;
    NPFEM_CUDA(cudaMemcpy(h->work + 2, &one, sizeof(unsigned), cudaMemcpyHostToDevice));
    return 0;
}

int npfem_get_inverse(npfem_handle* h, double* out_host)
{
    if (!h || !out_host) return fail(NPFEM_ERR_INVALID_ARG, "null argument");
    DeviceGuard guard(h->device);
    NPFEM_CUDA(cudaMemcpy(out_host, h->ainv64, sizeof(double) * (size_t)h->n * h->n, cudaMemcpyDeviceToHost));
    return 0;
}

int npfem_get_rest_info(npfem_handle* h, double* masses_host, double* scalars_host)
{
    if (!h) return fail(NPFEM_ERR_INVALID_ARG, "null handle");
    if (masses_host) memcpy(masses_host, h->host.mass.data(), sizeof(double) * h->n);
    if (scalars_host) {
        scalars_host[0] = h->host.V0;
        scalars_host[1] = h->host.A0;
        scalars_host[2] = h->host.lbar;
        scalars_host[3] = h->host.mtotal;
    }
    return 0;
}

}  // extern "C"
