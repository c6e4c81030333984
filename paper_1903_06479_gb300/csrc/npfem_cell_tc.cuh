#pragma once

#include "npfem_cell.cuh"

namespace npfem {
namespace {

// ---------------------------------------------------------------------------------
// Tensor-core contraction: a cluster of ceil(n / 128) blocks, one block per SM, each
// holding rows [128 r, 128 r + 128) of A^-1 (BF16) in tensor memory for the whole
// launch.  Blocks solve their cells independently; a contraction is a request that
// every block of the cluster serves asynchronously:
//   request -> the requesting block writes its vector (BF16) into rows 3 r + c of the
//              B operand of every block (DSMEM) and sets its bit in every block's
//              pending mask (release);
//   serve   -> at its next poll point a block takes its pending mask (acquire),
//              issues ceil(n/16) tcgen05.mma (M 128, N 16/32, K 16, A from TMEM, B
//              from shared memory, FP32 accumulate in TMEM) for the whole batch,
//              reads its 128 result rows and writes each requester's three columns
//              into that requester's contraction vector (DSMEM), then arrives on the
//              requester's delivery barrier (release);
//   wait    -> the requester serves at its own poll points until all blocks of the
//              cluster have delivered.
// Poll points: while waiting for a result, and between the solver's phases.  A block
// whose cells are done keeps serving until every block of the cluster is done.
// ---------------------------------------------------------------------------------

// Writes BF16(src) (3 rows of the cell, zero beyond n) into rows 3 rank + c of the B
// operand of every block in the cluster.  If with_residual, writes instead the
// refinement residual e = src - H~ r (H~ = ms M + L, sparse FP32) for r = R.
// tmp: 3 x n_pad scratch (the bending buffer, idle outside the evaluation).
template <typename T>
__device__ void tc_post(const TopoDev<T>& tp, const T* src, const T* R, bool with_residual, unsigned char* bbuf,
                        uint32_t rank, uint32_t cs, T* tmp)
{
    const int n = tp.n, np = tp.n_pad, kpad = tp.kpad, tid = threadIdx.x, NT = blockDim.x;
    const int chunks = 3 * (kpad >> 3);
    const uint32_t local = tc::smem_addr(bbuf);
    if (with_residual) {
        refine_residual(tp, src, R, tmp);
        src = tmp;
    }
    for (int q = tid; q < chunks; q += NT) {
        const int c = q / (kpad >> 3), kb = q - c * (kpad >> 3);
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = 8 * kb + u;
            v[u] = k < n ? (float)src[c * np + k] : 0.f;
        }
        const uint4 w = make_uint4(tc::pack_bf16(v[0], v[1]), tc::pack_bf16(v[2], v[3]), tc::pack_bf16(v[4], v[5]),
                                   tc::pack_bf16(v[6], v[7]));
        const uint32_t off = tc::b_offset(3 * (int)rank + c, 8 * kb, kpad);
        for (uint32_t d = 0; d < cs; ++d) tc::st_remote_v4(tc::map_rank(local + off, d), w);
    }
}

// The asynchronous rounds of one block (see above).  Every method is called by all
// threads of the block (control flow block-uniform).
template <typename T, int NCOL>
struct TcRounds {
    CellShared<T>* sh;
    const TopoDev<T>* tp;
    unsigned char* bbuf;
    T* GCv;
    unsigned* err;
    uint32_t tbase, dcol, idesc, sbo, bbase, rank, cs;
    uint32_t nserv, nreq;

    // Serves the requests pending at this block, if any.
    __device__ void serve()
    {
        const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
        if (tid == 0) {
            uint32_t b;
            asm volatile("atom.acquire.cluster.shared::cluster.exch.b32 %0, [%1], 0;"
                         : "=r"(b)
                         : "r"(tc::smem_addr(&sh->pend))
                         : "memory");
            sh->batch = b;
        }
        __syncthreads();
        const uint32_t batch = sh->batch;
        if (batch == 0u) return;
        const int kpad = tp->kpad, n = tp->n, np = tp->n_pad;
        if (tid == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int ks = 0; ks < (kpad >> 4); ++ks) {
                const uint64_t bd = tc::smem_desc(bbase + (uint32_t)ks * 256u, 128u, sbo);
                const uint32_t ta = tbase + (uint32_t)(ks * 8);
                const uint32_t acc = ks > 0;
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(tbase + dcol),
                    "r"(ta), "l"(bd), "r"(idesc), "r"(acc));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                tc::smem_addr(&sh->mbar)));
        }
        uint32_t done = 0;
        for (int it = 0; it < (1 << 22) && !done; ++it) {
            asm volatile(
                "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                : "=r"(done)
                : "r"(tc::smem_addr(&sh->mbar)), "r"(nserv & 1u));
        }
        if (!done && tid == 0) atomicExch(err, 1u);  // reported to the host; results invalid
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (warp < 4) {
            float dv[NCOL];
            tc::tmem_ld<NCOL>(tbase + ((uint32_t)(32 * warp) << 16) + dcol, dv);
            const int row = 128 * (int)rank + 32 * warp + lane;
            if (row < n) {
#pragma unroll
                for (int d = 0; d < NCOL / 3 && d < 8; ++d) {
                    if (!((batch >> d) & 1u)) continue;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const uint32_t loc = tc::smem_addr(GCv + c * np + row);
                        tc::st_remote_f32(tc::map_rank(loc, (uint32_t)d), dv[3 * d + c]);
                    }
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (tid < (int)cs && ((batch >> tid) & 1u)) {
            // the results written above (other threads, ordered by the barrier) are
            // released with the arrival
            const uint32_t rb = tc::map_rank(tc::smem_addr(&sh->dbar), (uint32_t)tid);
            asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(rb) : "memory");
        }
        ++nserv;
    }

    // r = A^-1 src into GCv (BF16 operands, FP32 accumulation); with refine one more
    // sweep r += A^-1 (src - H~ r).  tmp, keep: 3 x n_pad scratch.
    __device__ void contract(const T* src, bool refine, T* tmp, T* keep)
    {
        request(src, false, tmp);
        if (refine) {
            const int N3 = 3 * tp->n_pad;
            for (int e = threadIdx.x; e < N3; e += blockDim.x) keep[e] = GCv[e];
            __syncthreads();
            request(src, true, tmp);
            for (int e = threadIdx.x; e < N3; e += blockDim.x) GCv[e] += keep[e];
            __syncthreads();
        }
    }

    // Posts src (or the refinement residual of src for r = GCv) and waits, serving, for
    // the cs deliveries.
    __device__ void request(const T* src, bool residual, T* tmp)
    {
        const int tid = threadIdx.x;
        tc_post(*tp, src, GCv, residual, bbuf, rank, cs, tmp);
        asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");
        __syncthreads();
        if (tid < (int)cs) {
            const uint32_t pa = tc::map_rank(tc::smem_addr(&sh->pend), (uint32_t)tid);
            asm volatile("red.release.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(pa), "r"(1u << rank) : "memory");
        }
        const uint32_t par = nreq & 1u;
        bool ok = false;
        for (int it = 0; it < (1 << 22); ++it) {
            serve();
            if (tid == 0) {
                uint32_t d;
                asm volatile(
                    "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                    "selp.u32 %0, 1, 0, p;\n}"
                    : "=r"(d)
                    : "r"(tc::smem_addr(&sh->dbar)), "r"(par)
                    : "memory");
                // the error word (global memory) only now and then: each read costs a round trip
                sh->flag = d | ((it & 255) == 255 && *reinterpret_cast<volatile unsigned*>(err) != 0u ? 2u : 0u);
            }
            __syncthreads();
            const uint32_t f = sh->flag;
            if (f & 1u) {
                ok = true;
                break;
            }
            if (f & 2u) break;  // another block gave up: stop waiting
        }
        if (!ok && tid == 0) atomicExch(err, 1u);
        ++nreq;
    }

    // The block's cells are done: tell every block, then serve until all are done.
    __device__ void finish_and_drain()
    {
        const int tid = threadIdx.x;
        __syncthreads();
        if (tid < (int)cs) {
            const uint32_t fa = tc::map_rank(tc::smem_addr(&sh->fin), (uint32_t)tid);
            asm volatile("red.release.cluster.shared::cluster.add.u32 [%0], 1;" ::"r"(fa) : "memory");
        }
        bool ok = false;
        for (int it = 0; it < (1 << 24); ++it) {
            serve();
            if (tid == 0) {
                uint32_t f;
                asm volatile("ld.acquire.cluster.shared::cluster.u32 %0, [%1];"
                             : "=r"(f)
                             : "r"(tc::smem_addr(&sh->fin))
                             : "memory");
                sh->flag = (f >= cs ? 1u : 0u) |
                           ((it & 255) == 255 && *reinterpret_cast<volatile unsigned*>(err) != 0u ? 2u : 0u);
            }
            __syncthreads();
            const uint32_t f = sh->flag;
            if (f & 1u) {
                ok = true;
                break;
            }
            if (f & 2u) break;
        }
        if (!ok && tid == 0) atomicExch(err, 1u);
        // nothing is left pending: every request was delivered before its block finished
    }
};

template <typename T, int NCOL, int K>
__global__ void __launch_bounds__(512, 1) cell_kernel_tc(const __grid_constant__ LaunchArgs<T> a)
{
    unsigned char* smem = smem_dyn;
    const GroupDesc<T>& gd = a.g[0];
    const TopoDev<T>& tp = gd.topo;
    CellShared<T>* sh = cell_shared<T>(smem);
    unsigned char* bbuf = smem + kFixedSmem;  // B operand: NCOL rows x kpad BF16
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = tc::cta_rank(), cs = (uint32_t)a.p.cluster;
    const int kpad = tp.kpad;
    const uint32_t acols = (uint32_t)(kpad >> 1);
    const uint32_t dcol = (acols + 31u) & ~31u;

    // ---- set-up: zero B, flags, barriers, TMEM allocation, A^-1 rows of this block into TMEM
    for (int q = tid; q < NCOL * kpad / 8; q += blockDim.x) reinterpret_cast<uint4*>(bbuf)[q] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        sh->pend = 0u;
        sh->fin = 0u;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc::smem_addr(&sh->mbar)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_addr(&sh->dbar)), "r"(cs));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
            tc::smem_addr(&sh->taddr)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tbase = sh->taddr;
    if (warp < 4) {
        const int row = 128 * (int)rank + 32 * warp + lane;
        const uint32_t* src = reinterpret_cast<const uint32_t*>(tp.ainv_lp) + (size_t)row * (kpad >> 1);
        for (int c0 = 0; c0 < (int)acols; c0 += 8) {
            uint32_t r[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) r[j] = __ldg(&src[c0 + j]);
            const uint32_t ta = tbase + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0;
            asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(ta), "r"(r[0]),
                         "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]));
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    tc::cluster_sync();  // every block's barriers and flags are initialised
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    CellSolver<T, K> S;
    S.bind(a, gd, smem);
    TcRounds<T, NCOL> R;
    R.sh = sh;
    R.tp = &tp;
    R.bbuf = bbuf;
    R.GCv = S.GCv;
    R.err = &a.work[2];
    R.tbase = tbase;
    R.dcol = dcol;
    R.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NCOL >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    R.sbo = (uint32_t)(kpad >> 3) * 128u;
    R.bbase = tc::smem_addr(bbuf);
    R.rank = rank;
    R.cs = cs;
    R.nserv = 0u;
    R.nreq = 0u;
    const bool refine = a.p.refine != 0;

    for (;;) {
        R.serve();
        const long long item = next_item(a, smem);
        if (item < 0) break;
        S.begin(item, item);
        const bool wants = S.wants_direction();
        if (a.need && wants && tid == 0) atomicAdd(a.need, 1u);
        while (S.wants_direction()) {
            R.serve();
            S.first_loop();
            R.contract(S.Dv, refine, S.WRv, S.ut);  // r = H0 q
            S.second_loop();
            if (!S.descent()) {
                // not a descent direction: drop the history, d = -H~^-1 g
                S.count = 0;
                R.contract(S.g, refine, S.WRv, S.ut);
                S.negate_direction();
            }
            if (!S.line_search_update()) break;
        }
        S.finish();
    }
    R.finish_and_drain();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    tc::cluster_sync();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase));
    release_counters(a.work, a.total_blocks);
}

}  // namespace
}  // namespace npfem
