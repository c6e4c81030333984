// Immersed-boundary force step upstream of the solver (Sec. 2.3 of arXiv:1903.06479):
// the external force of Eq. Fext sampled from a lattice stress field, interpolation
// of a lattice velocity to the membrane vertices, and the multi-direct forcing
// iteration that makes the fluid follow the membrane (Steps 0-5 of Sec. 2.3).
//
// The four-point kernel w(r) of Sec. 2.3 gives each vertex a 4 x 4 x 4 stencil of
// lattice nodes with weights w(r_x - i) w(r_y - j) w(r_z - k).  Four lanes handle
// one vertex, lane q the nodes of x offset q, so that a stencil row of four consecutive
// nodes is one 64-byte (velocity, force) or 128-byte (stress) access: what bounds these
// kernels is the number of L1/L2 sectors and atomic operations per stencil.  The lanes
// share the vertex's triangles for its area share A_k (a third of its triangles' areas)
// and unit normal n_k at the current positions; their stencil sums meet in two shuffles.
// Lattice coordinates are sums of two floats (lattice_base), weights and sums FP32.
// Measured on 1024 cells of 642 vertices, 121^3 nodes: forcing with three cycles (four
// spreads and four gathers) 3.0 -> 1.02 ms against one thread per vertex with scalar
// atomics and FP64 coordinates.
//
// Conventions (the paper prints the formulas in lattice units, dx = 1):
//  * interpolation u(X_k) = sum_x u(x) w w w (the dx^3 of W dx^3 cancels);
//  * Eq. Fext: F_k = rho A_k (sum_x sigma(x) w w w) n_k;
//  * spreading f(x) = sum_k f_k (w w w / dx^3) A_k dx: a membrane one spacing thick, so
//    that spreading is the adjoint of interpolation;
//  * stencil nodes outside the lattice contribute nothing.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "npfem_device.cuh"
#include "npfem_internal.h"

namespace npfem {
namespace {

struct LatDev {
    float oh[3], ol[3];  // origin and 1 / dx as sums of two floats
    float ih, il;
    float dx;
    int nx, ny, nz;
};

struct IbmGroup {
    TopoDev<float> topo;
    long long vert_begin;  // first global vertex index of the group
    long long cell_begin;  // first global cell of the group
    long long state_off;   // element offset of the group's first cell in the SoA arrays
    int cells;
};

struct IbmArgs {
    IbmGroup g[kMaxGroups];
    int n_groups;
    long long total_verts, total_cells;
    LatDev lat;
    const float* x;       // SoA positions
    const float* field;   // sigma [nodes][8] (forces) or a velocity [nodes][4]
    const float* field2;  // forcing: the lattice force [nodes][4] (update phase)
    const float* uvert;   // forcing: membrane vertex velocities U_k (SoA)
    float* out;           // SoA vertex output
    float* lat_out;       // forcing: lattice force [nodes][4] (spread phase)
    int lat_vec;          // lat_out is 16-byte aligned (vector reductions)
    float rho, dt;
    int mode;             // forces: 0 full stencil, 1 exterior nodes, 2 farthest exterior node
    int phase;            // forcing: 0 f = (U - u*)/dt, 1 spread f, 2 f += (U - u_l)/dt
};

// The paper's one-dimensional four-point kernel (lattice units).
__device__ __forceinline__ float w4(float r)
{
    const float a = fabsf(r);
    if (a <= 1.f) return 0.125f * (3.f - 2.f * a + sqrtf(1.f + 4.f * a - 4.f * a * a));
    if (a <= 2.f) return 0.125f * (5.f - 2.f * a - sqrtf(fmaxf(-7.f + 12.f * a - 4.f * a * a, 0.f)));
    return 0.f;
}

struct Stencil {
    int i0, j0, k0;      // first node in each direction
    float t[3];          // fractional lattice offset of the point in [0, 1)
    float w[3][4];       // weights of nodes i0 + a, a = 0..3
};

// First node of a coordinate's stencil and its fractional offset t in [0, 1).  The lattice
// coordinate (X - origin) / dx is carried as a sum of two floats (error-free difference
// and product, about 48 bits: a single float would round the offset in a 100 um domain to
// ~1e-5; in FP64 this alone took a third of the forcing's time on the narrow FP64 pipe).  A
// point far outside the lattice (or not finite) gets a stencil with no nodes.
__device__ __forceinline__ int lattice_base(const LatDev& L, int d, float X, float* t)
{
    const float oh = d == 0 ? L.oh[0] : (d == 1 ? L.oh[1] : L.oh[2]), ol = d == 0 ? L.ol[0] : (d == 1 ? L.ol[1] : L.ol[2]);
    const float dh = X - oh, bb = dh - X;
    const float dl = ((X - (dh - bb)) - (oh + bb)) - ol;
    const float ph = dh * L.ih;
    if (!(fabsf(ph) <= 1.0e6f)) {
        *t = 0.f;
        return ph > 0.f ? 999999 : -1000001;
    }
    const float pl = fmaf(dh, L.ih, -ph) + fmaf(dh, L.il, dl * L.ih);
    float f = floorf(ph);
    float r = (ph - f) + pl;
    if (r < 0.f) {
        r += 1.f;
        f -= 1.f;
    } else if (r >= 1.f) {
        r -= 1.f;
        f += 1.f;
    }
    *t = r;
    return (int)f - 1;
}

// The stencil of vertex i (SoA positions xc of n vertices) for its four lanes: lane d < 3
// takes dimension d (its offset and four weights) and the lanes exchange them.  wq: lane q's weight along x.
__device__ __forceinline__ void make_stencil(const LatDev& L, const float* xc, int n, int i, int q, Stencil& s, float* wq)
{
    const int d = min(q, 2), from = (threadIdx.x & 31) & ~3;
    float t;
    const int base = lattice_base(L, d, xc[d * n + i], &t);
    const float w[4] = {w4(t + 1.f), w4(t), w4(t - 1.f), w4(t - 2.f)};
    s.i0 = __shfl_sync(kFull, base, from);
    s.j0 = __shfl_sync(kFull, base, from + 1);
    s.k0 = __shfl_sync(kFull, base, from + 2);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        s.t[e] = __shfl_sync(kFull, t, from + e);
#pragma unroll
        for (int k = 0; k < 4; ++k) s.w[e][k] = __shfl_sync(kFull, w[k], from + e);
    }
    *wq = q == 0 ? s.w[0][0] : (q == 1 ? s.w[0][1] : (q == 2 ? s.w[0][2] : s.w[0][3]));
}

// Global vertex index -> (group, its topology, cell, vertex).
__device__ __forceinline__ const IbmGroup& locate(const IbmArgs& a, long long gv, long long* cell, int* vert)
{
    int gi = 0;
    while (gi + 1 < a.n_groups && gv >= a.g[gi + 1].vert_begin) ++gi;
    const IbmGroup& G = a.g[gi];
    const long long local = gv - G.vert_begin;
    if (local <= UINT_MAX) {
        // every lane divides: in 32 bits wherever the group has fewer vertices
        const unsigned l = (unsigned)local, n = (unsigned)G.topo.n, c = l / n;
        *cell = c;
        *vert = (int)(l - c * n);
    } else {
        *cell = local / G.topo.n;
        *vert = (int)(local - *cell * G.topo.n);
    }
    return G;
}

__device__ __forceinline__ bool node_in(const LatDev& L, int i, int j, int k)
{
    return (unsigned)i < (unsigned)L.nx && (unsigned)j < (unsigned)L.ny && (unsigned)k < (unsigned)L.nz;
}

__device__ __forceinline__ long long node_index(const LatDev& L, int i, int j, int k)
{
    return ((long long)k * L.ny + j) * L.nx + i;
}

// Sum over the four lanes of a vertex.
__device__ __forceinline__ float sum4(float v)
{
    v += __shfl_xor_sync(kFull, v, 1);
    return v + __shfl_xor_sync(kFull, v, 2);
}

// vertex_area_normal() of vertex i shared by its four lanes (lane q takes every fourth
// incident triangle); the normal's sums only when N is given.
template <bool kNormal>
__device__ __forceinline__ void area_normal4(const TopoDev<float>& tp, const float* xc, int i, int q, float* A, float* nv)
{
    const int n_ = tp.n;
    float N[3] = {0.f, 0.f, 0.f}, S = 0.f;
    const int b0 = __ldg(&tp.inc_ptr[i]), b1 = __ldg(&tp.inc_ptr[i + 1]);
    for (int e = b0 + q; e < b1; e += 4) {
        const ushort4 tv = __ldg(&tp.tri[__ldg(&tp.inc_idx[e]) >> 2]);
        const int p0 = tv.x, p1 = tv.y, p2 = tv.z;
        float e1[3], e2[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float x0 = xc[c * n_ + p0];
            e1[c] = xc[c * n_ + p1] - x0;
            e2[c] = xc[c * n_ + p2] - x0;
        }
        const float cr[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
        if (kNormal)
#pragma unroll
            for (int c = 0; c < 3; ++c) N[c] += 0.5f * cr[c];
        S += sqrtf(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]);
    }
    *A = sum4(S) * (1.f / 6.f);
    if (kNormal) {
#pragma unroll
        for (int c = 0; c < 3; ++c) N[c] = sum4(N[c]);
        const float inv = rsqrtf(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) nv[c] = N[c] * inv;
    }
}

// Vertices per block of 256 threads; the loops below run to the rounded count so that the
// shuffles see whole warps (vertices past the end repeat the last and write nothing).
constexpr int kVertsPerBlock = 64;

// Row (b, c) of a vertex's stencil, lane q's node: its index, or -1 outside the lattice.
__device__ __forceinline__ long long row_node(const LatDev& L, const Stencil& s, int q, int b, int c)
{
    const int ii = s.i0 + q, jj = s.j0 + b, kk = s.k0 + c;
    return node_in(L, ii, jj, kk) ? node_index(L, ii, jj, kk) : -1;
}

// Eq. Fext, four lanes per vertex.
__global__ void __launch_bounds__(256) ibm_forces_kernel(const __grid_constant__ IbmArgs a)
{
    const LatDev& L = a.lat;
    const int q = threadIdx.x & 3;
    for (long long v0 = blockIdx.x * (long long)kVertsPerBlock; v0 < a.total_verts; v0 += (long long)gridDim.x * kVertsPerBlock) {
        const long long gv = v0 + (threadIdx.x >> 2);
        const bool live = gv < a.total_verts;
        long long cell;
        int i;
        const IbmGroup& G = locate(a, live ? gv : a.total_verts - 1, &cell, &i);
        const int n = G.topo.n;
        const long long so = G.state_off + cell * 3LL * n;
        const float* xc = a.x + so;
        float A, nv[3];
        area_normal4<true>(G.topo, xc, i, q, &A, nv);
        Stencil s;
        float wq;
        make_stencil(L, xc, n, i, q, s, &wq);
        float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, wsum = 0.f, dbest = -1.f;
        int first = 64;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const long long nd = row_node(L, s, q, b, c);
                if (nd < 0) continue;
                float wgt = wq * s.w[1][b] * s.w[2][c];
                if (a.mode != 0) {
                    // offset node - X in um; exterior when it points along n
                    const float d[3] = {((float)(q - 1) - s.t[0]) * L.dx, ((float)(b - 1) - s.t[1]) * L.dx,
                                        ((float)(c - 1) - s.t[2]) * L.dx};
                    if (!(d[0] * nv[0] + d[1] * nv[1] + d[2] * nv[2] > 0.f)) continue;
                    if (a.mode == 2) {
                        const float d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
                        if (!(d2 > dbest)) continue;  // keep the first among equals
                        dbest = d2;
                        first = 16 * c + 4 * b + q;
                        wgt = 1.f;
#pragma unroll
                        for (int e = 0; e < 6; ++e) acc[e] = 0.f;
                        wsum = 0.f;
                    }
                }
                const float4* P = reinterpret_cast<const float4*>(a.field + 8 * nd);
                const float4 s0 = __ldg(P), s1 = __ldg(P + 1);
                acc[0] += wgt * s0.x; acc[1] += wgt * s0.y; acc[2] += wgt * s0.z;
                acc[3] += wgt * s0.w; acc[4] += wgt * s1.x; acc[5] += wgt * s1.y;
                wsum += wgt;
            }
        if (a.mode == 2) {
            // the farthest node of the four lanes' (the first in z, y, x order among equals)
            float db = dbest;
            int fb = first;
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                const float d2 = __shfl_xor_sync(kFull, db, o);
                const int f2 = __shfl_xor_sync(kFull, fb, o);
                if (d2 > db || (d2 == db && f2 < fb)) {
                    db = d2;
                    fb = f2;
                }
            }
            if (fb != first) {
#pragma unroll
                for (int e = 0; e < 6; ++e) acc[e] = 0.f;
                wsum = 0.f;
            }
        }
#pragma unroll
        for (int e = 0; e < 6; ++e) acc[e] = sum4(acc[e]);
        if (a.mode != 0) {
            wsum = sum4(wsum);
            const float inv = wsum > 0.f ? 1.f / wsum : 0.f;
#pragma unroll
            for (int e = 0; e < 6; ++e) acc[e] *= inv;
        }
        // (xx, yy, zz, xy, xz, yz) times n, scaled by rho A_k: lane q writes component q
        const float sc = a.rho * A;
        const float f = q == 0 ? acc[0] * nv[0] + acc[3] * nv[1] + acc[4] * nv[2]
                      : q == 1 ? acc[3] * nv[0] + acc[1] * nv[1] + acc[5] * nv[2]
                               : acc[4] * nv[0] + acc[5] * nv[1] + acc[2] * nv[2];
        if (live && q < 3) a.out[so + q * n + i] = sc * f;
    }
}

// Stencil sum of a [nodes][4] field (plus dt times a second one, if given), over the
// four lanes of a vertex.  Eight rows in flight per lane and four blocks per SM: 642 x 3000,
// dx 1 um, interpolation 214 us, against 240 with all sixteen rows and three blocks and 344
// with eight rows and six blocks, whose registers spill.
__device__ __forceinline__ void gather4(const LatDev& L, const Stencil& s, int q, float wq, const float* F, const float* F2,
                                        float dt, float out[3])
{
    constexpr int R = 8;
    float o[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int r0 = 0; r0 < 16; r0 += R) {
        float4 u[R];
#pragma unroll
        for (int h = 0; h < R; ++h) {
            const long long nd = row_node(L, s, q, (r0 + h) & 3, (r0 + h) >> 2);
            u[h] = nd >= 0 ? __ldg(reinterpret_cast<const float4*>(F) + nd) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int h = 0; h < R; ++h) {
            const int r = r0 + h;
            const float wgt = wq * s.w[1][r & 3] * s.w[2][r >> 2];
            if (F2) {
                // the corrected lattice velocity u* + dt f (Step 2) is formed on the fly;
                // F2 is written by an earlier launch, so a plain (coherent) load
                const long long nd = row_node(L, s, q, r & 3, r >> 2);
                if (nd >= 0) {
                    const float4 f = reinterpret_cast<const float4*>(F2)[nd];
                    u[h].x += dt * f.x;
                    u[h].y += dt * f.y;
                    u[h].z += dt * f.z;
                }
            }
            o[0] += wgt * u[h].x;
            o[1] += wgt * u[h].y;
            o[2] += wgt * u[h].z;
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = sum4(o[c]);
}

// One 16-byte reduction per node instead of three scalar atomics (vec: p is 16-byte
// aligned; the node's unused fourth value gains zero).
__device__ __forceinline__ void red4(float* p, float x, float y, float z, int vec)
{
    if (!vec) {
        atomicAdd(p, x);
        atomicAdd(p + 1, y);
        atomicAdd(p + 2, z);
        return;
    }
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_global(p)), "f"(x), "f"(y), "f"(z),
                 "f"(0.f)
                 : "memory");
}

// What a vertex's four lanes do with its stencil sum u of the velocity: interpolation
// (phase -1) or Steps 0 and 4 of the multi-direct forcing.
__device__ __forceinline__ void take_sum(const IbmArgs& a, long long so, int n, int i, int q, bool live, const float (&u)[3])
{
    if (!live || q > 2) return;
    const float uq = q == 0 ? u[0] : (q == 1 ? u[1] : u[2]);
    const long long at = so + q * n + i;
    if (a.phase < 0) {
        a.out[at] = uq;
        return;
    }
    const float slip = (a.uvert[at] - uq) * (1.f / a.dt);
    a.out[at] = a.phase == 0 ? slip : a.out[at] + slip;
}

// One vertex of a phase straight on the lattice.
template <bool kSpread>
__device__ __forceinline__ void vertex_phase(const IbmArgs& a, const IbmGroup& G, long long cell, int i, int q, bool live)
{
    const LatDev& L = a.lat;
    const int n = G.topo.n;
    const long long so = G.state_off + cell * 3LL * n;
    const float* xc = a.x + so;
    Stencil s;
    float wq;
    make_stencil(L, xc, n, i, q, s, &wq);
    if constexpr (kSpread) {
        // Step 1: spread f_k with weight A_k dx / dx^3 per unit stencil weight
        float A;
        area_normal4<false>(G.topo, xc, i, q, &A, nullptr);
        const float* o = a.out + so;
        const float sc = A / (L.dx * L.dx) * wq;
        const float f[3] = {sc * o[i], sc * o[n + i], sc * o[2 * n + i]};
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const long long nd = row_node(L, s, q, r & 3, r >> 2);
            const float wgt = s.w[1][r & 3] * s.w[2][r >> 2];
            if (live && nd >= 0) red4(a.lat_out + 4 * nd, wgt * f[0], wgt * f[1], wgt * f[2], a.lat_vec);
        }
    } else {
        float u[3];
        gather4(L, s, q, wq, a.field, a.phase == 2 ? a.field2 : nullptr, a.dt, u);
        take_sum(a, so, n, i, q, live, u);
    }
}

// Velocity interpolation (phase -1) and the phases of the multi-direct forcing, vertex by
// vertex.  The gathers run with four blocks per SM (gather4), the spread with three.
template <bool kSpread>
__global__ void __launch_bounds__(256, kSpread ? 3 : 4) ibm_forcing_kernel(const __grid_constant__ IbmArgs a)
{
    for (long long v0 = blockIdx.x * (long long)kVertsPerBlock; v0 < a.total_verts; v0 += (long long)gridDim.x * kVertsPerBlock) {
        const long long gv = v0 + (threadIdx.x >> 2);
        const bool live = gv < a.total_verts;
        long long cell;
        int i;
        const IbmGroup& G = locate(a, live ? gv : a.total_verts - 1, &cell, &i);
        vertex_phase<kSpread>(a, G, cell, i, threadIdx.x & 3, live);
    }
}

// The gathering phases, a block per cell: the lattice nodes around the cell (a box of the
// stencils' extent) pass through shared memory, read once instead of once per stencil that
// meets them (a 642-vertex cell has 41 K stencil nodes in a box of about 1.7 K).  A cell
// whose box does not fit goes vertex by vertex.  Spreading through such a box was slower
// than vertex by vertex, with atomics on shared sums (1024 cells of 642 vertices, four
// spreads and gathers: 3.2 against 2.1 ms) and with the vertices sorted by node (2.8 ms).
constexpr int kBoxNodes = 3000;

__global__ void __launch_bounds__(256, 3) ibm_gather_kernel(const __grid_constant__ IbmArgs a)
{
    extern __shared__ __align__(16) float4 box[];
    __shared__ int lo[3], hi[3];
    const LatDev& L = a.lat;
    const int tid = threadIdx.x, NT = blockDim.x, q = tid & 3;
    for (long long gc = blockIdx.x; gc < a.total_cells; gc += gridDim.x) {
        int gi = 0;
        while (gi + 1 < a.n_groups && gc >= a.g[gi + 1].cell_begin) ++gi;
        const IbmGroup& G = a.g[gi];
        const long long cell = gc - G.cell_begin;
        const int n = G.topo.n;
        const long long so = G.state_off + cell * 3LL * n;
        const float* xc = a.x + so;
        if (tid < 3) {
            lo[tid] = INT_MAX;
            hi[tid] = INT_MIN;
        }
        __syncthreads();
        int l[3] = {INT_MAX, INT_MAX, INT_MAX}, h[3] = {INT_MIN, INT_MIN, INT_MIN};
        for (int i = tid; i < n; i += NT) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                float t;
                const int b = lattice_base(L, d, xc[d * n + i], &t);
                l[d] = min(l[d], b);
                h[d] = max(h[d], b);
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            l[d] = __reduce_min_sync(kFull, l[d]);
            h[d] = __reduce_max_sync(kFull, h[d]);
            if ((tid & 31) == 0) {
                atomicMin(&lo[d], l[d]);
                atomicMax(&hi[d], h[d]);
            }
        }
        __syncthreads();
        const int x0 = lo[0], y0 = lo[1], z0 = lo[2];
        const long long ex = (long long)hi[0] - x0 + 4, ey = (long long)hi[1] - y0 + 4, ez = (long long)hi[2] - z0 + 4;
        const bool fits = ex <= kBoxNodes && ey <= kBoxNodes && ez <= kBoxNodes && ex * ey * ez <= kBoxNodes;
        const int bx = (int)ex, by = (int)ey, nodes = fits ? (int)(ex * ey * ez) : 0;
        for (int e = tid; e < nodes; e += NT) {
            const int k = e / (bx * by), j = (e - k * bx * by) / bx, ii = e - (k * by + j) * bx;
            float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
            if (node_in(L, x0 + ii, y0 + j, z0 + k)) {
                const long long nd = node_index(L, x0 + ii, y0 + j, z0 + k);
                u = __ldg(reinterpret_cast<const float4*>(a.field) + nd);
                if (a.phase == 2) {
                    // the corrected velocity u* + dt f (Step 2); f is written by an earlier launch
                    const float4 f = reinterpret_cast<const float4*>(a.field2)[nd];
                    u.x += a.dt * f.x;
                    u.y += a.dt * f.y;
                    u.z += a.dt * f.z;
                }
            }
            box[e] = u;
        }
        __syncthreads();
        for (int v0 = 0; v0 < n; v0 += NT >> 2) {
            const bool live = v0 + (tid >> 2) < n;
            const int i = live ? v0 + (tid >> 2) : n - 1;
            if (!fits) {
                vertex_phase<false>(a, G, cell, i, q, live);
                continue;
            }
            Stencil s;
            float wq;
            make_stencil(L, xc, n, i, q, s, &wq);
            const int at = ((s.k0 - z0) * by + (s.j0 - y0)) * bx + (s.i0 - x0) + q;
            float o[3] = {0.f, 0.f, 0.f}, u[3];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const float wgt = wq * s.w[1][r & 3] * s.w[2][r >> 2];
                const float4 f = box[at + ((r >> 2) * by + (r & 3)) * bx];
                o[0] += wgt * f.x;
                o[1] += wgt * f.y;
                o[2] += wgt * f.z;
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) u[c] = sum4(o[c]);
            take_sum(a, so, n, i, q, live, u);
        }
        __syncthreads();
    }
}

int fill_ibm(IbmArgs* a, npfem_handle* const* meshes, int n_groups, const int32_t* cells, const npfem_lattice* lat,
             const char* who)
{
    memset(a, 0, sizeof(*a));
    if (!meshes || n_groups < 1 || n_groups > kMaxGroups || !cells || !lat)
        return set_error(NPFEM_ERR_INVALID_ARG, std::string(who) + ": need 1..8 handles, cell counts and a lattice");
    if (!(lat->dx > 0.0) || lat->nx < 1 || lat->ny < 1 || lat->nz < 1 || !std::isfinite(lat->origin[0]) ||
        !std::isfinite(lat->origin[1]) || !std::isfinite(lat->origin[2]))
        return set_error(NPFEM_ERR_INVALID_ARG, std::string(who) + ": lattice needs dx > 0 and positive sizes");
    long long v = 0, st = 0;
    for (int g = 0; g < n_groups; ++g) {
        npfem_handle* h = meshes[g];
        if (!h || cells[g] < 0) return set_error(NPFEM_ERR_INVALID_ARG, std::string(who) + ": bad handle or cell count");
        if (h->precision == NPFEM_PREC_FP64 || h->device != meshes[0]->device)
            return set_error(NPFEM_ERR_INVALID_ARG, std::string(who) + ": FP32-state handles of one device only");
        a->g[g].topo = h->tf;
        a->g[g].vert_begin = v;
        a->g[g].cell_begin = a->total_cells;
        a->total_cells += cells[g];
        a->g[g].state_off = st;
        a->g[g].cells = cells[g];
        v += (long long)h->n * cells[g];
        st += 3LL * h->n * cells[g];
    }
    a->n_groups = n_groups;
    a->total_verts = v;
    for (int d = 0; d < 3; ++d) {
        a->lat.oh[d] = (float)lat->origin[d];
        a->lat.ol[d] = (float)(lat->origin[d] - (double)a->lat.oh[d]);
    }
    const double inv = 1.0 / lat->dx;
    a->lat.ih = (float)inv;
    a->lat.il = (float)(inv - (double)a->lat.ih);
    a->lat.dx = (float)lat->dx;
    a->lat.nx = lat->nx;
    a->lat.ny = lat->ny;
    a->lat.nz = lat->nz;
    return 0;
}

int ibm_grid(const npfem_handle* h, long long verts)
{
    const long long blocks = (verts + kVertsPerBlock - 1) / kVertsPerBlock;
    return (int)std::max<long long>(1, std::min<long long>(blocks, (long long)std::max(h->sm_count, 1) * 8));
}

// A phase over all vertices: gathers by a block per cell where the cells fill the GPU, a cell's
// stencils overlap enough to pay for its box, and the boxes fit (node_box); else vertex by
// vertex.  Step 4 reads two fields per node and gains earlier.  Vertex by vertex / box:
// interpolation of 642 x 160, 250, 1000 and 3000 cells at dx 1 um 24 / 32, 31 / 32, 80 / 72 and
// 214 / 206 us, of 1026 x 1000 121 / 101, of 258 x 3000 97 / 121; forcing with two cycles, 258 x
// 1000 394 / 374, 642 x 1000 877 / 793; at dx 0.5 um, where no box fits, 642 x 1000 1017 / 1338.
constexpr long long kBoxMinCells = 250, kBoxMinVerts = 500, kBoxMinVertsTwo = 200;
constexpr double kBoxMeanNodes = 2200.0;  // above, tilted cells pass kBoxNodes (dx below 0.82 um)

// Nodes of a cell's box at this spacing on average over its orientations (from the mesh's rest
// extent).
double node_box(const npfem_handle* h, double dx)
{
    const double e = h->rest_extent / dx + 5.0;
    return e * e * e;
}

cudaError_t launch_forcing(const IbmArgs& a, npfem_handle* const* meshes, double dx, cudaStream_t s)
{
    const npfem_handle* h = meshes[0];
    bool box = a.phase != 1 && a.total_cells >= kBoxMinCells &&
               a.total_verts >= (a.phase == 2 ? kBoxMinVertsTwo : kBoxMinVerts) * a.total_cells;
    for (int g = 0; g < a.n_groups && box; ++g) box = a.g[g].cells == 0 || node_box(meshes[g], dx) <= kBoxMeanNodes;
    if (box) {
        const int smem = kBoxNodes * (int)sizeof(float4);
        const int grid = (int)std::min<long long>(a.total_cells, (long long)std::max(h->sm_count, 1) * 4);
        ibm_gather_kernel<<<grid, 256, smem, s>>>(a);
    } else {
        const int grid = ibm_grid(h, a.total_verts);
        if (a.phase == 1) ibm_forcing_kernel<true><<<grid, 256, 0, s>>>(a);
        else ibm_forcing_kernel<false><<<grid, 256, 0, s>>>(a);
    }
    count_launch();
    return cudaGetLastError();
}

struct DevGuard {
    int prev = -1;
    explicit DevGuard(int dev)
    {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DevGuard()
    {
        int cur = -1;
        cudaGetDevice(&cur);
        if (prev >= 0 && cur != prev) cudaSetDevice(prev);
    }
};

int launch_err(const char* who, cudaError_t e)
{
    return set_error(NPFEM_ERR_CUDA, std::string(who) + ": " + cudaGetErrorString(e));
}

}  // namespace
}  // namespace npfem

using namespace npfem;

extern "C" int npfem_ibm_forces(npfem_handle* const* meshes, int n_groups, const int32_t* cells_per_group,
                                const float* x, const npfem_lattice* lattice, const float* sigma, double rho_fluid,
                                int mode, float* f_ext, void* stream)
{
    IbmArgs a;
    if (int rc = fill_ibm(&a, meshes, n_groups, cells_per_group, lattice, "npfem_ibm_forces")) return rc;
    if (!x || !sigma || !f_ext || mode < 0 || mode > 2 || !std::isfinite(rho_fluid))
        return set_error(NPFEM_ERR_INVALID_ARG, "npfem_ibm_forces: null array, mode outside 0..2 or bad rho");
    if (a.total_verts == 0) return 0;
    DevGuard guard(meshes[0]->device);
    a.x = x;
    a.field = sigma;
    a.out = f_ext;
    a.rho = (float)rho_fluid;
    a.mode = mode;
    ibm_forces_kernel<<<ibm_grid(meshes[0], a.total_verts), 256, 0, static_cast<cudaStream_t>(stream)>>>(a);
    count_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 0 : launch_err("npfem_ibm_forces", e);
}

extern "C" int npfem_ibm_interpolate(npfem_handle* const* meshes, int n_groups, const int32_t* cells_per_group,
                                     const float* x, const npfem_lattice* lattice, const float* u_lattice,
                                     float* u_vertex, void* stream)
{
    IbmArgs a;
    if (int rc = fill_ibm(&a, meshes, n_groups, cells_per_group, lattice, "npfem_ibm_interpolate")) return rc;
    if (!x || !u_lattice || !u_vertex) return set_error(NPFEM_ERR_INVALID_ARG, "npfem_ibm_interpolate: null array");
    if (a.total_verts == 0) return 0;
    DevGuard guard(meshes[0]->device);
    a.x = x;
    a.field = u_lattice;
    a.out = u_vertex;
    a.phase = -1;
    const cudaError_t e = launch_forcing(a, meshes, lattice->dx, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? 0 : launch_err("npfem_ibm_interpolate", e);
}

extern "C" int npfem_ibm_forcing(npfem_handle* const* meshes, int n_groups, const int32_t* cells_per_group,
                                 const float* x, const float* u_vertex, const npfem_lattice* lattice,
                                 const float* u_lattice, double dt_fluid, int cycles, float* f_vertex, float* f_lattice,
                                 void* stream)
{
    IbmArgs a;
    if (int rc = fill_ibm(&a, meshes, n_groups, cells_per_group, lattice, "npfem_ibm_forcing")) return rc;
    if (!x || !u_vertex || !u_lattice || !f_vertex || !f_lattice || !(dt_fluid > 0.0) || cycles < 0 || cycles > 1000)
        return set_error(NPFEM_ERR_INVALID_ARG, "npfem_ibm_forcing: null array, dt <= 0 or cycles outside 0..1000");
    DevGuard guard(meshes[0]->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t lat_bytes = (size_t)lattice->nx * lattice->ny * lattice->nz * 4 * sizeof(float);
    a.x = x;
    a.uvert = u_vertex;
    a.field = u_lattice;
    a.field2 = f_lattice;
    a.out = f_vertex;
    a.lat_out = f_lattice;
    a.lat_vec = (reinterpret_cast<uintptr_t>(f_lattice) & 15) == 0;
    a.dt = (float)dt_fluid;
    cudaError_t e = cudaSuccess;
    auto run = [&](int phase) {
        a.phase = phase;
        return a.total_verts > 0 ? launch_forcing(a, meshes, lattice->dx, s) : cudaGetLastError();
    };
    e = run(0);  // Step 0: f_0 = (U - u*(X)) / dt
    for (int l = 0; l < cycles && e == cudaSuccess; ++l) {
        e = cudaMemsetAsync(f_lattice, 0, lat_bytes, s);
        if (e == cudaSuccess) e = run(1);  // Step 1: spread f_l
        if (e == cudaSuccess) e = run(2);  // Steps 2-4: f_{l+1} = f_l + (U - u_l(X)) / dt
    }
    // f_imm: the spread of the final Lagrangian force
    if (e == cudaSuccess) e = cudaMemsetAsync(f_lattice, 0, lat_bytes, s);
    if (e == cudaSuccess) e = run(1);
    return e == cudaSuccess ? 0 : launch_err("npfem_ibm_forcing", e);
}
