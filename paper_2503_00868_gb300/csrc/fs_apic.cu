// fs_apic.cu -- APIC transfers between particles and the MAC grid, and the
// deformation of the Gaussians (arXiv 2503.00868, Sec. 3.2.2, Sec. 3.4.3).
//
// Per face component c (nodes at index * dx along axis c, (index + 1/2) * dx along
// the others), quadratic B-spline weights over 3 x 3 x 3 nodes:
//   P2G (Eq. eq::particle_map): (m v)_i = sum_p w_ip m_p [v_p,c + (C_p (x_i - x_p))_c],
//        v_i = (m v)_i / sum_p w_ip m_p (0 where no particle reaches);
//   G2P: v_p,c = sum_i w_ip u_c,i,  C_p[c][a] = 4/dx^2 sum_i w_ip u_c,i (x_i - x_p)_a;
//   advance: x_p += dt v_p (clamped), F_p = (I + dt C_p) F_p, A_p = F_p A0_p F_p^T.
// Particles are arrays of structures: x, v [p][3]; C, F, A0, A [p][3][3] row-major;
// m [p].
//
// P2G takes one of two ways. Few particles scatter with FP32 atomics (one thread per
// particle, 2 x 81 atomic adds), which bound the transfer (11.4 ms for 26.7 M
// particles at 256^3, 380 G adds/s). Otherwise they are first put in the order of the
// cells (a counting sort into 64-byte records, 0.9 ms), and a thread marches through
// a few dozen of them along a row of cells with the sums of the 36 nodes that a
// cell's particles reach in registers (4 x 3 x 3: one base node on the two axes
// across the component, two on its own), adding a column of nodes to the grid when
// the march has passed it: per cell about 33 vector atomics (momentum and mass
// together) in place of 162 scalar ones per particle, 1.6 ms. The summation order,
// and the last bits, vary from run to run in both. G2P gathers (one thread per
// particle, 81 node reads).
//
// The line between them: the ordering costs a dozen launches and passes over the
// cells (88 us at 48^3, 129 at 128^3, 390 at 256^3), the scatter grows with the
// particles and with their disorder. Ordered against scattered, 65536 particles: 88
// and 94-150 us at 48^3, 129 and 123-159 at 128^3, 420 and 350-365 at 256^3; 262144:
// 106 and 408-456, 180 and 230-435, 492 and 505-617. So: from P2G_SORT particles and
// one per 64 cells.
#include <algorithm>
#include <cmath>
#include <new>

#include "fs_internal.cuh"

namespace fs {
namespace {

constexpr int TH = 256;
constexpr int P2G_SORT = 1 << 16;  // particles from which P2G orders them by cell
constexpr int P2G_PER = 32;        // most particles per thread of the march

// A node coordinate of a component whose nodes lie `off` cells into them (0 or 1/2),
// clamped to [-8, lim]. One rounding, spelled out: the passes that order the particles
// and the march that relies on their order must agree on a particle's cell to the last
// bit, whatever a compiler would fuse in each of them.
__device__ __forceinline__ float node_coord(float x, float off, float inv_dx, float lim)
{
    return fminf(fmaxf(__fmaf_rn(x, inv_dx, -off), -8.f), lim);
}

struct Spline {
    int base[3];
    float w[3][3];
};

// weights of component c's nodes around position x (metres); the node coordinate
// is clamped to [-8, lim] first (a position that far out, or NaN, reaches no node
// and cannot overflow the integer base)
__device__ __forceinline__ Spline spline(const float x[3], int c, float inv_dx, float lim)
{
    Spline s;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float sc = node_coord(x[a], a == c ? 0.f : 0.5f, inv_dx, lim);
        const int b = (int)floorf(sc - 0.5f);
        const float f = sc - (float)b;
        s.base[a] = b;
        s.w[a][0] = 0.5f * (1.5f - f) * (1.5f - f);
        s.w[a][1] = 0.75f - (f - 1.f) * (f - 1.f);
        s.w[a][2] = 0.5f * (f - 0.5f) * (f - 0.5f);
    }
    return s;
}

// one of the three weights of one axis
__device__ __forceinline__ float spline_weight(float x, int a, int c, float inv_dx, float lim, int k)
{
    const float sc = node_coord(x, a == c ? 0.f : 0.5f, inv_dx, lim);
    const float f = sc - floorf(sc - 0.5f);
    if (k == 1) return 0.75f - (f - 1.f) * (f - 1.f);
    const float g = k == 0 ? 1.5f - f : f - 0.5f;
    return 0.5f * g * g;
}

__device__ __forceinline__ bool in_faces(const Layout &L, int c, int i, int j, int k)
{
    const int di = L.nx + (c == 0), dj = L.ny + (c == 1), dk = L.nz + (c == 2);
    return i >= 0 && j >= 0 && k >= 0 && i < di && j < dj && k < dk;
}

__global__ void __launch_bounds__(TH) k_p2g(int np, const float *__restrict__ x, const float *__restrict__ v,
                                            const float *__restrict__ C, const float *__restrict__ m, F3 mv,
                                            F3 ms, Layout L, float dx)
{
    const float inv_dx = 1.f / dx;
    const float lim = (float)(max(L.nx, max(L.ny, L.nz)) + 8);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const float xp[3] = {x[3 * p], x[3 * p + 1], x[3 * p + 2]};
        const float mp = m[p];
#pragma unroll 1
        for (int c = 0; c < 3; c++) {
            const Spline s = spline(xp, c, inv_dx, lim);
            const float vc = v[3 * p + c];
            const float c0 = C[9 * p + 3 * c], c1 = C[9 * p + 3 * c + 1], c2 = C[9 * p + 3 * c + 2];
            for (int kz = 0; kz < 3; kz++)
                for (int ky = 0; ky < 3; ky++)
#pragma unroll
                    for (int kx = 0; kx < 3; kx++) {
                        const int i = s.base[0] + kx, j = s.base[1] + ky, k = s.base[2] + kz;
                        if (!in_faces(L, c, i, j, k)) continue;
                        const float wt = s.w[0][kx] * s.w[1][ky] * s.w[2][kz] * mp;
                        const float dxv = ((float)i + (c == 0 ? 0.f : 0.5f)) * dx - xp[0];
                        const float dyv = ((float)j + (c == 1 ? 0.f : 0.5f)) * dx - xp[1];
                        const float dzv = ((float)k + (c == 2 ? 0.f : 0.5f)) * dx - xp[2];
                        const int t = (k * L.R + j) * L.P + i;
                        atomicAdd(mv.c[c] + t, wt * (vc + c0 * dxv + c1 * dyv + c2 * dzv));
                        atomicAdd(ms.c[c] + t, wt);
                    }
        }
    }
}

// u = mv / ms where ms > 0 (in place on mv); mass copy when wanted
__global__ void __launch_bounds__(TH) k_p2g_norm(F3 mv, CF3 ms, F3 mass_out, long long S)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < 3 * S;
         e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e / S);
        const long long t = e - c * S;
        const float mm = ms.c[c][t];
        mv.c[c][t] = mm > 0.f ? mv.c[c][t] / mm : 0.f;
        if (mass_out.c[c]) mass_out.c[c][t] = mm;
    }
}

// ---- P2G over cell-ordered particles -------------------------------------------------
// Cells are counted from -2 to n + 1 on each axis: a particle farther out reaches no
// node. Cell (ci, cj, ck) holds the particles whose base node is ci - 1 on the x axis
// of the components across it, and so on.
struct CellBox {
    int nx, ny, nz;  // cells of the box: those of the grid + 4 per axis
    __host__ __device__ long long count() const { return (long long)nx * ny * nz; }
};

// the particle's cell in the box, or -1
__device__ __forceinline__ int particle_cell(const float x[3], const CellBox &B, float inv_dx, float lim)
{
    int cell[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float sc = node_coord(x[a], 0.5f, inv_dx, lim);
        cell[a] = (int)floorf(sc - 0.5f) + 3;  // base + 1, from -2
    }
    if (cell[0] < 0 || cell[1] < 0 || cell[2] < 0 || cell[0] >= B.nx || cell[1] >= B.ny || cell[2] >= B.nz) return -1;
    return (cell[2] * B.ny + cell[1]) * B.nx + cell[0];
}

__global__ void __launch_bounds__(TH) k_p2g_count(int np, const float *__restrict__ x, CellBox B, float inv_dx, float lim,
                                                  unsigned *count)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const float xp[3] = {x[3 * p], x[3 * p + 1], x[3 * p + 2]};
        const int c = particle_cell(xp, B, inv_dx, lim);
        if (c >= 0) atomicAdd(count + c, 1u);
    }
}

// exclusive scan of n counts in place: per block of SC_ITEMS its sum, the sums' scan
// by one block, then each block's own scan from its offset
constexpr int SC_PER = 16, SC_ITEMS = TH * SC_PER;

__device__ __forceinline__ unsigned block_scan(unsigned v, unsigned *warp_tot, unsigned &total)  // exclusive
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    __syncthreads();
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    unsigned before = 0;
    total = 0;
    for (int k = 0; k < (int)blockDim.x / 32; k++) {
        if (k < w) before += warp_tot[k];
        total += warp_tot[k];
    }
    return before + incl - v;
}

__global__ void __launch_bounds__(TH) k_scan_sums(const unsigned *__restrict__ count, long long n, unsigned *sums)
{
    __shared__ unsigned warp_tot[TH / 32];
    const long long base = (long long)blockIdx.x * SC_ITEMS;
    unsigned v = 0, total;
    for (int k = 0; k < SC_PER; k++) {
        const long long t = base + k * TH + threadIdx.x;
        if (t < n) v += count[t];
    }
    block_scan(v, warp_tot, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_scan_top(unsigned *sums, int nb)
{
    __shared__ unsigned warp_tot[32];
    unsigned run = 0;
    for (int b0 = 0; b0 < nb; b0 += 1024) {
        const int b = b0 + threadIdx.x;
        const unsigned v = b < nb ? sums[b] : 0u;
        unsigned total;
        const unsigned e = block_scan(v, warp_tot, total);
        if (b < nb) sums[b] = run + e;
        run += total;
    }
}

__global__ void __launch_bounds__(TH) k_scan_apply(unsigned *count, long long n, const unsigned *__restrict__ sums)
{
    __shared__ unsigned warp_tot[TH / 32];
    __shared__ unsigned items[SC_ITEMS];
    const long long base = (long long)blockIdx.x * SC_ITEMS;
    for (int k = 0; k < SC_PER; k++) {
        const long long t = base + k * TH + threadIdx.x;
        items[k * TH + threadIdx.x] = t < n ? count[t] : 0u;
    }
    __syncthreads();
    unsigned v = 0, total;
    for (int k = 0; k < SC_PER; k++) v += items[threadIdx.x * SC_PER + k];
    unsigned run = sums[blockIdx.x] + block_scan(v, warp_tot, total);
    for (int k = 0; k < SC_PER; k++) {
        unsigned &e = items[threadIdx.x * SC_PER + k];
        const unsigned c = e;
        e = run;
        run += c;
    }
    __syncthreads();
    for (int k = 0; k < SC_PER; k++) {
        const long long t = base + k * TH + threadIdx.x;
        if (t < n) count[t] = items[k * TH + threadIdx.x];
    }
}

// W floats per lane of a warp's n particles, to and from global memory through `sm`
template <int W>
__device__ __forceinline__ void warp_load(const float *__restrict__ g, size_t first, int n, float *sm, float (&v)[W])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < W; k++) {
        const int e = k * 32 + lane;
        sm[e] = e < n * W ? g[first * W + e] : 0.f;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < W; k++) v[k] = sm[lane * W + k];
    __syncwarp();
}
template <int W>
__device__ __forceinline__ void warp_store(float *__restrict__ g, size_t first, int n, float *sm, const float (&v)[W])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < W; k++) sm[lane * W + k] = v[k];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < W; k++) {
        const int e = k * 32 + lane;
        if (e < n * W) g[first * W + e] = sm[e];
    }
    __syncwarp();
}

// A particle in the order of the cells, as the march reads it: {x, m}, then {v_c, row c
// of C} per component, 64 bytes.
struct P2gItem {
    float4 xm, vc[3];
};

// The particles cell by cell; afterwards next[c] is the end of cell c. Read warp by
// warp through shared memory (consecutive words), written as whole 64-byte records.
__global__ void __launch_bounds__(128) k_p2g_place(int np, const float *__restrict__ x, const float *__restrict__ v,
                                                   const float *__restrict__ C, const float *__restrict__ m, CellBox B,
                                                   float inv_dx, float lim, unsigned *next, P2gItem *items)
{
    __shared__ float stage[4][32 * 9];
    float *sm = stage[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const size_t first = (size_t)blockIdx.x * 128 + (threadIdx.x & ~31u);
    if (first >= (size_t)np) return;
    const int n = (int)min((size_t)32, (size_t)np - first);
    float xp[3], vp[3], Cp[9];
    warp_load<3>(x, first, n, sm, xp);
    warp_load<3>(v, first, n, sm, vp);
    warp_load<9>(C, first, n, sm, Cp);
    if (lane >= n) return;
    const int c = particle_cell(xp, B, inv_dx, lim);
    if (c < 0) return;
    P2gItem *o = items + atomicAdd(next + c, 1u);
    o->xm = make_float4(xp[0], xp[1], xp[2], m[first + lane]);
#pragma unroll
    for (int k = 0; k < 3; k++) o->vc[k] = make_float4(vp[k], Cp[3 * k], Cp[3 * k + 1], Cp[3 * k + 2]);
}

__device__ __forceinline__ void red_add2(float2 *p, float a, float b)
{
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}

// One component: a thread takes particles [e, e1) in cell order. The window of nodes
// moves along x with the particles' cell; acc[x][y][z] = {momentum, mass}. The next
// particle is loaded while this one is added. (inv_dx and lim as in the passes that
// ordered the particles.)
template <int c>
__device__ __forceinline__ void p2g_march(const P2gItem *__restrict__ items, unsigned e, unsigned e1, float2 *out,
                                          const Layout &L, float dx, float inv_dx, float lim)
{
    constexpr int NX = c == 0 ? 4 : 3, NY = c == 1 ? 4 : 3, NZ = c == 2 ? 4 : 3;
    float2 acc[NX][NY][NZ];
#pragma unroll
    for (int a = 0; a < NX; a++)
#pragma unroll
        for (int b = 0; b < NY; b++)
#pragma unroll
            for (int d = 0; d < NZ; d++) acc[a][b][d] = make_float2(0.f, 0.f);
    int w0 = 0, live = 0;  // first node of the window along x; columns that hold something
    int j0 = 0, k0 = 0;    // first nodes of the window along y and z
    // the first column to the grid, the others one to the left
    auto advance = [&]() {
#pragma unroll
        for (int b = 0; b < NY; b++)
#pragma unroll
            for (int d = 0; d < NZ; d++) {
                const int j = j0 + b, k = k0 + d;
                if ((acc[0][b][d].y != 0.f || acc[0][b][d].x != 0.f) && in_faces(L, c, w0, j, k))
                    red_add2(out + (k * L.R + j) * L.P + w0, acc[0][b][d].x, acc[0][b][d].y);
#pragma unroll
                for (int a = 0; a + 1 < NX; a++) acc[a][b][d] = acc[a + 1][b][d];
                acc[NX - 1][b][d] = make_float2(0.f, 0.f);
            }
        w0 += 1;
        live -= 1;
    };
    float4 nx = __ldg(&items[e].xm), nv = __ldg(&items[e].vc[c]);
#pragma unroll 1
    for (; e < e1; e++) {
        struct {
            float x[3], v, k[3], m;
        } q = {{nx.x, nx.y, nx.z}, nv.x, {nv.y, nv.z, nv.w}, nx.w};
        if (e + 1 < e1) {
            nx = __ldg(&items[e + 1].xm);
            nv = __ldg(&items[e + 1].vc[c]);
        }
        const Spline s = spline(q.x, c, inv_dx, lim);
        if (!isfinite(q.v + q.k[0] + q.k[1] + q.k[2] + q.m)) {  // to its own 27 nodes only: zero weights would spread it
#pragma unroll 1
            for (int n = 0; n < 27; n++) {
                const int qx = n % 3, qy = (n / 3) % 3, qz = n / 9;
                const int i = s.base[0] + qx, j = s.base[1] + qy, k = s.base[2] + qz;
                if (!in_faces(L, c, i, j, k)) continue;
                const float wt = spline_weight(q.x[0], 0, c, inv_dx, lim, qx) * spline_weight(q.x[1], 1, c, inv_dx, lim, qy) *
                                 spline_weight(q.x[2], 2, c, inv_dx, lim, qz) * q.m;
                const float dxv = ((float)i + (c == 0 ? 0.f : 0.5f)) * dx - q.x[0];
                const float dyv = ((float)j + (c == 1 ? 0.f : 0.5f)) * dx - q.x[1];
                const float dzv = ((float)k + (c == 2 ? 0.f : 0.5f)) * dx - q.x[2];
                red_add2(out + (k * L.R + j) * L.P + i, wt * (q.v + q.k[0] * dxv + q.k[1] * dyv + q.k[2] * dzv), wt);
            }
            continue;
        }
        // first nodes of this particle's window: its cell less one on each axis
        int lo[3];
#pragma unroll
        for (int a = 0; a < 3; a++)
            lo[a] = a == c ? (int)floorf(node_coord(q.x[a], 0.5f, inv_dx, lim) - 0.5f) : s.base[a];
        if (lo[1] != j0 || lo[2] != k0) {  // another row of cells
            while (live > 0) advance();
            j0 = lo[1];
            k0 = lo[2];
        }
        while (live > 0 && w0 < lo[0]) advance();
        w0 = lo[0];
        live = NX;
        float wx[NX], wy[NY], wz[NZ], ax[NX], by[NY], bz[NZ];
        // weights in the window, zero where the own axis's base leaves a node out
        auto spread = [&](int a, float *w, int n) {
            const int o = n == 4 ? s.base[a] - lo[a] : 0;
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (k < n) {
                    const float at = k < 3 ? s.w[a][k < 3 ? k : 0] : 0.f, before = k > 0 ? s.w[a][k - 1] : 0.f;
                    w[k] = o == 0 ? at : before;
                }
        };
        spread(0, wx, NX);
        spread(1, wy, NY);
        spread(2, wz, NZ);
#pragma unroll
        for (int a = 0; a < NX; a++) ax[a] = q.v + q.k[0] * (((float)(lo[0] + a) + (c == 0 ? 0.f : 0.5f)) * dx - q.x[0]);
#pragma unroll
        for (int b = 0; b < NY; b++) by[b] = q.k[1] * (((float)(lo[1] + b) + (c == 1 ? 0.f : 0.5f)) * dx - q.x[1]);
#pragma unroll
        for (int d = 0; d < NZ; d++) {
            bz[d] = q.k[2] * (((float)(lo[2] + d) + (c == 2 ? 0.f : 0.5f)) * dx - q.x[2]);
            wz[d] *= q.m;
        }
#pragma unroll
        for (int a = 0; a < NX; a++)
#pragma unroll
            for (int b = 0; b < NY; b++) {
                const float wab = wx[a] * wy[b], vab = ax[a] + by[b];
#pragma unroll
                for (int d = 0; d < NZ; d++) {
                    const float wt = wab * wz[d];
                    acc[a][b][d].x += wt * (vab + bz[d]);
                    acc[a][b][d].y += wt;
                }
            }
    }
    while (live > 0) advance();
}

// blockIdx.y = component; the ordered particles end at *total (those that reach no
// node are not among them)
__global__ void __launch_bounds__(128) k_p2g_rows(const P2gItem *__restrict__ items, const unsigned *__restrict__ total,
                                                  int per, float2 *s0, float2 *s1, float2 *s2, Layout L, float dx,
                                                  float inv_dx, float lim)
{
    const unsigned n = *total;
    const unsigned long long e = (unsigned long long)(blockIdx.x * 128u + threadIdx.x) * (unsigned)per;
    if (e >= n) return;
    const unsigned e1 = (unsigned)min(e + per, (unsigned long long)n);
    if (blockIdx.y == 0)
        p2g_march<0>(items, (unsigned)e, e1, s0, L, dx, inv_dx, lim);
    else if (blockIdx.y == 1)
        p2g_march<1>(items, (unsigned)e, e1, s1, L, dx, inv_dx, lim);
    else
        p2g_march<2>(items, (unsigned)e, e1, s2, L, dx, inv_dx, lim);
}

// u = momentum / mass where mass > 0; mass copy when wanted
__global__ void __launch_bounds__(TH) k_p2g_norm2(const float2 *__restrict__ s0, const float2 *__restrict__ s1,
                                                  const float2 *__restrict__ s2, F3 u, F3 mass_out, int S)
{
    const int c = blockIdx.y;
    const float2 *s = c == 0 ? s0 : (c == 1 ? s1 : s2);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < S; t += gridDim.x * blockDim.x) {
        const float2 e = s[t];
        u.c[c][t] = e.y > 0.f ? e.x / e.y : 0.f;
        if (mass_out.c[c]) mass_out.c[c][t] = e.y;
    }
}

// ---- G2P ---------------------------------------------------------------------------
// A thread per particle. The particles' 3 and 9 floats pass through shared memory,
// warp by warp, so that global memory sees consecutive words (a thread reading its
// own 36-byte record makes every access touch nine lines); a row of three nodes is
// summed before its y and z weights apply. The latency of the gathers bounds it: at
// 128^3 with 3.3 M particles (181 us) most stalls wait for them, with L1 at 64 % of its
// rate, instructions on 60 % of the cycles and DRAM at 47 %.
constexpr int G2P_TH = 128;

__global__ void __launch_bounds__(G2P_TH) k_g2p(int np, float *x, float *v, float *C, float *F,
                                                const float *__restrict__ A0, float *A, CF3 u, Layout L, float dx,
                                                float dt, int advance, float lo, float hi)
{
    __shared__ float stage[G2P_TH / 32][32 * 9];
    float *sm = stage[threadIdx.x >> 5];
    const size_t first = (size_t)blockIdx.x * G2P_TH + (threadIdx.x & ~31u);  // the warp's particles
    if (first >= (size_t)np) return;
    const int n = (int)min((size_t)32, (size_t)np - first);
    const float inv_dx = 1.f / dx;
    const float cs = 4.f * inv_dx * inv_dx;
    const float lim = (float)(max(L.nx, max(L.ny, L.nz)) + 8);
    float xp[3], vp[3], Cp[9];
    warp_load<3>(x, first, n, sm, xp);
    // a particle whose position is not finite reaches no node: its offsets count as
    // finite ones, since each is multiplied by the zero that stands for such a node
    const bool placed = isfinite(xp[0]) && isfinite(xp[1]) && isfinite(xp[2]);
    const float xo[3] = {placed ? xp[0] : 0.f, placed ? xp[1] : 0.f, placed ? xp[2] : 0.f};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const Spline s = spline(xp, c, inv_dx, lim);
        const float *uc = u.c[c];
        float dxv[3];
#pragma unroll
        for (int q = 0; q < 3; q++) dxv[q] = ((float)(s.base[0] + q) + (c == 0 ? 0.f : 0.5f)) * dx - xo[0];
        const bool inside = in_faces(L, c, s.base[0], s.base[1], s.base[2]) &&
                            in_faces(L, c, s.base[0] + 2, s.base[1] + 2, s.base[2] + 2);
        const int t0 = (s.base[2] * L.R + s.base[1]) * L.P + s.base[0];
        float vc = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f;
        auto rows = [&](auto node) {
#pragma unroll
            for (int kz = 0; kz < 3; kz++)
#pragma unroll
                for (int ky = 0; ky < 3; ky++) {
                    const float a0 = s.w[0][0] * node(0, ky, kz), a1 = s.w[0][1] * node(1, ky, kz),
                                a2 = s.w[0][2] * node(2, ky, kz);
                    const float r0 = a0 + a1 + a2, r1 = a0 * dxv[0] + a1 * dxv[1] + a2 * dxv[2];
                    const float wyz = s.w[1][ky] * s.w[2][kz];
                    const float dyv = ((float)(s.base[1] + ky) + (c == 1 ? 0.f : 0.5f)) * dx - xo[1];
                    const float dzv = ((float)(s.base[2] + kz) + (c == 2 ? 0.f : 0.5f)) * dx - xo[2];
                    const float w = wyz * r0;
                    vc += w;
                    g0 += wyz * r1;
                    g1 += w * dyv;
                    g2 += w * dzv;
                }
        };
        if (inside)
            rows([&](int i, int j, int k) { return __ldg(uc + t0 + (k * L.R + j) * L.P + i); });
        else
            rows([&](int i, int j, int k) {
                return in_faces(L, c, s.base[0] + i, s.base[1] + j, s.base[2] + k)
                           ? __ldg(uc + t0 + (k * L.R + j) * L.P + i)
                           : 0.f;
            });
        vp[c] = vc;
        Cp[3 * c] = cs * g0;
        Cp[3 * c + 1] = cs * g1;
        Cp[3 * c + 2] = cs * g2;
    }
    warp_store<3>(v, first, n, sm, vp);
    warp_store<9>(C, first, n, sm, Cp);
    if (!advance) return;
    float xn[3];
#pragma unroll
    for (int a = 0; a < 3; a++) xn[a] = fminf(fmaxf(xp[a] + dt * vp[a], lo), hi);
    warp_store<3>(x, first, n, sm, xn);
    if (!F) return;
    float Fo[9], Fn[9];
    warp_load<9>(F, first, n, sm, Fo);
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int s = 0; s < 3; s++)
            Fn[3 * r + s] = Fo[3 * r + s] +
                            dt * (Cp[3 * r] * Fo[s] + Cp[3 * r + 1] * Fo[3 + s] + Cp[3 * r + 2] * Fo[6 + s]);
    warp_store<9>(F, first, n, sm, Fn);
    if (!A0 || !A) return;
    float T[9], B[9];
    warp_load<9>(A0, first, n, sm, Fo);
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int s = 0; s < 3; s++) T[3 * r + s] = Fn[3 * r] * Fo[s] + Fn[3 * r + 1] * Fo[3 + s] + Fn[3 * r + 2] * Fo[6 + s];
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int s = 0; s < 3; s++) B[3 * r + s] = T[3 * r] * Fn[3 * s] + T[3 * r + 1] * Fn[3 * s + 1] + T[3 * r + 2] * Fn[3 * s + 2];
    warp_store<9>(A, first, n, sm, B);
}

}  // namespace

// Workspace of the cell-ordered P2G, kept on the context and grown on demand: 64 bytes
// per particle, with room for an eighth more than the largest call so far (where that
// can be had), so that a count that rises from call to call does not free and allocate
// it, and wait for the device, each time.
struct ApicState {
    unsigned *ends = nullptr, *sums = nullptr;
    P2gItem *items = nullptr;
    long long cap = 0;  // of items
};

void apic_free(fs_ctx *c)
{
    ApicState *s = static_cast<ApicState *>(c->apic);
    if (!s) return;
    cudaFree(s->ends);
    cudaFree(s->sums);
    cudaFree(s->items);
    delete s;
    c->apic = nullptr;
}

// The workspace for np particles and a box of n cells; false when it cannot be had
// (the scatter needs none).
static bool apic_workspace(fs_ctx *c, long long np, long long n)
{
    ApicState *s = static_cast<ApicState *>(c->apic);
    if (!s) {
        s = new (std::nothrow) ApicState();
        if (!s) return false;
        c->apic = s;
    }
    auto have = [](auto **p, long long count) {
        if (*p) return true;
        if (cudaMalloc((void **)p, (size_t)count * sizeof(**p)) == cudaSuccess) return true;
        cudaGetLastError();
        *p = nullptr;
        return false;
    };
    if (!have(&s->ends, n) || !have(&s->sums, (n + SC_ITEMS - 1) / SC_ITEMS)) return false;
    if (np <= s->cap) return true;
    cudaFree(s->items);
    s->items = nullptr;
    s->cap = 0;
    for (long long cap : {np + np / 8, np})
        if (have(&s->items, cap)) {
            s->cap = cap;
            return true;
        }
    return false;
}

int launch_p2g(fs_ctx *c, int np, const float *x, const float *v, const float *C, const float *m, F3 u, F3 mass)
{
    const Layout &L = c->L;
    const float dx = (float)c->prm.dx;
    const CellBox B{L.nx + 4, L.ny + 4, L.nz + 4};
    const long long n = B.count();
    // momentum and mass side by side: a face-space vector of the viscosity solve per
    // component (no solve runs meanwhile, and each starts its vectors anew)
    float2 *s2[3] = {reinterpret_cast<float2 *>(c->vr), reinterpret_cast<float2 *>(c->vp[0]),
                     reinterpret_cast<float2 *>(c->vp[1])};
    if (np >= P2G_SORT && np >= n / 64 && apic_workspace(c, np, n)) {
        const ApicState *w = static_cast<const ApicState *>(c->apic);
        const float inv_dx = 1.f / dx, lim = (float)(std::max(L.nx, std::max(L.ny, L.nz)) + 8);
        const int gp = grid_blocks(c, np, TH), nb = (int)((n + SC_ITEMS - 1) / SC_ITEMS);
        FS_CUDA(cudaMemsetAsync(w->ends, 0, (size_t)n * sizeof(unsigned), c->stream));
        for (float2 *p : s2) FS_CUDA(cudaMemsetAsync(p, 0, (size_t)L.S * sizeof(float2), c->stream));
        k_p2g_count<<<gp, TH, 0, c->stream>>>(np, x, B, inv_dx, lim, w->ends);
        k_scan_sums<<<nb, TH, 0, c->stream>>>(w->ends, n, w->sums);
        k_scan_top<<<1, 1024, 0, c->stream>>>(w->sums, nb);
        k_scan_apply<<<nb, TH, 0, c->stream>>>(w->ends, n, w->sums);
        k_p2g_place<<<(np - 1) / 128 + 1, 128, 0, c->stream>>>(np, x, v, C, m, B, inv_dx, lim, w->ends, w->items);
        // particles per thread: enough threads for the GPU first, then long marches
        const int per = std::max(4, std::min(P2G_PER, np / (c->num_sms * 256)));
        const int gr = (int)(((long long)np + 128LL * per - 1) / (128LL * per));
        k_p2g_rows<<<dim3(gr, 3), 128, 0, c->stream>>>(w->items, w->ends + n - 1, per, s2[0], s2[1], s2[2], L, dx,
                                                     inv_dx, lim);
        k_p2g_norm2<<<dim3(grid_blocks(c, L.S, TH), 3), TH, 0, c->stream>>>(s2[0], s2[1], s2[2], u, mass, L.S);
        c->n_launches += 7;
        FS_CUDA(cudaGetLastError());
        return FS_OK;
    }
    const size_t sb = (size_t)L.S * sizeof(float);
    F3 ms{{c->fg[0], c->fg[1], c->fg[2]}};
    for (int k = 0; k < 3; k++) {
        FS_CUDA(cudaMemsetAsync(u.c[k], 0, sb, c->stream));
        FS_CUDA(cudaMemsetAsync(ms.c[k], 0, sb, c->stream));
    }
    if (np > 0) {
        k_p2g<<<grid_blocks(c, np, TH), TH, 0, c->stream>>>(np, x, v, C, m, u, ms, L, dx);
        c->n_launches += 1;
    }
    CF3 msc{{ms.c[0], ms.c[1], ms.c[2]}};
    k_p2g_norm<<<grid_blocks(c, 3LL * L.S, TH), TH, 0, c->stream>>>(u, msc, mass, (long long)L.S);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    return FS_OK;
}

int launch_g2p(fs_ctx *c, int np, float *x, float *v, float *C, float *F, const float *A0, float *A, CF3 u,
               double dt, int advance, double lo, double hi)
{
    if (np <= 0) return FS_OK;
    k_g2p<<<(np - 1) / G2P_TH + 1, G2P_TH, 0, c->stream>>>(np, x, v, C, F, A0, A, u, c->L, (float)c->prm.dx, (float)dt,
                                                           advance, (float)lo, (float)hi);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    return FS_OK;
}

}  // namespace fs
