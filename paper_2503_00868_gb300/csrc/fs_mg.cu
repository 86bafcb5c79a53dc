// fs_mg.cu -- geometric multigrid V-cycle as the preconditioner of the pressure
// CG (z = M r for the 7-point operator of Sec. 3.2.2's projection). The paper
// solves the projection with a fitted recurrent network (Sec. 3.4.1); this
// preconditioner is the library's own choice for speed, and the solve still
// stops at the same tolerance on the same operator, so it changes the number of
// iterations, not what the projection computes.
//
// Levels. Level 0 is the cell space of the context (flags CF_LIQ, CF_AIR and the
// neighbour count CF_D). A coarse cell covers 2 x 2 x 2 cells of the level above
// (cells beyond an odd edge count as solid): it is air (a Dirichlet cell, p = 0)
// when any child is air, else liquid when any child is liquid, else solid. Each
// coarse level stores the same flag bits, with its own neighbour counts, in a
// dense array with a solid halo (a plane and a row on each side, 4 elements
// before each row, the row pitch a multiple of 4). The operator on level l is the
// same 7-point stencil rediscretised on cells of size 2^l dx, i.e. scaled by 4^-l.
//
// V-cycle on level l for A_l e = r: two damped Jacobi sweeps from e = 0
// (omega = 0.8), the residual, restriction (the transpose of cell-centred
// trilinear prolongation, divided by 8), the V-cycle on level l + 1, prolongation
// of its correction (weights 3/4 and 1/4 per axis), and two more sweeps; one
// before and one after on a face volume's level 0, where the mass term of the
// Helmholtz operator makes the smoothing strong enough that the second costs more
// than the iterations it saves. The
// coarsest level (small enough for shared memory) takes a fixed number of sweeps. Every step is linear in r with symmetric smoothing and restriction
// proportional to the transposed prolongation, so M is symmetric, as CG needs.
//
// The sweeps, the residual and the transfers take four elements per thread and
// walk a list of a level's quads that hold an unknown (built with the hierarchy).
// Every array a V-cycle writes is written only on those quads (with zeros on
// their other elements) and is zero on every other quad: the work arrays are
// zeroed when the hierarchy is built, and the level-0 output (the solver's z) is
// a context buffer that is zeroed with each new mask and that every writer
// leaves zero off the unknowns. So a stencil at the edge of the liquid reads
// zeros, and the solver's operator apply reads z = 0 off the unknowns.
//
// The same V-cycle preconditions the implicit viscosity solve, one velocity
// component at a time: each face volume is a box of unknown faces (FF_FLUID),
// prescribed faces (FF_FIXED, Dirichlet) and mirror faces (Neumann), whose flag
// bits coincide with the cell bits used here (FF_FLUID = CF_LIQ, FF_FIXED =
// CF_AIR, FF_N = CF_D), and the operator gains the mass term: A_l = m I +
// 4^-l cc L_l with m = 1 (m = 0 for the pressure).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "fs_internal.cuh"

namespace fs {

constexpr int MG_MAX_LEVELS = 16;
constexpr int MG_COARSE_CELLS = 3072;  // padded cells of a level solved in shared memory
constexpr int MG_COARSE_SWEEPS = 30;
constexpr float MG_OMEGA = 0.8f;

// A level's array is `rows` rows of `sy` elements, `rpp` rows per plane; element
// e of row w is cell (e - ioff, w % rpp - joff, w / rpp - koff). The set-up
// kernels walk rows (a warp along a row), so they divide no element index.
struct MgGrid {
    int nx, ny, nz;    // cells of the level
    int sy, sz;        // element strides of a row and a plane
    int origin;        // element of cell (0, 0, 0)
    int n;             // elements of the whole array (halo, padding and guards included)
    int rows, rpp, ioff, joff, koff;
    __host__ __device__ int idx(int i, int j, int k) const { return origin + k * sz + j * sy + i; }
};

#define MG_FOR_ROWS(g)                                                                                   \
    for (int row = blockIdx.x * blockDim.y + threadIdx.y; row < (g).rows; row += gridDim.x * blockDim.y) \
        for (int e = threadIdx.x; e < (g).sy; e += blockDim.x)

struct MgLevel {
    MgGrid g;
    float scale = 1.f;  // 4^-l times the operator's coefficient
    float mass = 0.f;   // identity term (1 for the Helmholtz operator)
    uint8_t *fl = nullptr;
    float *r = nullptr, *a = nullptr, *b = nullptr;  // levels >= 1 (of the set's arrays): right-hand side, result, field
};

// The levels of one volume (the cell space, or one face component).
struct MgState {
    int nlev = 0;
    MgLevel lev[MG_MAX_LEVELS];
    long long epoch = -1;  // mask epoch the hierarchy was built for
    float coef = 0.f;      // operator coefficient it was built for
    int lb = 0;            // first level of the single-block launch
};

// The volumes of one level: each volume's grid and the first element of its array
// in the level's arrays, which hold the volumes one after another.
struct MgSpace {
    MgGrid g[3];
    int base[3];
    int nv;
};

// Volumes whose V-cycles run together, launch by launch: the cell space alone, or
// the three face components (one by one when one of them is its own coarsest
// level). Level 0 lies in the arrays of the whole cell or face space; the arrays of
// a level below belong to the set. The first levels take one launch per step over
// lists: the active quads (those holding an unknown) and, below level 0, the active
// restriction pairs, both counted in the level's arrays, volume after volume. The
// levels from `lf` on take the tile kernels of fs_mg_coarse.cuh.
struct MgSetLevel {
    MgSpace sp;
    uint8_t *fl = nullptr;
    float *r = nullptr, *a = nullptr, *b = nullptr, *c = nullptr;
    int *ql = nullptr, *pl = nullptr;
    int nq = 0, np = 0;
};
struct MgSet {
    int nv = 0, lf = 1;
    MgState *s[3] = {nullptr, nullptr, nullptr};
    MgSetLevel lev[MG_MAX_LEVELS];
    uint8_t *blob = nullptr;  // flags and lists of the single-block levels, volume after volume
    bool one = false;         // one smoothing sweep each side on level 0 (the face volumes)
    bool shared0 = false;     // level 0's list belongs to the context
    long long calls = 0;      // applies so far (profiling samples every prof_period-th)
    // algorithmic bytes of the level-0 kernels, in the order of K_MG0_SMOOTH2 ..
    // K_MG0_SMOOTH_Z (counted when first profiled; negative before)
    double by0[6] = {-1, 0, 0, 0, 0, 0};
};

// The pressure hierarchy and one per face volume (viscosity). The work arrays of
// level 0 belong here: one pair of cell-space length, one of face-space length.
struct MgAll {
    MgState cell, face[3];
    MgSet cset, fset[3];
    int nfset = 0;
    float *cb = nullptr, *cc = nullptr, *fb = nullptr, *fc = nullptr;
};

namespace {

constexpr int TH = 256;
const dim3 RT(32, 8);  // a warp along a row, 8 rows per block

__device__ __forceinline__ bool liq(uint8_t f) { return f & CF_LIQ; }

// A_l e at a liquid cell, without the scale
__device__ __forceinline__ float lap(const float *__restrict__ e, int t, uint8_t f, const MgGrid &g)
{
    return (float)(f & CF_D) * e[t] - ((e[t - 1] + e[t + 1]) + (e[t - g.sy] + e[t + g.sy]) + (e[t - g.sz] + e[t + g.sz]));
}

// omega / (m + scale d), zero where the diagonal vanishes
__device__ __forceinline__ float wtab_entry(float scale, float m, int d)
{
    const float dg = m + scale * (float)d;
    return dg > 0.f ? MG_OMEGA / dg : 0.f;
}

// the table for d = 0..7 in shared memory
__device__ __forceinline__ void fill_wtab(float *wt, float scale, float m)
{
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    if (tid < 8) wt[tid] = wtab_entry(scale, m, tid);
    __syncthreads();
}

// ---- four elements per thread -------------------------------------------------
// Every level but the coarsest has a row pitch, plane stride and origin that are
// multiples of 4 (level 0 by the context's layout, a coarse level by its 4-element
// x halo), so a quad of 4 consecutive elements never crosses a row and its
// float4 / uchar4 loads are aligned. A quad without an unknown is skipped; a quad
// with one is read whole (its row is interior, so every neighbour load is inside
// the array) and written whole, with zeros on the elements that are not unknowns.

__device__ __forceinline__ uchar4 ldf4(const uint8_t *__restrict__ p, int t)
{
    return __ldg(reinterpret_cast<const uchar4 *>(p + t));
}
__device__ __forceinline__ bool any_liq(uchar4 f) { return ((f.x | f.y | f.z | f.w) & CF_LIQ) != 0; }

// e_out on one element from e_in: c (centre), the sum of its six neighbours nb
__device__ __forceinline__ float sweep1(uint8_t f, float c, float nb, float rv, const float *wt, float scale, float m)
{
    return liq(f) ? c + wt[f & CF_D] * (rv - m * c - scale * ((float)(f & CF_D) * c - nb)) : 0.f;
}

// The kernels below walk a level's list of active quads (those holding an
// unknown, built with the hierarchy): no flag load stands between a thread and its
// data loads, and the quads without an unknown cost nothing.

__device__ __forceinline__ float4 ldv4(const float *p, int t) { return ldd4(p + t); }
__device__ __forceinline__ float ldv1(const float *p, int t) { return ldd1(p + t); }

// one damped Jacobi sweep on quad q: eout from ein; returns r.eout over the quad
__device__ __forceinline__ float smooth_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r,
                                          const float *ein, float *eout, const float *wt, float scale, float m, int q)
{
    const int t = q << 2;
    const uchar4 f = ldf4(fl, t);
    const float4 c = ldv4(ein, t), rv = ldv4(r, t);
    const float4 dn = ldv4(ein, t - g.sy), up = ldv4(ein, t + g.sy);
    const float4 bk = ldv4(ein, t - g.sz), fw = ldv4(ein, t + g.sz);
    const float lf = ldv1(ein, t - 1), rt = ldv1(ein, t + 4);
    float4 v;
    v.x = sweep1(f.x, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x, wt, scale, m);
    v.y = sweep1(f.y, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y, wt, scale, m);
    v.z = sweep1(f.z, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z, wt, scale, m);
    v.w = sweep1(f.w, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w, wt, scale, m);
    *reinterpret_cast<float4 *>(eout + t) = v;
    return rv.x * v.x + rv.y * v.y + rv.z * v.z + rv.w * v.w;
}

// res = r - A e on quad q
__device__ __forceinline__ void resid_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r,
                                        const float *ev, float *res, float scale, float m, int q)
{
    const int t = q << 2;
    const uchar4 f = ldf4(fl, t);
    const float4 c = ldv4(ev, t), rv = ldv4(r, t);
    const float4 dn = ldv4(ev, t - g.sy), up = ldv4(ev, t + g.sy);
    const float4 bk = ldv4(ev, t - g.sz), fw = ldv4(ev, t + g.sz);
    const float lf = ldv1(ev, t - 1), rt = ldv1(ev, t + 4);
    auto one = [&](uint8_t fe, float ce, float nb, float re) {
        return liq(fe) ? re - m * ce - scale * ((float)(fe & CF_D) * ce - nb) : 0.f;
    };
    float4 v;
    v.x = one(f.x, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x);
    v.y = one(f.y, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y);
    v.z = one(f.z, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z);
    v.w = one(f.w, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w);
    *reinterpret_cast<float4 *>(res + t) = v;
}

// the first two sweeps from e = 0 on quad q: e1 = omega D^-1 r on the fly, then one sweep
__device__ __forceinline__ void smooth2_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r, float *eo,
                                          const float *wt, float scale, float m, int q)
{
    const int t = q << 2;
    const uchar4 f = ldf4(fl, t);
    auto e1q = [&](int u) {  // e1 on the quad at u
        const uchar4 fu = ldf4(fl, u);
        const float4 ru = ldv4(r, u);
        return make_float4(liq(fu.x) ? wt[fu.x & CF_D] * ru.x : 0.f, liq(fu.y) ? wt[fu.y & CF_D] * ru.y : 0.f,
                           liq(fu.z) ? wt[fu.z & CF_D] * ru.z : 0.f, liq(fu.w) ? wt[fu.w & CF_D] * ru.w : 0.f);
    };
    auto e1s = [&](int u) {
        const uint8_t fu = fl[u];
        return liq(fu) ? wt[fu & CF_D] * ldv1(r, u) : 0.f;
    };
    const float4 c = e1q(t), rv = ldv4(r, t);
    const float4 dn = e1q(t - g.sy), up = e1q(t + g.sy), bk = e1q(t - g.sz), fw = e1q(t + g.sz);
    const float lf = e1s(t - 1), rt = e1s(t + 4);
    float4 v;
    v.x = sweep1(f.x, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x, wt, scale, m);
    v.y = sweep1(f.y, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y, wt, scale, m);
    v.z = sweep1(f.z, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z, wt, scale, m);
    v.w = sweep1(f.w, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w, wt, scale, m);
    *reinterpret_cast<float4 *>(eo + t) = v;
}

// e_fine += P e_coarse on the unknowns of an active quad q (in place). The quad's
// elements i .. i + 3 (i a multiple of 4) take their x samples from coarse
// I0 - 1 .. I0 + 2 (I0 = i / 2); indices past the coarse halo are clamped to it
// (a sample that only padding elements use).
__device__ __forceinline__ void prolong_q(const MgGrid &gf, const uint8_t *__restrict__ fl, float *ef,
                                          const MgGrid &gc, const float *ec, int q)
{
    const int qrow = gf.sy >> 2;
    const int t = q << 2;
    const uchar4 f = ldf4(fl, t);
    const int row = q / qrow, e = (q - row * qrow) << 2;
    const int i = e - gf.ioff, j = row % gf.rpp - gf.joff, k = row / gf.rpp - gf.koff;
    const int I0 = i >> 1, J = j >> 1, K = k >> 1;
    const int J2 = (j & 1) ? J + 1 : J - 1, K2 = (k & 1) ? K + 1 : K - 1;
    const int xs[4] = {max(I0 - 1, -1), I0, min(I0 + 1, gc.nx), min(I0 + 2, gc.nx)};
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    const int jj[2] = {J, J2}, kk[2] = {K, K2};
    const float wy[2] = {0.75f, 0.25f};
#pragma unroll
    for (int b = 0; b < 2; b++)
#pragma unroll
        for (int a = 0; a < 2; a++) {
            const int base = gc.idx(0, jj[a], kk[b]);
            const float w = wy[a] * wy[b];
            const float cm = ldv1(ec, base + xs[0]), c0 = ldv1(ec, base + xs[1]);
            const float c1 = ldv1(ec, base + xs[2]), c2 = ldv1(ec, base + xs[3]);
            s0 += w * (0.75f * c0 + 0.25f * cm);
            s1 += w * (0.75f * c0 + 0.25f * c1);
            s2 += w * (0.75f * c1 + 0.25f * c0);
            s3 += w * (0.75f * c1 + 0.25f * c2);
        }
    float4 v = ldv4(ef, t);
    if (liq(f.x)) v.x += s0;
    if (liq(f.y)) v.y += s1;
    if (liq(f.z)) v.z += s2;
    if (liq(f.w)) v.w += s3;
    *reinterpret_cast<float4 *>(ef + t) = v;
}

// Restriction of an active pair of the coarse level: t0 is the element of coarse
// cell (2m, J, K), and the pair (2m, 2m + 1) holds at least one unknown. Per fine
// row of the 4 x 4 window it reads the aligned quad 4m .. 4m + 3 and the scalars
// at 4m - 1 and 4m + 4 (excluded at or past nx, where the next row begins), and
// forms both cells' x weights from them.
__device__ __forceinline__ void restrict_pair(const MgGrid &gf, const float *res, const MgGrid &gc,
                                              const uint8_t *__restrict__ flc, float *rc, int t0)
{
    const float w[4] = {0.25f, 0.75f, 0.75f, 0.25f};
    const int rel = t0 - gc.origin;
    const int K = rel / gc.sz, J = (rel - K * gc.sz) / gc.sy, I0 = rel - K * gc.sz - J * gc.sy;
    const int m = I0 >> 1;
    const bool l0 = liq(flc[t0]), l1 = I0 + 1 < gc.nx && liq(flc[t0 + 1]);
    float a0 = 0.f, a1 = 0.f;
    // A row off the grid counts nothing: its weight is zero and the pair's own row
    // is read in its place, so that no branch stands between the 16 rows' loads
    // (with a skip per row each waited for the one before it: 12 us for the 64^3
    // level of the three face volumes of 128^3, and the sweeps 4).
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const int k = 2 * K - 1 + c;
        const bool kin = k >= 0 && k < gf.nz;
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const int j = 2 * J - 1 + b;
            const bool in = kin && j >= 0 && j < gf.ny;
            const int row = gf.idx(0, in ? j : 2 * J, in ? k : 2 * K) + 4 * m;  // a multiple of 4
            const float4 qd = ldv4(res, row);
            const float lf = ldv1(res, row - 1), rt = ldv1(res, row + 4);
            const float wyz = in ? w[c] * w[b] : 0.f;
            // coarse 2m: fine 4m - 1 .. 4m + 2; coarse 2m + 1: fine 4m + 1 .. 4m + 4
            a0 += wyz * (0.25f * (m > 0 ? lf : 0.f) + 0.75f * qd.x + 0.75f * qd.y + 0.25f * qd.z);
            a1 += wyz * (0.25f * qd.y + 0.75f * qd.z + 0.75f * qd.w + 0.25f * (4 * m + 4 < gf.nx ? rt : 0.f));
        }
    }
    if (l0) rc[t0] = 0.125f * a0;
    if (l1) rc[t0 + 1] = 0.125f * a1;
}

// one damped Jacobi sweep from zero and the residual it leaves, on quad q:
// eb = e1 = omega D^-1 r at the quad, res = r - A e1 (e1 at the neighbours formed
// on the fly)
__device__ __forceinline__ void pre1_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r, float *eb,
                                       float *res, const float *wt, float scale, float m, int q)
{
    const int t = q << 2;
    const uchar4 f = ldf4(fl, t);
    auto e1q = [&](int u) {  // e1 on the quad at u
        const uchar4 fu = ldf4(fl, u);
        const float4 ru = ldv4(r, u);
        return make_float4(liq(fu.x) ? wt[fu.x & CF_D] * ru.x : 0.f, liq(fu.y) ? wt[fu.y & CF_D] * ru.y : 0.f,
                           liq(fu.z) ? wt[fu.z & CF_D] * ru.z : 0.f, liq(fu.w) ? wt[fu.w & CF_D] * ru.w : 0.f);
    };
    auto e1s = [&](int u) {
        const uint8_t fu = fl[u];
        return liq(fu) ? wt[fu & CF_D] * ldv1(r, u) : 0.f;
    };
    const float4 c = e1q(t), rv = ldv4(r, t);
    const float4 dn = e1q(t - g.sy), up = e1q(t + g.sy), bk = e1q(t - g.sz), fw = e1q(t + g.sz);
    const float lf = e1s(t - 1), rt = e1s(t + 4);
    auto one = [&](uint8_t fe, float ce, float nb, float re) {
        return liq(fe) ? re - m * ce - scale * ((float)(fe & CF_D) * ce - nb) : 0.f;
    };
    float4 v;
    v.x = one(f.x, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x);
    v.y = one(f.y, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y);
    v.z = one(f.z, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z);
    v.w = one(f.w, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w);
    *reinterpret_cast<float4 *>(eb + t) = c;
    *reinterpret_cast<float4 *>(res + t) = v;
}

// ---- one launch per step ------------------------------------------------------
// Each walks one list over every volume of a level.

// the volume of an element of a level's arrays
__device__ __forceinline__ int vol_of(const MgSpace &S, int t)
{
    return S.nv > 1 ? (t >= S.base[1]) + (t >= S.base[2]) : 0;
}

// One sweep over the active quads. With rzs (the last sweep of a V-cycle's level
// 0), it also forms r.eout, which is the solver's r.z: each block's compensated
// sum goes to the partials as block boff + blockIdx.x of btot (the blocks of the
// face volumes' launches together), and the last block to arrive sets beta =
// rz_new / rz (first: 0) and rz, as the solver's separate r.z pass does.
__global__ void __launch_bounds__(256) k_mg0_smooth(const MgSpace S, const int *__restrict__ qlist, int na,
                                                    const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                    const float *__restrict__ ein, float *eout, float scale, float m,
                                                    const int *done, SolveScal *rzs, double *partials, int first)
{
    __shared__ float wt[8];
    fill_wtab(wt, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    KSum acc;
    FS_FOR_LIST(qlist, na) acc.add(smooth_q(S.g[vol_of(S, 4 * q)], fl, r, ein, eout, wt, scale, m, q));
    if (!rzs || *(volatile const int *)&rzs->done) return;  // (a timed sweep runs after convergence too)
    KSum v[1] = {acc};
    double tot[1];
    if (grid_reduce<1>(v, partials, &rzs->ticket, tot) && threadIdx.x == 0) {
        if (!isfinite(tot[0])) {
            rzs->done = 1;
            rzs->status = FS_ENONFINITE;
            return;
        }
        rzs->beta = first ? 0.0 : tot[0] / rzs->rz;
        rzs->rz = tot[0];
    }
}

__global__ void __launch_bounds__(256) k_mg0_pre1(const MgSpace S, const int *__restrict__ qlist, int na,
                                                  const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                  float *eb, float *res, float scale, float m, const int *done)
{
    __shared__ float wt[8];
    fill_wtab(wt, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    FS_FOR_LIST(qlist, na) pre1_q(S.g[vol_of(S, 4 * q)], fl, r, eb, res, wt, scale, m, q);
}

__global__ void __launch_bounds__(256, 8) k_mg0_residual(const MgSpace S, const int *__restrict__ qlist, int na,
                                                      const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                      const float *__restrict__ ev, float *res, float scale, float m,
                                                      const int *done)
{
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    FS_FOR_LIST(qlist, na) resid_q(S.g[vol_of(S, 4 * q)], fl, r, ev, res, scale, m, q);
}

__global__ void __launch_bounds__(256) k_mg0_smooth2(const MgSpace S, const int *__restrict__ qlist, int na,
                                                     const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                     float *eo, float scale, float m, const int *done)
{
    __shared__ float wt[8];
    fill_wtab(wt, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    FS_FOR_LIST(qlist, na) smooth2_q(S.g[vol_of(S, 4 * q)], fl, r, eo, wt, scale, m, q);
}

__global__ void __launch_bounds__(256) k_mg0_prolong(const MgSpace S, const MgSpace Sc, const int *__restrict__ qlist,
                                                     int na, const uint8_t *__restrict__ fl, float *ef,
                                                     const float *__restrict__ ec, const int *done)
{
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    FS_FOR_LIST(qlist, na)
    {
        const int v = vol_of(S, 4 * q), base = S.base[v];
        prolong_q(S.g[v], fl + base, ef + base, Sc.g[v], ec + Sc.base[v], q - (base >> 2));
    }
}

// restriction over the coarse level's list of active pairs
__global__ void __launch_bounds__(256) k_mg0_restrict(const MgSpace S, const float *__restrict__ res, const MgSpace Sc,
                                                      const int *__restrict__ plist, int np,
                                                      const uint8_t *__restrict__ flc, float *rc, const int *done)
{
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    FS_FOR_LIST(plist, np)
    {
        const int v = vol_of(Sc, q), base = Sc.base[v];
        restrict_pair(S.g[v], res + S.base[v], Sc.g[v], flc + base, rc + base, q - base);
    }
}

// ---- lists of the active quads and restriction pairs ------------------------------
// Sorted and deterministic: block b owns items [b LB_ITEMS, (b + 1) LB_ITEMS), four
// consecutive items per thread; a first pass counts each block's kept items, the
// host scans the counts, and a second pass writes each block's items in order
// at its offset.
constexpr int LB_TH = 256, LB_PER = 4, LB_ITEMS = LB_TH * LB_PER;

struct QuadPred {  // a quad of the volume holds an unknown; listed as a quad of the level's arrays
    MgGrid g;
    const uint8_t *fl;
    int base;
    __device__ long long items() const { return g.n >> 2; }
    __device__ bool keep(long long q, int &out) const
    {
        out = (base >> 2) + (int)q;
        return any_liq(ldf4(fl, (int)q << 2));
    }
};
struct PairPred {  // a restriction pair (2m, 2m + 1) of the coarse level holds an unknown; its first element
    MgGrid g;
    const uint8_t *fl;
    int base;
    __device__ long long items() const { return (long long)((g.nx + 1) >> 1) * g.ny * g.nz; }
    __device__ bool keep(long long it, int &out) const
    {
        const int npair = (g.nx + 1) >> 1;
        const int m = (int)(it % npair);
        const long long jk = it / npair;
        const int J = (int)(jk % g.ny), K = (int)(jk / g.ny);
        const int t = g.idx(2 * m, J, K);
        out = base + t;
        return liq(fl[t]) || (2 * m + 1 < g.nx && liq(fl[t + 1]));
    }
};

template <class P>
__global__ void __launch_bounds__(LB_TH) k_list_build(P pred, const int *__restrict__ offsets, int *count, int *list)
{
    __shared__ int warp_tot[LB_TH / 32];
    const long long n = pred.items();
    const long long base = (long long)blockIdx.x * LB_ITEMS + (long long)threadIdx.x * LB_PER;
    int ids[LB_PER];
    int kept = 0;
#pragma unroll
    for (int k = 0; k < LB_PER; k++) {
        int id = 0;
        const bool keep = base + k < n && pred.keep(base + k, id);
        ids[k] = keep ? id : -1;
        kept += keep ? 1 : 0;
    }
    // inclusive scan of the kept counts over the block (warp shuffles, then warps)
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = kept;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    int before = 0, total = 0;
    for (int k = 0; k < LB_TH / 32; k++) {
        if (k < w) before += warp_tot[k];
        total += warp_tot[k];
    }
    if (!list) {  // counting pass
        if (threadIdx.x == 0) count[blockIdx.x] = total;
        return;
    }
    int pos = offsets[blockIdx.x] + before + incl - kept;
#pragma unroll
    for (int k = 0; k < LB_PER; k++)
        if (ids[k] >= 0) list[pos++] = ids[k];
}

// ---- set-up ------------------------------------------------------------------

// coarse flags from the level above: air if any child is air, else liquid if any
// child is liquid; the halo stays solid (zero)
__global__ void k_mg_coarsen(MgGrid gf, const uint8_t *__restrict__ flf, MgGrid gc, uint8_t *flc)
{
    MG_FOR_ROWS(gc)
    {
        const int t = row * gc.sy + e;
        const int I = e - gc.ioff, J = row % gc.rpp - gc.joff, K = row / gc.rpp - gc.koff;
        uint8_t out = 0;
        if (I >= 0 && J >= 0 && K >= 0 && I < gc.nx && J < gc.ny && K < gc.nz) {
            bool air = false, lq = false;
            for (int c = 0; c < 2; c++)
                for (int b = 0; b < 2; b++)
                    for (int a = 0; a < 2; a++) {
                        const int i = 2 * I + a, j = 2 * J + b, k = 2 * K + c;
                        if (i >= gf.nx || j >= gf.ny || k >= gf.nz) continue;
                        const uint8_t f = flf[gf.idx(i, j, k)];
                        air |= (f & CF_AIR) != 0;
                        lq |= (f & CF_LIQ) != 0;
                    }
            out = air ? CF_AIR : (lq ? CF_LIQ : 0);
        }
        flc[t] = out;
    }
}

// neighbour counts of the liquid cells: neighbours that are liquid or air
__global__ void k_mg_count(MgGrid g, uint8_t *fl)
{
    MG_FOR_ROWS(g)
    {
        const int t = row * g.sy + e;
        const uint8_t f = fl[t];
        if (!liq(f)) continue;
        const int off[6] = {-1, 1, -g.sy, g.sy, -g.sz, g.sz};
        int d = 0;
#pragma unroll
        for (int m = 0; m < 6; m++) d += (fl[t + off[m]] & (CF_LIQ | CF_AIR)) ? 1 : 0;
        fl[t] = (uint8_t)((f & ~CF_D) | d);
    }
}

#include "fs_mg_coarse.cuh"

// r.z over the active quads of a set's level 0 (r is zero off the unknowns, so no
// other quad adds to it), in the list's order: beta = rz_new / rz (first: beta =
// 0), as the dense pass of the solver does.
__global__ void __launch_bounds__(TH) k_mg_rz(const int *__restrict__ qlist, int na, const float *__restrict__ r,
                                             const float *__restrict__ z, int first, SolveScal *s, double *partials)
{
    dep_wait();
    dep_go();
    if (s->done) return;
    KSum acc;
    FS_FOR_LIST(qlist, na)
    {
        const float4 a = ldd4(r + 4 * q), b = ldd4(z + 4 * q);
        acc.add(a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w);
    }
    KSum v[1] = {acc};
    double tot[1];
    if (grid_reduce<1>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        if (!isfinite(tot[0])) {
            s->done = 1;
            s->status = FS_ENONFINITE;
            return;
        }
        s->beta = first ? 0.0 : tot[0] / s->rz;
        s->rz = tot[0];
    }
}

// number of unknown cells of a level (once per mask, for the profiled byte count)
__global__ void k_mg_count_liq(MgGrid g, const uint8_t *__restrict__ fl, unsigned long long *out)
{
    unsigned long long k = 0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < g.n; t += gridDim.x * blockDim.x) k += liq(fl[t]) ? 1 : 0;
    for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    if ((threadIdx.x & 31) == 0 && k) atomicAdd(out, k);
}

int row_blocks(fs_ctx *c, const MgGrid &g) { return grid_blocks(c, g.rows, 8); }

// a box of nx x ny x nz cells in the guarded layout of the context (pitch P, R
// rows per plane, a guard plane before and after): the cell space, or one face
// volume counted from its leading guard plane
MgGrid level0_grid(const Layout &L, int nx, int ny, int nz)
{
    MgGrid g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.sy = L.P;
    g.sz = L.PL;
    g.origin = L.PL;
    g.n = L.S + 2 * L.PL;
    g.rows = g.n / L.P;
    g.rpp = L.R;
    g.ioff = 0;
    g.joff = 0;
    g.koff = 1;
    return g;
}

// a coarse level: a solid halo of one plane and one row on each side, and of 4
// elements before each row (at least 1 after it), with the row pitch a multiple
// of 4, so that its quads are aligned like level 0's
MgGrid coarse_grid(int nx, int ny, int nz)
{
    MgGrid g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.sy = (nx + 5 + 3) / 4 * 4;
    g.sz = g.sy * (ny + 2);
    g.origin = g.sz + g.sy + 4;
    g.n = g.sz * (nz + 2);
    g.rows = (ny + 2) * (nz + 2);
    g.rpp = ny + 2;
    g.ioff = 4;
    g.joff = 1;
    g.koff = 1;
    return g;
}

void free_set(MgSet *t)
{
    for (int l = 0; l < MG_MAX_LEVELS; l++) {
        MgSetLevel &v = t->lev[l];
        cudaFree(v.pl);
        if (l > 0 || !t->shared0) cudaFree(v.ql);
        if (l > 0) {  // level 0 lies in the context's arrays and in MgAll's
            cudaFree(v.fl);
            for (float *p : {v.r, v.a, v.b, v.c}) cudaFree(p);
        }
        v = MgSetLevel();
    }
    cudaFree(t->blob);
    t->blob = nullptr;
    for (MgState *s : t->s)
        if (s) *s = MgState();
    t->nv = 0;
    t->by0[0] = -1.0;
}

// Resident blocks per SM of the list-walking kernels, for one-wave grids.
struct MgResidency {
    int smooth2, residual, pre1, restrict_, prolong, smooth;
};
const MgResidency &mg_residency()
{
    static const MgResidency r{resident_blocks((const void *)k_mg0_smooth2, 0),
                               resident_blocks((const void *)k_mg0_residual, 0),
                               resident_blocks((const void *)k_mg0_pre1, 0),
                               resident_blocks((const void *)k_mg0_restrict, 0),
                               resident_blocks((const void *)k_mg0_prolong, 0),
                               resident_blocks((const void *)k_mg0_smooth, 0)};
    return r;
}

MgcLevel coarse_level(const MgLevel &v) { return MgcLevel{v.g, v.fl, v.r, v.a, v.b, v.scale, v.mass}; }

// One leg (down or up) of level l >= 1 for the volumes of the set that hold it
// above their single-block levels.
int launch_leg(fs_ctx *c, const MgSet &t, int l, bool down, const int *done)
{
    MgLegArgs a;
    std::memset((void *)&a, 0, sizeof(a));
    a.done = done;
    int nv = 0, tiles = 0;
    size_t sm = 0;
    for (int v = 0; v < t.nv; v++) {
        const MgState &s = *t.s[v];
        if (l >= s.lb) continue;
        MgLegVol &x = a.v[nv++];
        x.f = coarse_level(s.lev[l]);
        x.c = coarse_level(s.lev[l + 1]);
    }
    for (int v = 0; v < nv; v++) {
        MgLegVol &x = a.v[v];
        x.t = make_tiles(x.f.g, nv, c->num_sms);
        tiles = std::max(tiles, x.t.ntx * x.t.nty * x.t.ntz);
        sm = std::max(sm, leg_smem(x.t, down));
    }
    if (!nv) return FS_OK;
    if (down)
        launch_dep(k_mg_down, dim3(tiles, nv), MGT_TH, sm, c->stream, a);
    else
        launch_dep(k_mg_up, dim3(tiles, nv), MGT_TH, sm, c->stream, a);
    c->n_launches += 1;
    return FS_OK;
}

// The arguments of the single-block levels lb .. nlev - 1 of every volume of the
// set (level 0's right-hand side and result left out), and their shared memory.
size_t bottom_args(const MgSet &t, MgBottomArgs &a)
{
    std::memset((void *)&a, 0, sizeof(a));
    size_t sm = 0, blob = 0;
    for (int v = 0; v < t.nv; v++) {
        const MgState &s = *t.s[v];
        MgBottomVol &x = a.v[v];
        x.nlev = s.nlev - s.lb;
        size_t off = 0, n = 0;
        for (int l = s.lb; l < s.nlev; l++) n += (size_t)s.lev[l].g.n;
        size_t foff = MGB_HEAD, qoff = foff + n;
        for (int l = s.lb; l < s.nlev; l++) {
            MgBottomLevel &b = x.lev[l - s.lb];
            b.l = coarse_level(s.lev[l]);
            b.off = (int)off;
            b.foff = (int)foff;
            b.qoff = (int)qoff;
            b.dsy = FastDiv(b.l.g.sy);
            b.dsz = FastDiv(b.l.g.sz);
            off += 3 * (size_t)b.l.g.n;
            foff += (size_t)b.l.g.n;
            qoff += (size_t)b.l.g.n / 2;
        }
        x.n = (int)n;
        x.bytes = (int)bottom_blob(n);
        x.blob = t.blob ? t.blob + blob : nullptr;
        blob += (size_t)x.bytes;
        sm = std::max(sm, bottom_smem(n));
    }
    return sm;
}

// One block for each volume's single-block levels. For a volume whose level 0 is
// its coarsest one, r0 and z0 are that level's arrays.
int launch_bottom(fs_ctx *c, const MgSet &t, const float *r0, float *z0, const int *done)
{
    MgBottomArgs a;
    const size_t sm = bottom_args(t, a);
    a.done = done;
    for (int v = 0; v < t.nv; v++)
        if (t.s[v]->lb == 0) {
            a.v[v].lev[0].l.r = const_cast<float *>(r0) + t.lev[0].sp.base[v];
            a.v[v].lev[0].l.a = z0 + t.lev[0].sp.base[v];
        }
    launch_dep(k_mg_bottom, t.nv, MGB_TH, sm, c->stream, a);
    c->n_launches += 1;
    return FS_OK;
}

// unknowns of levels 0 and 1, for the profiled byte counts: the least each level-0
// kernel must move is the list entry and the flags of each active quad (or pair)
// it visits and 4 bytes per unknown for each vector it reads or writes there
int count_bytes(fs_ctx *c, MgSet &t)
{
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(c->partials), nl[2] = {0, 0};
    FS_CUDA(cudaMemsetAsync(cnt, 0, sizeof(nl), c->stream));
    for (int v = 0; v < t.nv; v++) {
        const MgState &s = *t.s[v];
        k_mg_count_liq<<<grid_blocks(c, s.lev[0].g.n, TH), TH, 0, c->stream>>>(s.lev[0].g, s.lev[0].fl, cnt);
        if (s.nlev > 1)
            k_mg_count_liq<<<grid_blocks(c, s.lev[1].g.n, TH), TH, 0, c->stream>>>(s.lev[1].g, s.lev[1].fl, cnt + 1);
    }
    FS_CUDA(cudaMemcpyAsync(nl, cnt, sizeof(nl), cudaMemcpyDeviceToHost, c->stream));
    FS_CUDA(cudaStreamSynchronize(c->stream));
    const double u0 = (double)nl[0], u1 = (double)nl[1], q0 = (double)t.lev[0].nq, p1 = (double)t.lev[1].np;
    t.by0[0] = 8.0 * q0 + 8.0 * u0;             // smooth2: read r, write e
    t.by0[1] = 8.0 * q0 + 12.0 * u0;            // residual: read r, e, write res
    t.by0[2] = 6.0 * p1 + 4.0 * u0 + 4.0 * u1;  // restrict: pair list and flags, read res, write level-1 r
    t.by0[3] = 8.0 * q0 + 8.0 * u0 + 4.0 * u1;  // prolong: read and write e, read the level-1 e
    t.by0[4] = 8.0 * q0 + 12.0 * u0;            // smooth: read r, e, write e
    t.by0[5] = 8.0 * q0 + 12.0 * u0;            // last smooth: read r, e, write z
    return FS_OK;
}

// One V-cycle of a set: z = M r (whole-space arrays). With `sample` (the pressure
// V-cycle), every level-0 kernel and the coarse levels as a whole are timed; a
// timed kernel always runs in full (an early exit would record work not done).
// With rzs, r.z of the solver is formed in the last level-0 sweep.
int vcycle(fs_ctx *c, MgSet &t, const float *r, float *z, const int *done_, bool sample, SolveScal *rzs, int first)
{
    const MgState &s0 = *t.s[0];
    if (s0.nlev == 1) return launch_bottom(c, t, r, z, done_);
    if (sample && t.by0[0] < 0.0)
        if (int rc = count_bytes(c, t)) return rc;
    // an event pair around each timed launch (an event belongs to one pair)
    cudaEvent_t e0 = nullptr;
    auto begin = [&](int l) {
        if (sample && l == 0) e0 = prof_mark(c);
    };
    auto end = [&](int l, int kind, double bytes) {
        if (sample && l == 0) prof_add(c, kind, e0, prof_mark(c), bytes);
    };
    // four elements per thread, each kernel over the active quads in one wave of
    // its resident blocks (the volumes of a set share their scale)
    const MgResidency &res = mg_residency();
    cudaStream_t st = c->stream;
    for (int l = 0; l < t.lf; l++) {
        MgSetLevel &v = t.lev[l], &w = t.lev[l + 1];
        const float *rl = l == 0 ? r : v.r, scale = s0.lev[l].scale, mass = s0.lev[l].mass;
        const int *done = sample && l == 0 ? nullptr : done_;
        if (l == 0 && t.one) {  // the sweep from zero and the residual it leaves, in one pass
            launch_dep(k_mg0_pre1, wave_blocks(c, v.nq, res.pre1), TH, 0, st, v.sp, v.ql, v.nq, v.fl, rl, v.b, v.c, scale, mass,
                                                                      done);
            c->n_launches += 1;
        } else {
            begin(l);
            launch_dep(k_mg0_smooth2, wave_blocks(c, v.nq, res.smooth2), TH, 0, st, v.sp, v.ql, v.nq, v.fl, rl, v.b, scale,
                                                                            mass, done);
            end(l, K_MG0_SMOOTH2, t.by0[0]);
            begin(l);
            launch_dep(k_mg0_residual, wave_blocks(c, v.nq, res.residual), TH, 0, st, v.sp, v.ql, v.nq, v.fl, rl, v.b, v.c,
                                                                              scale, mass, done);
            end(l, K_MG0_RESIDUAL, t.by0[1]);
            c->n_launches += 2;
        }
        begin(l);
        launch_dep(k_mg0_restrict, wave_blocks(c, w.np, res.restrict_), TH, 0, st, v.sp, v.c, w.sp, w.pl, w.np, w.fl, w.r,
                                                                           done);
        end(l, K_MG0_RESTRICT, t.by0[2]);
        c->n_launches += 1;
        begin(l);
    }
    int lb = 0;
    for (int v = 0; v < t.nv; v++) lb = std::max(lb, t.s[v]->lb);
    for (int l = t.lf; l < lb; l++)
        if (int rc = launch_leg(c, t, l, true, done_)) return rc;
    if (int rc = launch_bottom(c, t, r, z, done_)) return rc;
    for (int l = lb - 1; l >= t.lf; l--)
        if (int rc = launch_leg(c, t, l, false, done_)) return rc;
    for (int l = t.lf - 1; l >= 0; l--) {
        MgSetLevel &v = t.lev[l], &w = t.lev[l + 1];
        const float *rl = l == 0 ? r : v.r, scale = s0.lev[l].scale, mass = s0.lev[l].mass;
        const int *done = sample && l == 0 ? nullptr : done_;
        const int nb = wave_blocks(c, v.nq, res.smooth);
        end(l, K_MG_COARSE, 0.0);
        begin(l);
        launch_dep(k_mg0_prolong, wave_blocks(c, v.nq, res.prolong), TH, 0, st, v.sp, w.sp, v.ql, v.nq, v.fl, v.b, w.a, done);
        end(l, K_MG0_PROLONG, t.by0[3]);
        const float *ez = v.c;  // the input of the last sweep
        if (l == 0 && t.one) {
            ez = v.b;
        } else {
            begin(l);
            launch_dep(k_mg0_smooth, nb, TH, 0, st, v.sp, v.ql, v.nq, v.fl, rl, v.b, v.c, scale, mass, done, nullptr, nullptr,
                                            0);
            end(l, K_MG0_SMOOTH, t.by0[4]);
            c->n_launches += 1;
        }
        begin(l);
        launch_dep(k_mg0_smooth, nb, TH, 0, st, v.sp, v.ql, v.nq, v.fl, rl, ez, l == 0 ? z : v.a, scale, mass, done,
                                        l == 0 ? rzs : nullptr, c->partials, first);
        end(l, K_MG0_SMOOTH_Z, t.by0[5]);
        c->n_launches += 2;
    }
    FS_CUDA(cudaGetLastError());
    return FS_OK;
}

// The grids of a volume's levels under level 0 (grid g0), and its single-block levels.
int plan_levels(fs_ctx *c, MgState *s, const MgGrid &g0, float coef, float mass)
{
    *s = MgState();
    s->lev[0].g = g0;
    s->nlev = 1;
    while (s->lev[s->nlev - 1].g.n > MG_COARSE_CELLS && s->nlev < MG_MAX_LEVELS) {
        const MgGrid &gf = s->lev[s->nlev - 1].g;
        MgLevel &v = s->lev[s->nlev++];
        v.g = coarse_grid((gf.nx + 1) / 2, (gf.ny + 1) / 2, (gf.nz + 1) / 2);
        if (v.g.nx == 1 && v.g.ny == 1 && v.g.nz == 1) break;
    }
    float sc = coef;
    for (int l = 0; l < s->nlev; l++, sc *= 0.25f) {
        s->lev[l].scale = sc;
        s->lev[l].mass = mass;
    }
    if (s->lev[s->nlev - 1].g.n > MG_COARSE_CELLS)
        return set_error(FS_EINVAL, "multigrid: the coarsest level does not fit in shared memory");
    for (int l = 0; l + 1 < s->nlev; l++) {  // the quad kernels' alignment (true by construction)
        const MgGrid &g = s->lev[l].g;
        if (g.sy % 4 || g.sz % 4 || g.origin % 4 || g.n % 4)
            return set_error(FS_EINVAL, "multigrid: level %d rows are not quad-aligned", l);
    }
    // the single-block launch takes the levels from the first one below level 0
    // (or the only level) that fits in shared memory with all below it
    size_t n = (size_t)s->lev[s->nlev - 1].g.n;
    s->lb = s->nlev - 1;
    while (s->lb > 1 && s->nlev - s->lb < MGB_MAXLEV && bottom_smem(n + (size_t)s->lev[s->lb - 1].g.n) <= MGB_SMEM) {
        s->lb -= 1;
        n += (size_t)s->lev[s->lb].g.n;
    }
    s->epoch = c->mask_epoch;
    s->coef = coef;
    return FS_OK;
}

// A list over the volumes of a level of a set, in order: counted, allocated, filled.
template <class P>
int make_list(fs_ctx *c, const MgSetLevel &v, long long (*items)(const MgGrid &), int **list, int *count)
{
    int *dcnt = nullptr;
    std::vector<int> hcnt;
    int blocks[3] = {0, 0, 0}, boff[4] = {0, 0, 0, 0};
    for (int k = 0; k < v.sp.nv; k++) {
        blocks[k] = (int)std::max(1LL, (items(v.sp.g[k]) + LB_ITEMS - 1) / LB_ITEMS);
        boff[k + 1] = boff[k] + blocks[k];
    }
    const int nb = boff[v.sp.nv];
    hcnt.resize((size_t)nb);
    if (cudaMalloc(&dcnt, sizeof(int) * (size_t)nb * 2) != cudaSuccess) {
        cudaGetLastError();
        return FS_ENOMEM;
    }
    auto launch = [&](const int *offs, int *out) {
        for (int k = 0; k < v.sp.nv; k++) {
            k_list_build<<<blocks[k], LB_TH, 0, c->stream>>>(P{v.sp.g[k], v.fl + v.sp.base[k], v.sp.base[k]},
                                                             offs ? offs + boff[k] : nullptr, dcnt + boff[k], out);
            c->n_launches += 1;
        }
    };
    int rc = FS_OK;
    launch(nullptr, nullptr);
    if ((rc = check_cuda(cudaGetLastError(), "k_list_build")) ||
        (rc = check_cuda(cudaMemcpyAsync(hcnt.data(), dcnt, sizeof(int) * (size_t)nb, cudaMemcpyDeviceToHost,
                                         c->stream), "cudaMemcpyAsync")) ||
        (rc = check_cuda(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize"))) {
        cudaFree(dcnt);
        return rc;
    }
    int total = 0;
    for (int b = 0; b < nb; b++) {  // exclusive scan of the block counts
        const int n = hcnt[b];
        hcnt[b] = total;
        total += n;
    }
    *count = total;
    if (cudaMalloc(list, sizeof(int) * (size_t)std::max(total, 1)) != cudaSuccess) {
        cudaGetLastError();
        *list = nullptr;
        cudaFree(dcnt);
        return FS_ENOMEM;
    }
    if (!(rc = check_cuda(cudaMemcpyAsync(dcnt + nb, hcnt.data(), sizeof(int) * (size_t)nb, cudaMemcpyHostToDevice,
                                          c->stream), "cudaMemcpyAsync"))) {
        launch(dcnt + nb, *list);
        rc = check_cuda(cudaGetLastError(), "k_list_build");
    }
    // the host counts must outlive the copy above
    if (!rc) rc = check_cuda(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    cudaFree(dcnt);
    return rc;
}

long long quad_items(const MgGrid &g) { return g.n / 4; }

// Arrays, flags and lists of a set whose volumes' levels are planned and whose
// level 0 is given (flags, work arrays, bases, and the list where it is shared).
int build_set(fs_ctx *c, MgSet &t)
{
    int nlev = 1, minlb = MG_MAX_LEVELS;
    for (int v = 0; v < t.nv; v++) {
        nlev = std::max(nlev, t.s[v]->nlev);
        minlb = std::min(minlb, t.s[v]->lb);
    }
    for (int l = 0; l < nlev; l++) {
        MgSetLevel &x = t.lev[l];
        x.sp.nv = t.nv;
        size_t n = 0;
        for (int v = 0; v < t.nv; v++) {
            x.sp.g[v] = t.s[v]->lev[l].g;
            if (l == 0) continue;
            x.sp.base[v] = (int)n;
            if (l < t.s[v]->nlev) n += (size_t)x.sp.g[v].n;
        }
        if (l == 0) {
            for (int v = 0; v < t.nv; v++) t.s[v]->lev[0].fl = x.fl + x.sp.base[v];
            continue;
        }
        bool ok = cudaMalloc(&x.fl, n) == cudaSuccess;
        for (float **p : {&x.r, &x.a, &x.b, &x.c}) ok = ok && cudaMalloc(p, n * 4) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            return set_error(FS_ENOMEM, "multigrid level arrays");
        }
        for (float *p : {x.r, x.a, x.b, x.c}) FS_CUDA(cudaMemsetAsync(p, 0, n * 4, c->stream));
        for (int v = 0; v < t.nv; v++) {
            if (l >= t.s[v]->nlev) continue;
            MgLevel &L = t.s[v]->lev[l];
            L.fl = x.fl + x.sp.base[v];
            L.r = x.r + x.sp.base[v];
            L.a = x.a + x.sp.base[v];
            L.b = x.b + x.sp.base[v];
            const int blocks = row_blocks(c, L.g);
            k_mg_coarsen<<<blocks, RT, 0, c->stream>>>(t.s[v]->lev[l - 1].g, t.s[v]->lev[l - 1].fl, L.g, L.fl);
            k_mg_count<<<blocks, RT, 0, c->stream>>>(L.g, L.fl);
            c->n_launches += 2;
        }
        FS_CUDA(cudaGetLastError());
    }
    {
        MgBottomArgs a;
        bottom_args(t, a);
        size_t bytes = 0;
        for (int v = 0; v < t.nv; v++) bytes += (size_t)a.v[v].bytes;
        if (cudaMalloc(&t.blob, bytes) != cudaSuccess) {
            cudaGetLastError();
            t.blob = nullptr;
            return set_error(FS_ENOMEM, "multigrid coarse lists");
        }
        bottom_args(t, a);
        k_mg_bottom_lists<<<t.nv, MGB_TH, 0, c->stream>>>(a);
        c->n_launches += 1;
        FS_CUDA(cudaGetLastError());
    }
    if (nlev == 1) return FS_OK;
    // A level takes the tile kernels where its tiles run in one wave: at 64^3 with
    // one volume a leg takes 7 us, the three list kernels with their gaps 14; with
    // three volumes (648 tiles on 304 slots) 20 us against 17.
    t.lf = 1;
    while (t.lf < minlb) {
        long long tiles = 0;
        for (int v = 0; v < t.nv; v++) {
            const MgTiles m = make_tiles(t.s[v]->lev[t.lf].g, t.nv, c->num_sms);
            tiles += (long long)m.ntx * m.nty * m.ntz;
        }
        if (tiles <= (long long)MGT_PER_SM * c->num_sms) break;
        t.lf += 1;
    }
    for (int l = 0; l <= t.lf; l++) {
        MgSetLevel &x = t.lev[l];
        int rc = FS_OK;
        if (l < t.lf && !x.ql)
            rc = make_list<QuadPred>(c, x, quad_items, &x.ql, &x.nq);
        if (!rc && l > 0)
            rc = make_list<PairPred>(
                c, x, [](const MgGrid &g) { return (long long)((g.nx + 1) >> 1) * g.ny * g.nz; }, &x.pl, &x.np);
        if (rc == FS_ENOMEM) return set_error(FS_ENOMEM, "multigrid active lists");
        if (rc) return rc;
    }
    return FS_OK;
}

MgAll *state(fs_ctx *c)
{
    MgAll *m = static_cast<MgAll *>(c->mg);
    if (!m) {
        m = new (std::nothrow) MgAll();
        c->mg = m;
    }
    return m;
}

// shared memory limits of the coarse-level kernels on the current device
int coarse_attributes()
{
    const int most = 218 * 1024;  // beside the static shared memory
    for (const void *f : {(const void *)k_mg_down, (const void *)k_mg_up, (const void *)k_mg_bottom})
        FS_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    return FS_OK;
}

// two zeroed work arrays of n floats, allocated once
int work_arrays(fs_ctx *c, float **a, float **b, size_t n, bool zero)
{
    if (!*a) {
        if (cudaMalloc(a, n * 4) != cudaSuccess || cudaMalloc(b, n * 4) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(*a);
            *a = nullptr;
            return set_error(FS_ENOMEM, "multigrid level-0 work arrays");
        }
        zero = true;
    }
    if (zero) {
        FS_CUDA(cudaMemsetAsync(*a, 0, n * 4, c->stream));
        FS_CUDA(cudaMemsetAsync(*b, 0, n * 4, c->stream));
    }
    return FS_OK;
}

}  // namespace

void mg_free(fs_ctx *c)
{
    MgAll *m = static_cast<MgAll *>(c->mg);
    if (!m) return;
    free_set(&m->cset);
    for (MgSet &t : m->fset) free_set(&t);
    for (float *p : {m->cb, m->cc, m->fb, m->fc}) cudaFree(p);
    delete m;
    c->mg = nullptr;
}

int cell_quads(fs_ctx *c, const int **ql, int *n)
{
    if (c->cq_epoch != c->mask_epoch || !c->cq) {
        cudaFree(c->cq);
        c->cq = nullptr;
        MgSetLevel v;
        v.sp.nv = 1;
        v.sp.g[0] = level0_grid(c->L, c->L.nx, c->L.ny, c->L.nz);
        v.sp.base[0] = 0;
        v.fl = c->cflag;
        if (int rc = make_list<QuadPred>(c, v, quad_items, &c->cq, &c->ncq))
            return rc == FS_ENOMEM ? set_error(FS_ENOMEM, "list of active quads") : rc;
        c->cq_epoch = c->mask_epoch;
    }
    *ql = c->cq;
    *n = c->ncq;
    return FS_OK;
}

// z = M r on the cell space (r and z of length nC, zero off the liquid); with
// rzs, r.z in the last level-0 sweep when the hierarchy has one (*fused tells)
static int apply_cell(fs_ctx *c, const float *r, float *z, const int *done, SolveScal *rzs, int first, bool *fused)
{
    if (fused) *fused = false;
    MgAll *m = state(c);
    if (!m) return set_error(FS_ENOMEM, "host allocation failed");
    const Layout &L = c->L;
    int rc;
    if (m->cell.epoch != c->mask_epoch) {
        MgSet &t = m->cset;
        free_set(&t);
        if ((rc = coarse_attributes()) || (rc = work_arrays(c, &m->cb, &m->cc, (size_t)L.nC, true)) ||
            (rc = plan_levels(c, &m->cell, level0_grid(L, L.nx, L.ny, L.nz), 1.f, 0.f)))
            return rc;
        t.nv = 1;
        t.s[0] = &m->cell;
        t.lev[0].fl = c->cflag;
        t.lev[0].b = m->cb;
        t.lev[0].c = m->cc;
        t.shared0 = true;
        const int *ql = nullptr;
        if ((rc = cell_quads(c, &ql, &t.lev[0].nq))) {
            free_set(&t);
            return rc;
        }
        t.lev[0].ql = const_cast<int *>(ql);
        if ((rc = build_set(c, t))) {
            free_set(&t);
            return rc;
        }
    }
    const bool fuse = rzs && m->cell.nlev >= 2;
    const bool sample = c->prof_on && (m->cset.calls++ % std::max(1, c->prof_period)) == 0;
    cudaEvent_t e0 = sample ? prof_mark(c) : nullptr;
    rc = vcycle(c, m->cset, r, z, done, sample, fuse ? rzs : nullptr, first);
    if (sample) prof_add(c, K_MG_VCYCLE_P, e0, prof_mark(c), 0.0);
    if (fused) *fused = fuse && rc == FS_OK;
    return rc;
}

int mg_apply(fs_ctx *c, const float *r, float *z, const int *done)
{
    return apply_cell(c, r, z, done, nullptr, 0, nullptr);
}

bool mg_apply_rz(fs_ctx *c, const float *r, float *z, const int *done, SolveScal *s, int first, int &rc)
{
    bool fused = false;
    rc = apply_cell(c, r, z, done, s, first, &fused);
    return fused;
}

// The three face hierarchies and their sets for the current mask.
static int build_faces(fs_ctx *c, MgAll *m, float cc)
{
    const Layout &L = c->L;
    int rc;
    for (MgSet &t : m->fset) free_set(&t);
    m->nfset = 0;
    if ((rc = coarse_attributes()) || (rc = work_arrays(c, &m->fb, &m->fc, (size_t)L.nF, true))) return rc;
    bool all = true;
    for (int k = 0; k < 3; k++) {
        if ((rc = plan_levels(c, &m->face[k], level0_grid(L, L.nx + (k == 0), L.ny + (k == 1), L.nz + (k == 2)), cc,
                              1.f)))
            return rc;
        all = all && m->face[k].nlev >= 2;
    }
    const int nset = all ? 1 : 3;
    for (int n = 0; n < nset; n++) {
        MgSet &t = m->fset[n];
        t.nv = all ? 3 : 1;
        t.lev[0].fl = c->fflag;
        t.lev[0].b = m->fb;
        t.lev[0].c = m->fc;
        t.one = true;
        for (int v = 0; v < t.nv; v++) {
            const int k = all ? v : n;
            t.s[v] = &m->face[k];
            t.lev[0].sp.base[v] = L.face_origin(k) - L.PL;  // the volume's leading guard plane
        }
        if ((rc = build_set(c, t))) {
            for (MgSet &f : m->fset) free_set(&f);
            return rc;
        }
    }
    m->nfset = nset;
    return FS_OK;
}

// z = M r on the face space for the Helmholtz operator I + cc L of the viscosity
// solve (r and z of length nF, zero off the unknown faces), the three velocity
// components' V-cycles launch by launch together. With `done` set, every kernel
// returns at once once *done != 0.
static int apply_faces(fs_ctx *c, const float *r, float *z, float cc, const int *done, SolveScal *rzs, int first,
                       bool *fused)
{
    if (fused) *fused = false;
    MgAll *m = state(c);
    if (!m) return set_error(FS_ENOMEM, "host allocation failed");
    if (m->nfset == 0 || m->face[0].epoch != c->mask_epoch) {
        if (int rc = build_faces(c, m, cc)) {
            m->nfset = 0;
            return rc;
        }
    } else if (m->face[0].coef != cc) {  // a new viscosity or time step: rescale the levels only
        for (MgState &s : m->face) {
            float sc = cc;
            for (int l = 0; l < s.nlev; l++, sc *= 0.25f) s.lev[l].scale = sc;
            s.coef = cc;
        }
    }
    const bool fuse = rzs && m->nfset == 1;
    const bool sample = c->prof_on && (m->fset[0].calls++ % std::max(1, c->prof_period)) == 0;
    cudaEvent_t e0 = sample ? prof_mark(c) : nullptr;
    for (int n = 0; n < m->nfset; n++)
        if (int rc = vcycle(c, m->fset[n], r, z, done, false, fuse ? rzs : nullptr, first)) return rc;
    if (sample) prof_add(c, K_MG_VCYCLE_V, e0, prof_mark(c), 0.0);
    if (fused) *fused = fuse;
    return FS_OK;
}

int mg_apply_faces(fs_ctx *c, const float *r, float *z, float cc, const int *done)
{
    return apply_faces(c, r, z, cc, done, nullptr, 0, nullptr);
}

bool mg_apply_faces_rz(fs_ctx *c, const float *r, float *z, float cc, const int *done, SolveScal *s, int first,
                       int &rc)
{
    bool fused = false;
    rc = apply_faces(c, r, z, cc, done, s, first, &fused);
    return fused;
}

// Launch counts of the level-0 kernels (fs_profile): `vcycles` V-cycles that did
// work on the pressure hierarchy, or on the face volumes together.
void mg_count(fs_ctx *c, long long vcycles, bool faces)
{
    const MgAll *m = static_cast<const MgAll *>(c->mg);
    if (!m || !c->prof_on) return;
    const int nlev = faces ? m->face[0].nlev : m->cell.nlev;
    if (nlev < 2) return;
    for (int id : {K_MG0_SMOOTH2, K_MG0_RESIDUAL, K_MG0_SMOOTH})
        if (!faces) prof_count(c, id, vcycles);  // the face volumes' level 0 skips three of the six kinds
    for (int id : {K_MG0_RESTRICT, K_MG0_PROLONG, K_MG0_SMOOTH_Z}) prof_count(c, id, vcycles);
    prof_count(c, faces ? K_MG_VCYCLE_V : K_MG_VCYCLE_P, vcycles);
    if (!faces) prof_count(c, K_MG_COARSE, vcycles);
}

// the set with level-0 lists for the current mask (of the pressure, or of the
// face volumes together), or null
static const MgSet *listed_set(const fs_ctx *c, bool faces)
{
    const MgAll *m = static_cast<const MgAll *>(c->mg);
    if (!m) return nullptr;
    const MgState &h = faces ? m->face[0] : m->cell;
    if (h.epoch != c->mask_epoch || h.nlev < 2 || (faces && m->nfset != 1)) return nullptr;
    return faces ? &m->fset[0] : &m->cset;
}

// r.z over the active quads of the pressure hierarchy's level 0 (or of the three
// face volumes'); false when the hierarchy has no lists (a level 0 that is its
// own coarsest level), and the caller takes the dense pass
bool mg_rz(fs_ctx *c, bool faces, const float *r, const float *z, int first, SolveScal *s)
{
    const MgSet *t = listed_set(c, faces);
    if (!t) return false;
    launch_dep(k_mg_rz, grid_blocks(c, t->lev[0].nq, TH), TH, 0, c->stream, t->lev[0].ql, t->lev[0].nq, r, z, first, s, c->partials);
    c->n_launches += 1;
    return cudaPeekAtLastError() == cudaSuccess;
}

// The level-0 list of active quads of the pressure hierarchy, or of the three
// face volumes together (quads of the whole face space); false when a hierarchy
// has no list for the current mask.
bool mg_level0_list(const fs_ctx *c, bool faces, const int **ql, int *n)
{
    const MgSet *t = listed_set(c, faces);
    if (!t) return false;
    *ql = t->lev[0].ql;
    *n = t->lev[0].nq;
    return true;
}

int mg_levels(const fs_ctx *c)
{
    const MgAll *m = static_cast<const MgAll *>(c->mg);
    return m ? m->cell.nlev : 0;
}

}  // namespace fs
