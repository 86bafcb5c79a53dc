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
// their other elements) and is zero on every other quad (but for the residual's x
// restriction, restrict_x): the work arrays are
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

// n / d for n d < 2^32 by one high multiply (m = ceil(2^32 / d); d = 1 kept apart)
struct FastDiv {
    unsigned m, d;
    __host__ __device__ FastDiv() : m(0), d(1) {}
    __host__ __device__ explicit FastDiv(unsigned dv) : m(dv > 1 ? (unsigned)(((1ull << 32) + dv - 1) / dv) : 0u), d(dv) {}
    __device__ __forceinline__ unsigned div(unsigned n) const { return d == 1 ? n : __umulhi(n, m); }
    __device__ __forceinline__ void split(unsigned n, unsigned &q, unsigned &r) const
    {
        q = div(n);
        r = n - q * d;
    }
    // any n: m exceeds 2^32 / d by less than 1, so the quotient is at most 1 too large
    __device__ __forceinline__ void split_any(unsigned n, unsigned &q, unsigned &r) const
    {
        q = div(n);
        r = n - q * d;
        if (r >= d) {
            q -= 1;
            r += d;
        }
    }
};

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
    FastDiv dq[3], dr[3];  // by the quads of a row and the rows of a plane
    void divisors()
    {
        for (int v = 0; v < nv; v++) {
            dq[v] = FastDiv((unsigned)g[v].sy / 4);
            dr[v] = FastDiv((unsigned)g[v].rpp);
        }
    }
};

// Where each volume's entries lie in a level's list: off[v] .. off[v + 1]. A launch
// gives each volume the same number of blocks, so that its grid is uniform over a
// block: picked per entry, its fields were loads from constant memory at a varying
// index and sat among the instructions that bound the large levels' kernels.
struct MgCut {
    int off[4];
    int blocks;  // per volume
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
    float *d = nullptr;  // the residual's x restriction, half the level's length, behind b
    int *ql = nullptr, *pl = nullptr;
    int nq = 0, np = 0;
    int qoff[4] = {0, 0, 0, 0}, poff[4] = {0, 0, 0, 0};
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
// level 0 belong here (work_arrays), of cell-space and face-space length.
struct MgAll {
    MgState cell, face[3];
    MgSet cset, fset[3];
    int nfset = 0;
    float *cb = nullptr, *cc = nullptr, *fb = nullptr;
};

namespace {

constexpr int TH = 256;
const dim3 RT(32, 8);  // a warp along a row, 8 rows per block

__device__ __forceinline__ bool liq(uint8_t f) { return f & CF_LIQ; }

// omega / (m + scale d), zero where the diagonal vanishes
__device__ __forceinline__ float wtab_entry(float scale, float m, int d)
{
    const float dg = m + scale * (float)d;
    return dg > 0.f ? MG_OMEGA / dg : 0.f;
}

// What a flag byte's low four bits (the count d and whether it is an unknown) stand
// for, in shared memory: omega / (m + scale d), and that with m + scale d; zero off
// the unknowns. The sweeps from zero form the first at five quads of r per quad, and
// were bound by their instructions: a lookup takes a byte permute, the load and the
// product, where testing and converting the byte took six.
struct WTab {
    float w[16];
    float2 c[16];
};
__device__ __forceinline__ void fill_wtab(WTab &tab, float scale, float m)
{
    const int i = threadIdx.x;
    if (i < 16) {
        const int d = i & CF_D;
        const float w = i & CF_LIQ ? wtab_entry(scale, m, d) : 0.f;
        tab.w[i] = w;
        tab.c[i] = make_float2(w, i & CF_LIQ ? m + scale * (float)d : 0.f);
    }
    __syncthreads();
}
static_assert((CF_D | CF_LIQ) == 15, "the table's index");

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
__device__ __forceinline__ unsigned ldw4(const uint8_t *__restrict__ p, int t)
{
    return __ldg(reinterpret_cast<const unsigned *>(p + t));
}
// the entries of element k of a quad's flag word W
__device__ __forceinline__ float w_of(const WTab &tab, unsigned W, int k)
{
    return *reinterpret_cast<const float *>(reinterpret_cast<const char *>(tab.w) +
                                            __byte_perm((W << 2) & 0x3c3c3c3cu, 0, 0x4440 | k));
}
__device__ __forceinline__ float2 c_of(const WTab &tab, unsigned W, int k)
{
    return *reinterpret_cast<const float2 *>(reinterpret_cast<const char *>(tab.c) +
                                             __byte_perm((W << 3) & 0x78787878u, 0, 0x4440 | k));
}
__device__ __forceinline__ bool any_liq(uchar4 f) { return ((f.x | f.y | f.z | f.w) & CF_LIQ) != 0; }

// e_out on element k of a quad from e_in: c (centre), the sum of its six neighbours nb
__device__ __forceinline__ float sweep1(const WTab &tab, unsigned W, int k, float c, float nb, float rv, float scale)
{
    const float2 t = c_of(tab, W, k);
    return W & (CF_LIQ << 8 * k) ? c + t.x * (rv - (t.y * c - scale * nb)) : 0.f;
}
// r - A e there
__device__ __forceinline__ float resid1(const WTab &tab, unsigned W, int k, float c, float nb, float rv, float scale)
{
    return W & (CF_LIQ << 8 * k) ? rv - (c_of(tab, W, k).y * c - scale * nb) : 0.f;
}

// The kernels below walk a level's list of active quads (those holding an
// unknown, built with the hierarchy): no flag load stands between a thread and its
// data loads, and the quads without an unknown cost nothing.

__device__ __forceinline__ float4 ldv4(const float *p, int t) { return ldd4(p + t); }
__device__ __forceinline__ float ldv1(const float *p, int t) { return ldd1(p + t); }

// one damped Jacobi sweep on quad q: eout from ein; returns r.eout over the quad
__device__ __forceinline__ float smooth_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r,
                                          const float *ein, float *eout, const WTab &tab, float scale, int q)
{
    const int t = q << 2;
    const unsigned W = ldw4(fl, t);
    const float4 c = ldv4(ein, t), rv = ldv4(r, t);
    const float4 dn = ldv4(ein, t - g.sy), up = ldv4(ein, t + g.sy);
    const float4 bk = ldv4(ein, t - g.sz), fw = ldv4(ein, t + g.sz);
    const float lf = ldv1(ein, t - 1), rt = ldv1(ein, t + 4);
    float4 v;
    v.x = sweep1(tab, W, 0, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x, scale);
    v.y = sweep1(tab, W, 1, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y, scale);
    v.z = sweep1(tab, W, 2, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z, scale);
    v.w = sweep1(tab, W, 3, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w, scale);
    *reinterpret_cast<float4 *>(eout + t) = v;
    return rv.x * v.x + rv.y * v.y + rv.z * v.z + rv.w * v.w;
}

// The x part of the restriction of a residual, v on the quad at element t of a
// volume's array: coarse cell 2m (fine 4m - 1 .. 4m + 2) and 2m + 1 (fine 4m + 1 ..
// 4m + 4) of the quad 4m .. 4m + 3, to elements t / 2 and t / 2 + 1 of d. So a residual
// is written and read at half its size, and the restriction needs no x neighbours.
// A neighbour that is not listed gets what this quad's end adds to it from here: its
// own elements add nothing, and its two cells each border one quad only. Nothing is
// added across the ends of a row.
__device__ __forceinline__ void restrict_x(const MgGrid &g, FastDiv dq, Links lk, float4 v, float *d, int t)
{
    unsigned row, e;
    dq.split_any((unsigned)t >> 2, row, e);
    const int i = (int)(4 * e) - g.ioff;
    const bool lin = i > 0, rin = i + 4 < g.nx;
    const float l = lk.left(v.w), r = lk.right(v.x);
    if (!lk.own) return;
    float *o = d + (t >> 1);
    *reinterpret_cast<float2 *>(o) =
        make_float2(0.25f * (lin ? l : 0.f) + 0.75f * v.x + 0.75f * v.y + 0.25f * v.z,
                    0.25f * v.y + 0.75f * v.z + 0.75f * v.w + 0.25f * (rin ? r : 0.f));
    if (lin && !lk.l) o[-1] = 0.25f * v.x;
    if (rin && !lk.r) o[2] = 0.25f * v.w;
}

// r - A e on quad q
__device__ __forceinline__ float4 resid_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r,
                                          const float *ev, const WTab &tab, float scale, int q, Links lk)
{
    const int t = q << 2;
    const unsigned W = ldw4(fl, t);
    const float4 c = ldv4(ev, t), rv = ldv4(r, t);
    const float4 dn = ldv4(ev, t - g.sy), up = ldv4(ev, t + g.sy);
    const float4 bk = ldv4(ev, t - g.sz), fw = ldv4(ev, t + g.sz);
    const float lf = lk.left(c.w), rt = lk.right(c.x);
    float4 v;
    v.x = resid1(tab, W, 0, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x, scale);
    v.y = resid1(tab, W, 1, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y, scale);
    v.z = resid1(tab, W, 2, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z, scale);
    v.w = resid1(tab, W, 3, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w, scale);
    return v;
}

// omega D^-1 r on the quad at element u
__device__ __forceinline__ float4 jacobi_q(const uint8_t *__restrict__ fl, const float *r, const WTab &tab, int u)
{
    const unsigned W = ldw4(fl, u);
    const float4 v = ldv4(r, u);
    return make_float4(w_of(tab, W, 0) * v.x, w_of(tab, W, 1) * v.y, w_of(tab, W, 2) * v.z, w_of(tab, W, 3) * v.w);
}

// the first two sweeps from e = 0 on quad q: e1 = omega D^-1 r on the fly, then one sweep
__device__ __forceinline__ void smooth2_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r, float *eo,
                                          const WTab &tab, float scale, int q, Links lk)
{
    const int t = q << 2;
    const unsigned W = ldw4(fl, t);
    const float4 c = jacobi_q(fl, r, tab, t), rv = ldv4(r, t);
    const float4 dn = jacobi_q(fl, r, tab, t - g.sy), up = jacobi_q(fl, r, tab, t + g.sy);
    const float4 bk = jacobi_q(fl, r, tab, t - g.sz), fw = jacobi_q(fl, r, tab, t + g.sz);
    const float lf = lk.left(c.w), rt = lk.right(c.x);
    float4 v;
    v.x = sweep1(tab, W, 0, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x, scale);
    v.y = sweep1(tab, W, 1, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y, scale);
    v.z = sweep1(tab, W, 2, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z, scale);
    v.w = sweep1(tab, W, 3, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w, scale);
    if (lk.own) *reinterpret_cast<float4 *>(eo + t) = v;
}

// cell (i, j, k) of element t of a volume's array
__device__ __forceinline__ void cell_of(const MgGrid &g, FastDiv dq, FastDiv dr, int t, int &i, int &j, int &k)
{
    unsigned row, e, pl, r;
    dq.split_any((unsigned)t >> 2, row, e);
    dr.split_any(row, pl, r);
    i = (int)(4 * e + ((unsigned)t & 3u)) - g.ioff;
    j = (int)r - g.joff;
    k = (int)pl - g.koff;
}

// e_fine += P e_coarse on the unknowns of an active quad q (in place). The quad's
// elements i .. i + 3 (i a multiple of 4) take their x samples from coarse
// I0 - 1 .. I0 + 2 (I0 = i / 2, even, so that I0 and I0 + 1 are one aligned load;
// the outer two are the neighbour lanes' where those hold the row's next quads).
// I0 + 2 past the coarse halo is clamped to it (a sample that only padding
// elements use). With FIRST, e_fine before it is the sweep from zero, omega D^-1 r,
// formed here.
template <bool FIRST>
__device__ __forceinline__ void prolong_q(const MgGrid &gf, FastDiv dq, FastDiv dr, const uint8_t *__restrict__ fl,
                                          float *ef, const MgGrid &gc, const float *ec, const float *r,
                                          const WTab &tab, int q, Links lk)
{
    const int t = q << 2;
    const uchar4 f = ldf4(fl, t);
    int i, j, k;
    cell_of(gf, dq, dr, t, i, j, k);
    const int I0 = i >> 1, J = j >> 1, K = k >> 1;
    const int J2 = (j & 1) ? J + 1 : J - 1, K2 = (k & 1) ? K + 1 : K - 1;
    const int xr = min(I0 + 2, gc.nx);
    const bool ll = lk.l && i > 0, lr = lk.r && i + 4 < gf.nx;  // the neighbour's quad is in this row
    const int base[4] = {gc.idx(0, J, K), gc.idx(0, J2, K), gc.idx(0, J, K2), gc.idx(0, J2, K2)};
    const float w[4] = {0.5625f, 0.1875f, 0.1875f, 0.0625f};
    float4 v = FIRST ? jacobi_q(fl, r, tab, t) : ldv4(ef, t);
    // the y and z parts first: the neighbour lanes' quads of the row share them
    float c0 = 0.f, c1 = 0.f, cm = 0.f, c2 = 0.f;
#pragma unroll
    for (int x = 0; x < 4; x++) {
        const float2 c = ldd2(ec + base[x] + I0);
        c0 += w[x] * c.x;
        c1 += w[x] * c.y;
    }
    if (!ll)
#pragma unroll
        for (int x = 0; x < 4; x++) cm += w[x] * ldv1(ec, base[x] + I0 - 1);
    if (!lr)
#pragma unroll
        for (int x = 0; x < 4; x++) c2 += w[x] * ldv1(ec, base[x] + xr);
    const float sl = __shfl_up_sync(FULL_WARP, c1, 1), sr = __shfl_down_sync(FULL_WARP, c0, 1);
    if (ll) cm = sl;
    if (lr) c2 = sr;
    const float s0 = 0.75f * c0 + 0.25f * cm, s1 = 0.75f * c0 + 0.25f * c1;
    const float s2 = 0.75f * c1 + 0.25f * c0, s3 = 0.75f * c1 + 0.25f * c2;
    if (liq(f.x)) v.x += s0;
    if (liq(f.y)) v.y += s1;
    if (liq(f.z)) v.z += s2;
    if (liq(f.w)) v.w += s3;
    if (lk.own) *reinterpret_cast<float4 *>(ef + t) = v;
}

// Restriction of an active pair of the coarse level: t0 is the element of coarse
// cell (2m, J, K), and the pair (2m, 2m + 1) holds at least one unknown. It weighs
// the x parts (restrict_x) of a 4 x 4 window of fine rows: all of it (WHOLE), or the
// plane c of each of four lanes, 8 apart, that share the pair.
template <bool WHOLE>
__device__ __forceinline__ void restrict_pair(const MgGrid &gf, const float *d, const MgGrid &gc, FastDiv dq,
                                              FastDiv dr, const uint8_t *__restrict__ flc, float *rc, int t0, int c,
                                              bool own)
{
    int I0, J, K;
    cell_of(gc, dq, dr, t0, I0, J, K);
    const bool l0 = liq(flc[t0]), l1 = I0 + 1 < gc.nx && liq(flc[t0 + 1]);
    // A row off the grid counts nothing: its weight is zero and the pair's own row
    // is read in its place, so that no branch stands between the rows' loads (with a
    // skip per row each waited for the one before it: 12 us for the 64^3 level of
    // the three face volumes of 128^3, and the sweeps 4). Rows -1 and ny, planes -1
    // and nz are the only ones off the grid.
    const float wy0 = J > 0 ? 0.25f : 0.f, wy2 = 2 * J + 1 < gf.ny ? 0.75f : 0.f, wy3 = 2 * J + 2 < gf.ny ? 0.25f : 0.f;
    const float wz0 = K > 0 ? 0.25f : 0.f, wz2 = 2 * K + 1 < gf.nz ? 0.75f : 0.f, wz3 = 2 * K + 2 < gf.nz ? 0.25f : 0.f;
    const int y0 = J > 0 ? -gf.sy : 0, y2 = 2 * J + 1 < gf.ny ? gf.sy : 0, y3 = 2 * J + 2 < gf.ny ? 2 * gf.sy : 0;
    const int z0 = K > 0 ? -gf.sz : 0, z2 = 2 * K + 1 < gf.nz ? gf.sz : 0, z3 = 2 * K + 2 < gf.nz ? 2 * gf.sz : 0;
    const int own_row = gf.idx(0, 2 * J, 2 * K) + 2 * I0;  // a multiple of 4
    float a0 = 0.f, a1 = 0.f;
    auto plane = [&](int z, float wz) {
        const int p = own_row + z;
        const float2 x0 = ldd2(d + ((p + y0) >> 1)), x1 = ldd2(d + (p >> 1));
        const float2 x2 = ldd2(d + ((p + y2) >> 1)), x3 = ldd2(d + ((p + y3) >> 1));
        a0 += wz * (wy0 * x0.x + 0.75f * x1.x + wy2 * x2.x + wy3 * x3.x);
        a1 += wz * (wy0 * x0.y + 0.75f * x1.y + wy2 * x2.y + wy3 * x3.y);
    };
    if (WHOLE) {
        plane(z0, wz0);
        plane(0, 0.75f);
        plane(z2, wz2);
        plane(z3, wz3);
        if (own && l0) rc[t0] = 0.125f * a0;
        if (own && l1) rc[t0 + 1] = 0.125f * a1;
        return;
    }
    plane(c == 0 ? z0 : c == 1 ? 0 : c == 2 ? z2 : z3, c == 0 ? wz0 : c == 1 ? 0.75f : c == 2 ? wz2 : wz3);
#pragma unroll
    for (int o = 8; o < 32; o *= 2) {
        a0 += __shfl_xor_sync(FULL_WARP, a0, o);
        a1 += __shfl_xor_sync(FULL_WARP, a1, o);
    }
    if (own && c == 0 && l0) rc[t0] = 0.125f * a0;
    if (own && c == 1 && l1) rc[t0 + 1] = 0.125f * a1;
}

// r - A e1 on quad q for the damped Jacobi sweep from zero, e1 = omega D^-1 r
// (formed on the fly, here and where it is used again)
__device__ __forceinline__ float4 pre1_q(const MgGrid &g, const uint8_t *__restrict__ fl, const float *r,
                                         const WTab &tab, float scale, int q, Links lk)
{
    const int t = q << 2;
    const unsigned W = ldw4(fl, t);
    const float4 c = jacobi_q(fl, r, tab, t), rv = ldv4(r, t);
    const float4 dn = jacobi_q(fl, r, tab, t - g.sy), up = jacobi_q(fl, r, tab, t + g.sy);
    const float4 bk = jacobi_q(fl, r, tab, t - g.sz), fw = jacobi_q(fl, r, tab, t + g.sz);
    const float lf = lk.left(c.w), rt = lk.right(c.x);
    float4 v;
    v.x = resid1(tab, W, 0, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), rv.x, scale);
    v.y = resid1(tab, W, 1, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), rv.y, scale);
    v.z = resid1(tab, W, 2, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), rv.z, scale);
    v.w = resid1(tab, W, 3, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), rv.w, scale);
    return v;
}

// ---- one launch per step ------------------------------------------------------
// Each walks one list over every volume of a level, with blocks of its own for
// each volume.

// What bounds them (measured one by one): above a few million unknowns the bytes,
// and for the kernels that form a sweep on the fly or take two grids the
// instructions; below, latency (a launch, the list, the loads). The three face
// volumes at 256^3, 20 M unknowns: pre1 66 us (with a test and a conversion of each
// flag byte 73), prolong 51 (56), smooth 59 (4.8 TB/s of its bytes).
// The sweeps that are not followed by a restriction keep the plain walk: windows of
// 30 quads start off a 128-byte line, which cost a sweep 4% there.

// One sweep over the active quads. With rzs (the last sweep of a V-cycle's level
// 0), it also forms r.eout, which is the solver's r.z: each block's compensated
// sum goes to the partials as block boff + blockIdx.x of btot (the blocks of the
// face volumes' launches together), and the last block to arrive sets beta =
// rz_new / rz (first: 0) and rz, as the solver's separate r.z pass does.
__global__ void __launch_bounds__(256) k_mg0_smooth(const __grid_constant__ MgSpace S, const int *__restrict__ qlist, const __grid_constant__ MgCut cut,
                                                    const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                    const float *__restrict__ ein, float *eout, float scale, float m,
                                                    const int *done, SolveScal *rzs, double *partials, int first)
{
    __shared__ WTab tab;
    fill_wtab(tab, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    KSum acc;
    const int v = blockIdx.x / cut.blocks, blk = blockIdx.x - v * cut.blocks;
    const int na = cut.off[v + 1] - cut.off[v];
    FS_FOR_LIST_PART(qlist + cut.off[v], na, blk, cut.blocks)
    acc.add(smooth_q(S.g[v], fl, r, ein, eout, tab, scale, q));
    if (!rzs || *(volatile const int *)&rzs->done) return;  // (a timed sweep runs after convergence too)
    KSum sum[1] = {acc};
    double tot[1];
    if (grid_reduce<1>(sum, partials, &rzs->ticket, tot) && threadIdx.x == 0) {
        if (!isfinite(tot[0])) {
            rzs->done = 1;
            rzs->status = FS_ENONFINITE;
            return;
        }
        rzs->beta = first ? 0.0 : tot[0] / rzs->rz;
        rzs->rz = tot[0];
    }
}

__global__ void __launch_bounds__(256, 6) k_mg0_pre1(const __grid_constant__ MgSpace S, const int *__restrict__ qlist, const __grid_constant__ MgCut cut,
                                                  const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                  float *d, float scale, float m, const int *done)
{
    __shared__ WTab tab;
    fill_wtab(tab, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    const int v = blockIdx.x / cut.blocks, blk = blockIdx.x - v * cut.blocks, base = S.base[v];
    const int na = cut.off[v + 1] - cut.off[v];
    FS_FOR_LIST_LINKED(qlist + cut.off[v], na, blk, cut.blocks)
    {
        const Links lk = links(q, fl_i, na);
        const float4 res = pre1_q(S.g[v], fl, r, tab, scale, q, lk);
        restrict_x(S.g[v], S.dq[v], lk, res, d + (base >> 1), 4 * q - base);
    }
}

__global__ void __launch_bounds__(256, 6) k_mg0_residual(const __grid_constant__ MgSpace S, const int *__restrict__ qlist, const __grid_constant__ MgCut cut,
                                                      const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                      const float *__restrict__ ev, float *d, float scale, float m,
                                                      const int *done)
{
    __shared__ WTab tab;
    fill_wtab(tab, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    const int v = blockIdx.x / cut.blocks, blk = blockIdx.x - v * cut.blocks, base = S.base[v];
    const int na = cut.off[v + 1] - cut.off[v];
    FS_FOR_LIST_LINKED(qlist + cut.off[v], na, blk, cut.blocks)
    {
        const Links lk = links(q, fl_i, na);
        const float4 res = resid_q(S.g[v], fl, r, ev, tab, scale, q, lk);
        restrict_x(S.g[v], S.dq[v], lk, res, d + (base >> 1), 4 * q - base);
    }
}

__global__ void __launch_bounds__(256, 6) k_mg0_smooth2(const __grid_constant__ MgSpace S, const int *__restrict__ qlist, const __grid_constant__ MgCut cut,
                                                     const uint8_t *__restrict__ fl, const float *__restrict__ r,
                                                     float *eo, float scale, float m, const int *done)
{
    __shared__ WTab tab;
    fill_wtab(tab, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    const int v = blockIdx.x / cut.blocks, blk = blockIdx.x - v * cut.blocks;
    const int na = cut.off[v + 1] - cut.off[v];
    FS_FOR_LIST_LINKED(qlist + cut.off[v], na, blk, cut.blocks)
    smooth2_q(S.g[v], fl, r, eo, tab, scale, q, links(q, fl_i, na));
}

template <bool FIRST>
__global__ void __launch_bounds__(256) k_mg0_prolong(const __grid_constant__ MgSpace S, const __grid_constant__ MgSpace Sc, const int *__restrict__ qlist,
                                                     const __grid_constant__ MgCut cut, const uint8_t *__restrict__ fl, float *ef,
                                                     const float *__restrict__ ec, const float *r, float scale, float m,
                                                     const int *done)
{
    __shared__ WTab tab;
    if (FIRST) fill_wtab(tab, scale, m);
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    const int v = blockIdx.x / cut.blocks, blk = blockIdx.x - v * cut.blocks, base = S.base[v];
    const int na = cut.off[v + 1] - cut.off[v];
    FS_FOR_LIST_LINKED(qlist + cut.off[v], na, blk, cut.blocks)
    {
        prolong_q<FIRST>(S.g[v], S.dq[v], S.dr[v], fl + base, ef + base, Sc.g[v], ec + Sc.base[v], r + base, tab,
                         q - (base >> 2), links(q, fl_i, na));
    }
}

// Restriction over the coarse level's list of active pairs. Pairs take a thread each
// (WHOLE): the index arithmetic bounds the large levels (the three face volumes,
// 20 M unknowns at 256^3: 20 us against 37 with four lanes per pair, and 45 over whole
// residuals with their x neighbours; 2.5 M at 128^3: 7.4 against 9.3 and 13.5). Where
// four lanes per pair fit in one wave they are used, for four times the loads in
// flight (the 64^3 level below a pressure blob: 4.7 us against 6.0 and 9.1).
template <bool WHOLE>
__global__ void __launch_bounds__(256) k_mg0_restrict(const __grid_constant__ MgSpace S, const float *__restrict__ d,
                                                      const __grid_constant__ MgSpace Sc,
                                                      const int *__restrict__ plist, const __grid_constant__ MgCut cut,
                                                      const uint8_t *__restrict__ flc, float *rc, const int *done)
{
    dep_wait();
    dep_go();
    if (done && *(volatile const int *)done) return;  // the solve has converged
    const int v = blockIdx.x / cut.blocks, blk = blockIdx.x - v * cut.blocks, base = Sc.base[v];
    const int np = cut.off[v + 1] - cut.off[v];
    plist += cut.off[v];
    // a warp takes 32 or 8 consecutive pairs, all lanes in each step
    constexpr int PER = WHOLE ? 32 : 8;
    const int lane = threadIdx.x & 31, st = cut.blocks * (int)(blockDim.x >> 5) * PER;
    int i = (int)((blk * blockDim.x + threadIdx.x) >> 5) * PER + (lane & (PER - 1));
    int next = (i & ~(PER - 1)) < np ? __ldg(plist + min(i, np - 1)) : 0;
    for (; (i & ~(PER - 1)) < np; i += st) {
        const int q = next;
        next = (i & ~(PER - 1)) + st < np ? __ldg(plist + min(i + st, np - 1)) : 0;
        restrict_pair<WHOLE>(S.g[v], d + (S.base[v] >> 1), Sc.g[v], Sc.dq[v], Sc.dr[v], flc + base, rc + base, q - base,
                             lane >> 3, i < np);
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
    int smooth2, residual, pre1, whole, split, prolong, first, smooth;
};
const MgResidency &mg_residency()
{
    static const MgResidency r{resident_blocks((const void *)k_mg0_smooth2, 0),
                               resident_blocks((const void *)k_mg0_residual, 0),
                               resident_blocks((const void *)k_mg0_pre1, 0),
                               resident_blocks((const void *)k_mg0_restrict<true>, 0),
                               resident_blocks((const void *)k_mg0_restrict<false>, 0),
                               resident_blocks((const void *)k_mg0_prolong<false>, 0),
                               resident_blocks((const void *)k_mg0_prolong<true>, 0),
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
    t.by0[1] = 8.0 * q0 + 10.0 * u0;            // residual: read r, e, write its x restriction
    t.by0[2] = 6.0 * p1 + 2.0 * u0 + 4.0 * u1;  // restrict: pair list and flags, read that, write level-1 r
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
    auto cut = [&](const int *off, int kind, int resident) {  // kind: threads per entry, or 0 for linked quads
        MgCut m;
        long long most = 0;
        for (int v = 0; v < 4; v++) m.off[v] = off[v];
        for (int v = 0; v < t.nv; v++) {
            const long long n = off[v + 1] - off[v];
            most = std::max(most, kind ? kind * n : linked_threads(n));
        }
        m.blocks = (int)std::max(1LL, std::min((most + TH - 1) / TH, (long long)c->num_sms * std::max(resident, 1) / t.nv));
        return m;
    };
    MgCut k;
    for (int l = 0; l < t.lf; l++) {
        MgSetLevel &v = t.lev[l], &w = t.lev[l + 1];
        const float *rl = l == 0 ? r : v.r, scale = s0.lev[l].scale, mass = s0.lev[l].mass;
        const int *done = sample && l == 0 ? nullptr : done_;
        if (l == 0 && t.one) {  // the sweep from zero and the residual it leaves, in one pass
            k = cut(v.qoff, 0, res.pre1);
            launch_dep(k_mg0_pre1, k.blocks * t.nv, TH, 0, st, v.sp, v.ql, k, v.fl, rl, v.d, scale, mass,
                       done);
            c->n_launches += 1;
        } else {
            k = cut(v.qoff, 0, res.smooth2);
            begin(l);
            launch_dep(k_mg0_smooth2, k.blocks * t.nv, TH, 0, st, v.sp, v.ql, k, v.fl, rl, v.b, scale,
                       mass, done);
            end(l, K_MG0_SMOOTH2, t.by0[0]);
            k = cut(v.qoff, 0, res.residual);
            begin(l);
            launch_dep(k_mg0_residual, k.blocks * t.nv, TH, 0, st, v.sp, v.ql, k, v.fl, rl, v.b, v.d,
                       scale, mass, done);
            end(l, K_MG0_RESIDUAL, t.by0[1]);
            c->n_launches += 2;
        }
        const bool whole = 4LL * w.np > (long long)c->num_sms * res.split * TH;
        k = cut(w.poff, whole ? 1 : 4, whole ? res.whole : res.split);
        begin(l);
        launch_dep(whole ? k_mg0_restrict<true> : k_mg0_restrict<false>, k.blocks * t.nv, TH, 0, st, v.sp, v.d, w.sp, w.pl, k, w.fl, w.r,
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
        end(l, K_MG_COARSE, 0.0);
        begin(l);
        const bool one = l == 0 && t.one;
        k = cut(v.qoff, 0, one ? res.first : res.prolong);
        launch_dep(one ? k_mg0_prolong<true> : k_mg0_prolong<false>, k.blocks * t.nv, TH, 0, st, v.sp, w.sp, v.ql,
                   k, v.fl, v.b, w.a, rl, scale, mass, done);
        end(l, K_MG0_PROLONG, t.by0[3]);
        const float *ez = v.c;  // the input of the last sweep
        k = cut(v.qoff, 1, res.smooth);
        if (l == 0 && t.one) {
            ez = v.b;
        } else {
            begin(l);
            launch_dep(k_mg0_smooth, k.blocks * t.nv, TH, 0, st, v.sp, v.ql, k, v.fl, rl, v.b, v.c, scale, mass, done, nullptr, nullptr,
                                            0);
            end(l, K_MG0_SMOOTH, t.by0[4]);
            c->n_launches += 1;
        }
        begin(l);
        launch_dep(k_mg0_smooth, k.blocks * t.nv, TH, 0, st, v.sp, v.ql, k, v.fl, rl, ez, l == 0 ? z : v.a, scale, mass, done,
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

// A list over the volumes of a level of a set, in order: counted, allocated, filled;
// off[v] is where volume v begins (the whole count past the last).
template <class P>
int make_list(fs_ctx *c, const MgSetLevel &v, long long (*items)(const MgGrid &), int **list, int *count, int *off)
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
    for (int k = 0; k < 4; k++) off[k] = k < v.sp.nv ? hcnt[boff[k]] : total;
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
        x.sp.divisors();
        if (l == 0) {
            for (int v = 0; v < t.nv; v++) t.s[v]->lev[0].fl = x.fl + x.sp.base[v];
            continue;
        }
        bool ok = cudaMalloc(&x.fl, n) == cudaSuccess;
        for (float **p : {&x.r, &x.a, &x.c}) ok = ok && cudaMalloc(p, n * 4) == cudaSuccess;
        ok = ok && cudaMalloc(&x.b, n * 6) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            return set_error(FS_ENOMEM, "multigrid level arrays");
        }
        for (float *p : {x.r, x.a, x.c}) FS_CUDA(cudaMemsetAsync(p, 0, n * 4, c->stream));
        FS_CUDA(cudaMemsetAsync(x.b, 0, n * 6, c->stream));
        x.d = x.b + n;
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
            rc = make_list<QuadPred>(c, x, quad_items, &x.ql, &x.nq, x.qoff);
        if (!rc && l > 0)
            rc = make_list<PairPred>(
                c, x, [](const MgGrid &g) { return (long long)((g.nx + 1) >> 1) * g.ny * g.nz; }, &x.pl, &x.np, x.poff);
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

// level 0's zeroed work arrays, allocated once: *a with the half-length one behind
// it (MgSetLevel::b and d), and where b is given a second one of n floats
int work_arrays(fs_ctx *c, float **a, float **b, size_t n)
{
    if (!*a) {
        if (cudaMalloc(a, n * 6) != cudaSuccess || (b && cudaMalloc(b, n * 4) != cudaSuccess)) {
            cudaGetLastError();
            cudaFree(*a);
            *a = nullptr;
            return set_error(FS_ENOMEM, "multigrid level-0 work arrays");
        }
    }
    FS_CUDA(cudaMemsetAsync(*a, 0, n * 6, c->stream));
    if (b) FS_CUDA(cudaMemsetAsync(*b, 0, n * 4, c->stream));
    return FS_OK;
}

}  // namespace

void mg_free(fs_ctx *c)
{
    MgAll *m = static_cast<MgAll *>(c->mg);
    if (!m) return;
    free_set(&m->cset);
    for (MgSet &t : m->fset) free_set(&t);
    for (float *p : {m->cb, m->cc, m->fb}) cudaFree(p);
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
        if (int rc = make_list<QuadPred>(c, v, quad_items, &c->cq, &c->ncq, v.qoff))
            return rc == FS_ENOMEM ? set_error(FS_ENOMEM, "list of active quads") : rc;
        c->cq_epoch = c->mask_epoch;
    }
    *ql = c->cq;
    *n = c->ncq;
    return FS_OK;
}

// the same over the three face volumes, in the face space's quads; off: where each
// volume begins
int face_quads(fs_ctx *c, const int **ql, int *n, int *off)
{
    if (c->fq_epoch != c->mask_epoch || !c->fq) {
        cudaFree(c->fq);
        c->fq = nullptr;
        MgSetLevel v;
        v.sp.nv = 3;
        for (int k = 0; k < 3; k++) {
            v.sp.g[k] = level0_grid(c->L, c->L.nx + (k == 0), c->L.ny + (k == 1), c->L.nz + (k == 2));
            v.sp.base[k] = c->L.face_origin(k) - c->L.PL;
        }
        v.fl = c->fflag;
        if (int rc = make_list<QuadPred>(c, v, quad_items, &c->fq, &c->nfq, c->fq_off))
            return rc == FS_ENOMEM ? set_error(FS_ENOMEM, "list of active face quads") : rc;
        c->fq_epoch = c->mask_epoch;
    }
    *ql = c->fq;
    *n = c->nfq;
    if (off)
        for (int k = 0; k < 4; k++) off[k] = c->fq_off[k];
    return FS_OK;
}

// The pressure hierarchy and its set for the current mask.
static int build_cell(fs_ctx *c, MgAll *m)
{
    const Layout &L = c->L;
    int rc;
    MgSet &t = m->cset;
    free_set(&t);
    if ((rc = coarse_attributes()) || (rc = work_arrays(c, &m->cb, &m->cc, (size_t)L.nC)) ||
        (rc = plan_levels(c, &m->cell, level0_grid(L, L.nx, L.ny, L.nz), 1.f, 0.f)))
        return rc;
    t.nv = 1;
    t.s[0] = &m->cell;
    t.lev[0].fl = c->cflag;
    t.lev[0].b = m->cb;
    t.lev[0].c = m->cc;
    t.lev[0].d = m->cb + L.nC;
    t.shared0 = true;
    const int *ql = nullptr;
    if ((rc = cell_quads(c, &ql, &t.lev[0].nq))) {
        free_set(&t);
        return rc;
    }
    t.lev[0].ql = const_cast<int *>(ql);
    for (int v = 1; v < 4; v++) t.lev[0].qoff[v] = t.lev[0].nq;
    if ((rc = build_set(c, t))) {
        free_set(&t);
        return rc;
    }
    return FS_OK;
}

// The three face hierarchies and their sets for the current mask.
static int build_faces(fs_ctx *c, MgAll *m, float cc)
{
    const Layout &L = c->L;
    int rc;
    for (MgSet &t : m->fset) free_set(&t);
    m->nfset = 0;
    if ((rc = coarse_attributes()) || (rc = work_arrays(c, &m->fb, nullptr, (size_t)L.nF))) return rc;
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
        t.lev[0].d = m->fb + L.nF;
        t.one = true;
        if (all) {  // the context's list; one volume at a time, lists of their own
            const int *ql = nullptr;
            if ((rc = face_quads(c, &ql, &t.lev[0].nq, t.lev[0].qoff))) return rc;
            t.lev[0].ql = const_cast<int *>(ql);
        }
        t.shared0 = all;
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

// The hierarchy of the pressure, or of the face volumes for the operator's
// coefficient cc, for the current mask.
int mg_prepare(fs_ctx *c, bool faces, float cc)
{
    MgAll *m = state(c);
    if (!m) return set_error(FS_ENOMEM, "host allocation failed");
    if (!faces) return m->cell.epoch != c->mask_epoch ? build_cell(c, m) : FS_OK;
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
    return FS_OK;
}

// z = M r on the cell space (r and z of length nC, zero off the liquid); with
// rzs, r.z in the last level-0 sweep when the hierarchy has one (*fused tells)
static int apply_cell(fs_ctx *c, const float *r, float *z, const int *done, SolveScal *rzs, int first, bool *fused)
{
    if (fused) *fused = false;
    int rc = mg_prepare(c, false, 1.f);
    if (rc) return rc;
    MgAll *m = state(c);
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

// z = M r on the face space for the Helmholtz operator I + cc L of the viscosity
// solve (r and z of length nF, zero off the unknown faces), the three velocity
// components' V-cycles launch by launch together. With `done` set, every kernel
// returns at once once *done != 0.
static int apply_faces(fs_ctx *c, const float *r, float *z, float cc, const int *done, SolveScal *rzs, int first,
                       bool *fused)
{
    if (fused) *fused = false;
    if (int rc = mg_prepare(c, true, cc)) return rc;
    MgAll *m = state(c);
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
    return cudaPeekAtLastError() == cudaSuccess;  // (the caller counts the launch)
}

int mg_levels(const fs_ctx *c)
{
    const MgAll *m = static_cast<const MgAll *>(c->mg);
    return m ? m->cell.nlev : 0;
}

}  // namespace fs
