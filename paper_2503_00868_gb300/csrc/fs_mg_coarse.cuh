// fs_mg_coarse.cuh -- the multigrid V-cycle below level 0 (included by fs_mg.cu):
// per level one launch down (both pre-sweeps, the residual, its restriction) and
// one up (prolongation, both post-sweeps), and one single-block launch for the
// levels that fit together in one SM's shared memory. Each launch serves up to
// three volumes (the face components of the viscosity solve) at once.
//
// What bounds them: these levels hold 1/8 of the unknowns of level 0 and less, a
// few MB that stay in L2, so a step of the cycle costs its latency (a launch or a
// barrier, then two dependent L2 round trips), not its bytes. Before, one launch
// of a 16-CTA cluster walked the levels at or below 64^3 with a cluster barrier
// after each of the six steps of a level: up to 101 us below a 128^3 blob (the
// three volumes of the viscosity at once) and 46 below 53 x 44 x 39; these kernels
// take 62 and 20. A block loads a tile with the halo its steps need (three cells
// down, two up), so a level has two dependent global round trips instead of six,
// on all SMs.
//
// Every element gets the same operations in the same order as in the one-step
// kernels of level 0.

// A level as the kernels see it.
struct MgcLevel {
    MgGrid g;
    const uint8_t *fl;
    float *r, *a, *b;  // right-hand side, result, the field between the two legs
    float scale, mass;
};

// Tiles of a level: tqx quads x ty rows x tz planes (ty, tz even, so that a tile
// holds whole 2 x 2 x 2 children of its coarse cells).
struct MgTiles {
    int tqx, ty, tz, ntx, nty, ntz;
    FastDiv dntx, dnty;      // tile index
    FastDiv dq;              // quads of a loaded row (tqx + 2)
    FastDiv dyd, dyu;        // rows of a loaded plane, down (ty + 6) and up (ty + 4)
};

struct MgLegVol {
    MgcLevel f, c;  // the level and the one below it
    MgTiles t;
};
struct MgLegArgs {
    MgLegVol v[3];
    const int *done;
};

constexpr int MGT_TH = 512;     // threads of a tile block
constexpr int MGT_PER_SM = 2;   // resident tile blocks per SM

inline size_t leg_smem(const MgTiles &t, bool down)
{
    const size_t h = down ? 6 : 4;
    const size_t n = (size_t)(t.tqx + 2) * 4 * (t.ty + h) * (t.tz + h);
    const size_t ec = down ? 0 : (size_t)(2 * t.tqx + 6) * (t.ty / 2 + 4) * (t.tz / 2 + 4);
    return 64 + n * 13 + ec * 4;
}

// Tiles of 32 x 8 x 8 cells (102 KB of shared memory on the way down, two blocks
// per SM); a level with fewer such tiles than three quarters of the SMs takes
// 4 x 4 rows instead: more halo per cell, but every SM works and a block's serial
// steps are a third as long.
inline MgTiles make_tiles(const MgGrid &g, int nv, int num_sms)
{
    MgTiles t;
    const int nq = (g.nx + 3) / 4, pieces = (nq + 7) / 8;
    t.tqx = (nq + pieces - 1) / pieces;
    t.ntx = (nq + t.tqx - 1) / t.tqx;
    const long long at8 = (long long)t.ntx * ((g.ny + 7) / 8) * ((g.nz + 7) / 8) * nv;
    t.ty = t.tz = at8 * 4 >= 3LL * num_sms ? 8 : 4;
    t.nty = (g.ny + t.ty - 1) / t.ty;
    t.ntz = (g.nz + t.tz - 1) / t.tz;
    t.dntx = FastDiv(t.ntx);
    t.dnty = FastDiv(t.nty);
    t.dq = FastDiv(t.tqx + 2);
    t.dyd = FastDiv(t.ty + 6);
    t.dyu = FastDiv(t.ty + 4);
    return t;
}

// e_out on one element from e_in: c (centre), the sum of its six neighbours nb
__device__ __forceinline__ float sweep1(uint8_t f, float c, float nb, float rv, const float *wt, float scale, float m)
{
    return liq(f) ? c + wt[f & CF_D] * (rv - m * c - scale * ((float)(f & CF_D) * c - nb)) : 0.f;
}

// omega D^-1 r on a quad
__device__ __forceinline__ float4 jac4(uchar4 f, float4 r, const float *wt)
{
    return make_float4(liq(f.x) ? wt[f.x & CF_D] * r.x : 0.f, liq(f.y) ? wt[f.y & CF_D] * r.y : 0.f,
                       liq(f.z) ? wt[f.z & CF_D] * r.z : 0.f, liq(f.w) ? wt[f.w & CF_D] * r.w : 0.f);
}

// the seven quads around element t of a shared-memory array with row pitch P and
// plane pitch PL: the sums of the six neighbours of each of its four elements
struct Nb4 {
    float4 c, nb;
};
__device__ __forceinline__ Nb4 neighbours(const float *e, int t, int P, int PL)
{
    Nb4 o;
    o.c = *reinterpret_cast<const float4 *>(e + t);
    const float4 dn = *reinterpret_cast<const float4 *>(e + t - P), up = *reinterpret_cast<const float4 *>(e + t + P);
    const float4 bk = *reinterpret_cast<const float4 *>(e + t - PL), fw = *reinterpret_cast<const float4 *>(e + t + PL);
    const float lf = e[t - 1], rt = e[t + 4];
    o.nb.x = (lf + o.c.y) + (dn.x + up.x) + (bk.x + fw.x);
    o.nb.y = (o.c.x + o.c.z) + (dn.y + up.y) + (bk.y + fw.y);
    o.nb.z = (o.c.y + o.c.w) + (dn.z + up.z) + (bk.z + fw.z);
    o.nb.w = (o.c.z + rt) + (dn.w + up.w) + (bk.w + fw.w);
    return o;
}
__device__ __forceinline__ float4 sweep4(uchar4 f, const Nb4 &n, float4 r, const float *wt, float scale, float m)
{
    return make_float4(sweep1(f.x, n.c.x, n.nb.x, r.x, wt, scale, m), sweep1(f.y, n.c.y, n.nb.y, r.y, wt, scale, m),
                       sweep1(f.z, n.c.z, n.nb.z, r.z, wt, scale, m), sweep1(f.w, n.c.w, n.nb.w, r.w, wt, scale, m));
}
__device__ __forceinline__ float4 resid4(uchar4 f, const Nb4 &n, float4 r, float scale, float m)
{
    auto one = [&](uint8_t fe, float ce, float nb, float re) {
        return liq(fe) ? re - m * ce - scale * ((float)(fe & CF_D) * ce - nb) : 0.f;
    };
    return make_float4(one(f.x, n.c.x, n.nb.x, r.x), one(f.y, n.c.y, n.nb.y, r.y), one(f.z, n.c.z, n.nb.z, r.z),
                       one(f.w, n.c.w, n.nb.w, r.w));
}

// restriction of the coarse pair whose fine quad is element t of a shared-memory
// residual (row 2J, plane 2K); zeros stand off the grid and off the unknowns
__device__ __forceinline__ void restrict_smem(const float *res, int t, int P, int PL, float &a0, float &a1)
{
    const float w[4] = {0.25f, 0.75f, 0.75f, 0.25f};
    a0 = a1 = 0.f;
#pragma unroll
    for (int c = 0; c < 4; c++)
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const int row = t + (c - 1) * PL + (b - 1) * P;
            const float4 qd = *reinterpret_cast<const float4 *>(res + row);
            const float lf = res[row - 1], rt = res[row + 4];
            const float wyz = w[c] * w[b];
            a0 += wyz * (0.25f * lf + 0.75f * qd.x + 0.75f * qd.y + 0.25f * qd.z);
            a1 += wyz * (0.25f * qd.y + 0.75f * qd.z + 0.75f * qd.w + 0.25f * rt);
        }
}

// the prolongation of a coarse field onto the quad of cells (i .. i + 3, j, k), i a
// multiple of 4: element t of `ec` is coarse cell (i/2, j/2, k/2)
__device__ __forceinline__ float4 prolong4(const float *ec, int t, int j, int k, int P, int PL)
{
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    const int oy[2] = {0, (j & 1) ? P : -P}, oz[2] = {0, (k & 1) ? PL : -PL};
    const float wy[2] = {0.75f, 0.25f};
#pragma unroll
    for (int b = 0; b < 2; b++)
#pragma unroll
        for (int a = 0; a < 2; a++) {
            const float *row = ec + t + oy[a] + oz[b];
            const float w = wy[a] * wy[b];
            const float cm = row[-1], c0 = row[0], c1 = row[1], c2 = row[2];
            s.x += w * (0.75f * c0 + 0.25f * cm);
            s.y += w * (0.75f * c0 + 0.25f * c1);
            s.z += w * (0.75f * c1 + 0.25f * c0);
            s.w += w * (0.75f * c1 + 0.25f * c2);
        }
    return s;
}

__device__ __forceinline__ float4 add_on(uchar4 f, float4 v, float4 s)
{
    if (liq(f.x)) v.x += s.x;
    if (liq(f.y)) v.y += s.y;
    if (liq(f.z)) v.z += s.z;
    if (liq(f.w)) v.w += s.w;
    return v;
}

// the tile of this block: its first quad, row and plane; false past the last
__device__ __forceinline__ bool leg_tile(const MgTiles &T, int &q0, int &j0, int &k0)
{
    if ((int)blockIdx.x >= T.ntx * T.nty * T.ntz) return false;
    unsigned row, tx, ty, tz;
    T.dntx.split(blockIdx.x, row, tx);
    T.dnty.split(row, tz, ty);
    q0 = (int)tx * T.tqx;
    j0 = (int)ty * T.ty;
    k0 = (int)tz * T.tz;
    return true;
}

// Down one level: b = two sweeps from zero on r, and the coarse right-hand side =
// the restriction of r - A b. A tile without an unknown returns after its flags.
__global__ void __launch_bounds__(MGT_TH, 2) k_mg_down(const __grid_constant__ MgLegArgs a)
{
    extern __shared__ __align__(16) float mg_sm[];
    __shared__ float wt[8];
    const MgLegVol &V = a.v[blockIdx.y];
    const MgTiles &T = V.t;
    const MgcLevel &L = V.f;
    int q0, j0, k0;
    const bool mine = leg_tile(T, q0, j0, k0);
    dep_wait();
    dep_go();
    if (!mine || (a.done && *(volatile const int *)a.done)) return;  // (or the solve has converged)
    if (threadIdx.x < 8) wt[threadIdx.x] = wtab_entry(L.scale, L.mass, threadIdx.x);
    const int nq = T.tqx + 2, ny = T.ty + 6, nz = T.tz + 6;
    const int P = nq * 4, PL = P * ny, n = PL * nz;
    float *R = mg_sm + 4, *E1 = R + n, *E2 = E1 + n;
    uint8_t *FL = reinterpret_cast<uint8_t *>(E2 + n + 4);
    const int nx_ = L.g.nx, ny_ = L.g.ny, nz_ = L.g.nz;
    bool any = false;
    for (int s = threadIdx.x; s < (n >> 2); s += MGT_TH) {
        unsigned row, qx, y, z;
        T.dq.split(s, row, qx);
        T.dyd.split(row, z, y);
        const int i = 4 * (q0 + (int)qx - 1), j = j0 + (int)y - 3, k = k0 + (int)z - 3;
        uchar4 f = make_uchar4(0, 0, 0, 0);
        float4 rv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i >= 0 && i < nx_ && j >= 0 && j < ny_ && k >= 0 && k < nz_) {
            const int t = L.g.idx(i, j, k);
            f = ldf4(L.fl, t);
            rv = ldv4(L.r, t);
            any |= any_liq(f) && qx >= 1 && (int)qx <= T.tqx && y >= 3 && (int)y < T.ty + 3 && z >= 3 &&
                   (int)z < T.tz + 3;
        }
        *reinterpret_cast<float4 *>(R + 4 * s) = rv;
        *reinterpret_cast<uchar4 *>(FL + 4 * s) = f;
    }
    if (!__syncthreads_or(any)) return;
    for (int s = threadIdx.x; s < (n >> 2); s += MGT_TH)
        *reinterpret_cast<float4 *>(E1 + 4 * s) =
            jac4(*reinterpret_cast<const uchar4 *>(FL + 4 * s), *reinterpret_cast<const float4 *>(R + 4 * s), wt);
    __syncthreads();
    // the second sweep on the tile and two cells around it
    for (int s = threadIdx.x; s < nq * ny * (nz - 2); s += MGT_TH) {
        unsigned row, qx, y, z;
        T.dq.split(s, row, qx);
        T.dyd.split(row, z, y);
        z += 1;
        if (y < 1 || (int)y > ny - 2) continue;
        const int t = (int)z * PL + (int)y * P + 4 * (int)qx;
        const uchar4 f = *reinterpret_cast<const uchar4 *>(FL + t);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (any_liq(f)) {
            v = sweep4(f, neighbours(E1, t, P, PL), *reinterpret_cast<const float4 *>(R + t), wt, L.scale, L.mass);
            if (qx >= 1 && (int)qx <= T.tqx && y >= 3 && (int)y < T.ty + 3 && z >= 3 && (int)z < T.tz + 3)
                *reinterpret_cast<float4 *>(
                    L.b + L.g.idx(4 * (q0 + (int)qx - 1), j0 + (int)y - 3, k0 + (int)z - 3)) = v;
        }
        *reinterpret_cast<float4 *>(E2 + t) = v;
    }
    __syncthreads();
    // the residual on the tile and one cell around it, over e1
    for (int s = threadIdx.x; s < nq * ny * (nz - 4); s += MGT_TH) {
        unsigned row, qx, y, z;
        T.dq.split(s, row, qx);
        T.dyd.split(row, z, y);
        z += 2;
        if (y < 2 || (int)y > ny - 3) continue;
        const int t = (int)z * PL + (int)y * P + 4 * (int)qx;
        const uchar4 f = *reinterpret_cast<const uchar4 *>(FL + t);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (any_liq(f))
            v = resid4(f, neighbours(E2, t, P, PL), *reinterpret_cast<const float4 *>(R + t), L.scale, L.mass);
        *reinterpret_cast<float4 *>(E1 + t) = v;
    }
    __syncthreads();
    const MgcLevel &W = V.c;
    for (int s = threadIdx.x; s < T.tqx * (T.ty / 2) * (T.tz / 2); s += MGT_TH) {
        const int m = s % T.tqx, J = (s / T.tqx) % (T.ty / 2), K = s / (T.tqx * (T.ty / 2));
        const int I0 = 2 * (q0 + m), Jg = j0 / 2 + J, Kg = k0 / 2 + K;
        if (I0 >= W.g.nx || Jg >= W.g.ny || Kg >= W.g.nz) continue;
        const int t0 = W.g.idx(I0, Jg, Kg);
        const bool l0 = liq(W.fl[t0]), l1 = I0 + 1 < W.g.nx && liq(W.fl[t0 + 1]);
        if (!l0 && !l1) continue;
        float a0, a1;
        restrict_smem(E1, (2 * K + 3) * PL + (2 * J + 3) * P + 4 * (m + 1), P, PL, a0, a1);
        if (l0) W.r[t0] = 0.125f * a0;
        if (l1) W.r[t0 + 1] = 0.125f * a1;
    }
}

// Up one level: the coarse result prolonged onto b, then two sweeps, into a.
__global__ void __launch_bounds__(MGT_TH, 2) k_mg_up(const __grid_constant__ MgLegArgs a)
{
    extern __shared__ __align__(16) float mg_sm[];
    __shared__ float wt[8];
    const MgLegVol &V = a.v[blockIdx.y];
    const MgTiles &T = V.t;
    const MgcLevel &L = V.f, &W = V.c;
    int q0, j0, k0;
    const bool mine = leg_tile(T, q0, j0, k0);
    dep_wait();
    dep_go();
    if (!mine || (a.done && *(volatile const int *)a.done)) return;  // (or the solve has converged)
    if (threadIdx.x < 8) wt[threadIdx.x] = wtab_entry(L.scale, L.mass, threadIdx.x);
    const int nq = T.tqx + 2, ny = T.ty + 4, nz = T.tz + 4;
    const int P = nq * 4, PL = P * ny, n = PL * nz;
    const int CP = 2 * T.tqx + 6, CPL = CP * (T.ty / 2 + 4), cn = CPL * (T.tz / 2 + 4);
    float *R = mg_sm + 4, *E = R + n, *S = E + n, *EC = S + n + 4;
    uint8_t *FL = reinterpret_cast<uint8_t *>(EC + cn);
    const int nx_ = L.g.nx, ny_ = L.g.ny, nz_ = L.g.nz;
    bool any = false;
    for (int s = threadIdx.x; s < (n >> 2); s += MGT_TH) {
        unsigned row, qx, y, z;
        T.dq.split(s, row, qx);
        T.dyu.split(row, z, y);
        const int i = 4 * (q0 + (int)qx - 1), j = j0 + (int)y - 2, k = k0 + (int)z - 2;
        uchar4 f = make_uchar4(0, 0, 0, 0);
        float4 rv = make_float4(0.f, 0.f, 0.f, 0.f), bv = rv;
        if (i >= 0 && i < nx_ && j >= 0 && j < ny_ && k >= 0 && k < nz_) {
            const int t = L.g.idx(i, j, k);
            f = ldf4(L.fl, t);
            rv = ldv4(L.r, t);
            bv = ldv4(L.b, t);
            any |= any_liq(f) && qx >= 1 && (int)qx <= T.tqx && y >= 2 && (int)y < T.ty + 2 && z >= 2 &&
                   (int)z < T.tz + 2;
        }
        *reinterpret_cast<float4 *>(R + 4 * s) = rv;
        *reinterpret_cast<float4 *>(E + 4 * s) = bv;
        *reinterpret_cast<uchar4 *>(FL + 4 * s) = f;
    }
    // the coarse cells that the loaded quads sample: from (2 q0 - 3, j0/2 - 2, k0/2 - 2)
    for (int s = threadIdx.x; s < cn; s += MGT_TH) {
        const int x = s % CP, y = (s / CP) % (T.ty / 2 + 4), z = s / CPL;
        const int I = 2 * q0 - 3 + x, J = j0 / 2 - 2 + y, K = k0 / 2 - 2 + z;
        EC[s] = I >= 0 && J >= 0 && K >= 0 && I < W.g.nx && J < W.g.ny && K < W.g.nz ? ldd1(W.a + W.g.idx(I, J, K))
                                                                                      : 0.f;
    }
    if (!__syncthreads_or(any)) return;
    for (int s = threadIdx.x; s < (n >> 2); s += MGT_TH) {
        const uchar4 f = *reinterpret_cast<const uchar4 *>(FL + 4 * s);
        if (!any_liq(f)) continue;
        unsigned row, qx, y, z;
        T.dq.split(s, row, qx);
        T.dyu.split(row, z, y);
        const int ct = ((int)z / 2 + 1) * CPL + ((int)y / 2 + 1) * CP + 2 * (int)qx + 1;
        const float4 p = prolong4(EC, ct, (int)y, (int)z, CP, CPL);  // j0, k0 and the halo are even
        float4 *e = reinterpret_cast<float4 *>(E + 4 * s);
        *e = add_on(f, *e, p);
    }
    __syncthreads();
    for (int s = threadIdx.x; s < nq * ny * (nz - 2); s += MGT_TH) {
        unsigned row, qx, y, z;
        T.dq.split(s, row, qx);
        T.dyu.split(row, z, y);
        z += 1;
        if (y < 1 || (int)y > ny - 2) continue;
        const int t = (int)z * PL + (int)y * P + 4 * (int)qx;
        const uchar4 f = *reinterpret_cast<const uchar4 *>(FL + t);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (any_liq(f))
            v = sweep4(f, neighbours(E, t, P, PL), *reinterpret_cast<const float4 *>(R + t), wt, L.scale, L.mass);
        *reinterpret_cast<float4 *>(S + t) = v;
    }
    __syncthreads();
    for (int s = threadIdx.x; s < nq * ny * (nz - 4); s += MGT_TH) {
        unsigned row, qx, y, z;
        T.dq.split(s, row, qx);
        T.dyu.split(row, z, y);
        z += 2;
        if (y < 2 || (int)y > ny - 3 || qx < 1 || (int)qx > T.tqx) continue;
        const int t = (int)z * PL + (int)y * P + 4 * (int)qx;
        const uchar4 f = *reinterpret_cast<const uchar4 *>(FL + t);
        if (!any_liq(f)) continue;
        *reinterpret_cast<float4 *>(L.a + L.g.idx(4 * (q0 + (int)qx - 1), j0 + (int)y - 2, k0 + (int)z - 2)) =
            sweep4(f, neighbours(S, t, P, PL), *reinterpret_cast<const float4 *>(R + t), wt, L.scale, L.mass);
    }
}

// ---- the levels that fit in one SM's shared memory ------------------------------
// One block per volume: the same V-cycle with every array of its levels in shared
// memory (three of floats) and a block barrier between steps. What does not change
// with the mask comes as one blob, copied to shared memory beside the arrays: the
// flags and the active quads of every level. The MG_COARSE_SWEEPS damped Jacobi
// sweeps of the coarsest level keep each thread's quad, its flags and right-hand
// side in registers. What bounds it is one SM's shared-memory bandwidth and the
// latency of a barrier and a chain of loads and sums per step (130 cycles for one
// warp): a sweep over the 326 unknowns of a 9^3 level took 480 cycles with three
// cells of one float per thread, lists in the order of an atomic counter and the
// geometry read from the kernel's parameters by dynamic index (18.5 us in all for
// 17^3 and 9^3 levels).
constexpr int MGB_TH = 1024;
constexpr int MGB_MAXLEV = 8;
constexpr size_t MGB_SMEM = 216 * 1024;
constexpr int MGB_HEAD = 64;  // bytes of the blob's counts
static_assert(MG_COARSE_CELLS / 4 <= MGB_TH, "one quad of the coarsest level per thread");

struct MgBottomLevel {
    MgcLevel l;
    int off;               // first float of R, B and C (n floats each)
    int foff, qoff;        // first byte of the flags and of the list in the blob
    FastDiv dsy, dsz;      // elements of a row and of a plane
};
struct MgBottomVol {
    MgBottomLevel lev[MGB_MAXLEV];
    int nlev;
    int n;                 // elements of all levels
    int bytes;             // of the blob, a multiple of 16
    uint8_t *blob;         // counts [MGB_MAXLEV] of int, flags, lists of uint16
};
struct MgBottomArgs {
    MgBottomVol v[3];
    const int *done;
};

// blob of levels of n elements in all, and the shared memory
inline size_t bottom_blob(size_t n) { return (MGB_HEAD + n + n / 2 + 15) / 16 * 16; }
inline size_t bottom_smem(size_t n) { return 32 + n * 12 + bottom_blob(n); }

// Fills the blobs (once per mask), the lists in ascending order, so that the lanes
// of a warp read neighbouring words.
__global__ void __launch_bounds__(MGB_TH, 1) k_mg_bottom_lists(const __grid_constant__ MgBottomArgs a)
{
    __shared__ int part[MGB_TH / 32];
    const MgBottomVol &V = a.v[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < MGB_MAXLEV) reinterpret_cast<int *>(V.blob)[tid] = 0;
    __syncthreads();
    for (int l = 0; l < V.nlev; l++) {
        const MgBottomLevel &b = V.lev[l];
        const int n = b.l.g.n, items = n >> 2;
        for (int t = tid; t < n; t += MGB_TH) V.blob[b.foff + t] = b.l.fl[t];
        unsigned short *list = reinterpret_cast<unsigned short *>(V.blob + b.qoff);
        int total = 0;
        for (int t0 = 0; t0 < items; t0 += MGB_TH) {
            const int t = t0 + tid;
            const bool u = t < items && any_liq(ldf4(b.l.fl, 4 * t));
            const unsigned mask = __ballot_sync(0xffffffffu, u);
            if (lane == 0) part[warp] = __popc(mask);
            __syncthreads();
            int at = total + __popc(mask & ((1u << lane) - 1u));
            for (int w = 0; w < MGB_TH / 32; w++) {
                if (w < warp) at += part[w];
                total += part[w];
            }
            if (u) list[at] = (unsigned short)t;
            __syncthreads();
        }
        if (tid == 0) reinterpret_cast<int *>(V.blob)[l] = total;
    }
}

// a barrier of the block's first `threads` threads (a multiple of 32)
__device__ __forceinline__ void bar_some(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }

__global__ void __launch_bounds__(MGB_TH, 1) k_mg_bottom(const __grid_constant__ MgBottomArgs a)
{
    dep_wait();
    dep_go();
    if (a.done && *(volatile const int *)a.done) return;  // the solve has converged
    extern __shared__ __align__(16) float mg_sm[];
    __shared__ float wts[MGB_MAXLEV][8];
    __shared__ MgBottomVol V;
    const int tid = threadIdx.x;
    for (int t = tid; t < (int)(sizeof(MgBottomVol) / 4); t += MGB_TH)
        reinterpret_cast<int *>(&V)[t] = reinterpret_cast<const int *>(&a.v[blockIdx.x])[t];
    const int n = a.v[blockIdx.x].n, n0 = a.v[blockIdx.x].lev[0].l.g.n >> 2, nl = a.v[blockIdx.x].nlev;
    float *F0 = mg_sm + 4;
    uint8_t *G0 = reinterpret_cast<uint8_t *>(F0 + 3 * n + 4);
    {
        const int words = a.v[blockIdx.x].bytes >> 4;
        const uint4 *src = reinterpret_cast<const uint4 *>(a.v[blockIdx.x].blob);
        const float *r = a.v[blockIdx.x].lev[0].l.r;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 *A = reinterpret_cast<float4 *>(F0);
        for (int t = tid; t < words; t += MGB_TH) reinterpret_cast<uint4 *>(G0)[t] = __ldg(src + t);
        for (int t = tid; t < n0; t += MGB_TH) A[t] = ldv4(r, 4 * t);
        for (int t = n0 + tid; t < (3 * n) >> 2; t += MGB_TH) A[t] = zero;
    }
    __syncthreads();
    if (tid < MGB_MAXLEV * 8 && tid / 8 < nl)
        wts[tid / 8][tid % 8] = wtab_entry(V.lev[tid / 8].l.scale, V.lev[tid / 8].l.mass, tid % 8);
    __syncthreads();
    const int *count = reinterpret_cast<const int *>(G0);
    for (int l = 0; l + 1 < nl; l++) {
        const MgGrid g = V.lev[l].l.g;
        const float scale = V.lev[l].l.scale, m = V.lev[l].l.mass, *wt = wts[l];
        float *R = F0 + V.lev[l].off, *B = R + g.n, *C = B + g.n;
        const uint8_t *FL = G0 + V.lev[l].foff;
        const unsigned short *ql = reinterpret_cast<const unsigned short *>(G0 + V.lev[l].qoff);
        const int quads = count[l];
        for (int s = tid; s < quads; s += MGB_TH) {
            const int t = 4 * ql[s];
            *reinterpret_cast<float4 *>(C + t) =
                jac4(*reinterpret_cast<const uchar4 *>(FL + t), *reinterpret_cast<const float4 *>(R + t), wt);
        }
        __syncthreads();
        for (int s = tid; s < quads; s += MGB_TH) {
            const int t = 4 * ql[s];
            *reinterpret_cast<float4 *>(B + t) =
                sweep4(*reinterpret_cast<const uchar4 *>(FL + t), neighbours(C, t, g.sy, g.sz),
                       *reinterpret_cast<const float4 *>(R + t), wt, scale, m);
        }
        __syncthreads();
        for (int s = tid; s < quads; s += MGB_TH) {
            const int t = 4 * ql[s];
            *reinterpret_cast<float4 *>(C + t) =
                resid4(*reinterpret_cast<const uchar4 *>(FL + t), neighbours(B, t, g.sy, g.sz),
                       *reinterpret_cast<const float4 *>(R + t), scale, m);
        }
        __syncthreads();
        // one thread per coarse pair, which is one fine quad of the even rows; a row
        // off the grid has weight zero and the pair's own row in its place
        const MgGrid gc = V.lev[l + 1].l.g;
        float *Rc = F0 + V.lev[l + 1].off;
        const uint8_t *FC = G0 + V.lev[l + 1].foff;
        const int np = (gc.nx + 1) >> 1;
        const float wg[4] = {0.25f, 0.75f, 0.75f, 0.25f};
        for (int s = tid; s < np * gc.ny * gc.nz; s += MGB_TH) {
            const int mm = s % np, J = (s / np) % gc.ny, K = s / (np * gc.ny);
            const int t0 = gc.idx(2 * mm, J, K);
            const bool l0 = liq(FC[t0]), l1 = 2 * mm + 1 < gc.nx && liq(FC[t0 + 1]);
            if (!l0 && !l1) continue;
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int c = 0; c < 4; c++)
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    const int k = 2 * K - 1 + c, j = 2 * J - 1 + r;  // (-1 is the halo)
                    const bool in = k < g.nz && j < g.ny;
                    const int row = g.idx(4 * mm, in ? j : 2 * J, in ? k : 2 * K);
                    const float4 qd = *reinterpret_cast<const float4 *>(C + row);
                    const float lf = C[row - 1], rt = C[row + 4];
                    const float wyz = in ? wg[c] * wg[r] : 0.f;
                    a0 += wyz * (0.25f * lf + 0.75f * qd.x + 0.75f * qd.y + 0.25f * qd.z);
                    a1 += wyz * (0.25f * qd.y + 0.75f * qd.z + 0.75f * qd.w + 0.25f * rt);
                }
            if (l0) Rc[t0] = 0.125f * a0;
            if (l1) Rc[t0 + 1] = 0.125f * a1;
        }
        __syncthreads();
    }
    {  // the coarsest level: result in e0 (or in global memory when it is the only one)
        const MgGrid g = V.lev[nl - 1].l.g;
        const float scale = V.lev[nl - 1].l.scale, m = V.lev[nl - 1].l.mass;
        float *R = F0 + V.lev[nl - 1].off, *e0 = R + g.n, *e1 = e0 + g.n;
        // only the warps that hold an unknown take part in a sweep
        const int nc = count[nl - 1], nthr = (nc + 31) & ~31;
        if (tid < nthr) {
            const bool on = tid < nc;
            const int t = on ? 4 * reinterpret_cast<const unsigned short *>(G0 + V.lev[nl - 1].qoff)[tid] : 0;
            const uchar4 f = *reinterpret_cast<const uchar4 *>(G0 + V.lev[nl - 1].foff + t);
            const float4 r = *reinterpret_cast<const float4 *>(R + t);
            const float *wt = wts[nl - 1];
            const float4 w = make_float4(wt[f.x & CF_D], wt[f.y & CF_D], wt[f.z & CF_D], wt[f.w & CF_D]);
            Nb4 e;
            e.c = jac4(f, r, wt);
            if (on) *reinterpret_cast<float4 *>(e0 + t) = e.c;
            bar_some(nthr);
            auto one = [&](uint8_t fe, float c, float nb, float rv, float we) {
                return liq(fe) ? c + we * (rv - m * c - scale * ((float)(fe & CF_D) * c - nb)) : 0.f;
            };
            auto sweep = [&](const float *ein, float *eout) {
                if (on) {
                    e = neighbours(ein, t, g.sy, g.sz);
                    e.c = make_float4(one(f.x, e.c.x, e.nb.x, r.x, w.x), one(f.y, e.c.y, e.nb.y, r.y, w.y),
                                      one(f.z, e.c.z, e.nb.z, r.z, w.z), one(f.w, e.c.w, e.nb.w, r.w, w.w));
                    *reinterpret_cast<float4 *>(eout + t) = e.c;
                }
                bar_some(nthr);
            };
            static_assert(MG_COARSE_SWEEPS % 2 == 0, "the first sweep is in e0, the last one in e1");
            for (int s = 1; s + 1 < MG_COARSE_SWEEPS; s += 2) {
                sweep(e0, e1);
                sweep(e1, e0);
            }
            sweep(e0, e1);
            if (on) *reinterpret_cast<float4 *>(e0 + t) = e.c;
        }
        __syncthreads();
        if (nl == 1)
            for (int t = tid; t < g.n; t += MGB_TH) V.lev[0].l.a[t] = e0[t];
    }
    for (int l = nl - 2; l >= 0; l--) {
        const MgGrid g = V.lev[l].l.g, gc = V.lev[l + 1].l.g;
        const float scale = V.lev[l].l.scale, m = V.lev[l].l.mass, *wt = wts[l];
        float *R = F0 + V.lev[l].off, *B = R + g.n, *C = B + g.n;
        const float *EC = F0 + V.lev[l + 1].off + gc.n;
        const uint8_t *FL = G0 + V.lev[l].foff;
        const unsigned short *ql = reinterpret_cast<const unsigned short *>(G0 + V.lev[l].qoff);
        const FastDiv dsy = V.lev[l].dsy, dsz = V.lev[l].dsz;
        const int quads = count[l];
        for (int s = tid; s < quads; s += MGB_TH) {
            const int t = 4 * ql[s];
            const uchar4 f = *reinterpret_cast<const uchar4 *>(FL + t);
            unsigned row, x, y, z;
            dsz.split(t, z, row);
            dsy.split(row, y, x);
            const int i = (int)x - g.ioff, j = (int)y - g.joff, k = (int)z - g.koff;
            float4 *e = reinterpret_cast<float4 *>(B + t);
            *e = add_on(f, *e, prolong4(EC, gc.idx(i >> 1, j >> 1, k >> 1), j, k, gc.sy, gc.sz));
        }
        __syncthreads();
        for (int s = tid; s < quads; s += MGB_TH) {
            const int t = 4 * ql[s];
            *reinterpret_cast<float4 *>(C + t) =
                sweep4(*reinterpret_cast<const uchar4 *>(FL + t), neighbours(B, t, g.sy, g.sz),
                       *reinterpret_cast<const float4 *>(R + t), wt, scale, m);
        }
        __syncthreads();
        float *out = l == 0 ? V.lev[0].l.a : B;
        for (int s = tid; s < quads; s += MGB_TH) {
            const int t = 4 * ql[s];
            *reinterpret_cast<float4 *>(out + t) =
                sweep4(*reinterpret_cast<const uchar4 *>(FL + t), neighbours(C, t, g.sy, g.sz),
                       *reinterpret_cast<const float4 *>(R + t), wt, scale, m);
        }
        __syncthreads();
    }
}
