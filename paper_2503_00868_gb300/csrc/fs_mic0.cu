// fs_mic0.cu -- MIC(0) preconditioner of the pressure solve (the modified
// incomplete Cholesky of Bridson's "Fluid Simulation for Computer Graphics",
// which the paper cites for its pressure projection, Sec. 3.2.2): factor, forward
// and backward substitution in LEXICOGRAPHIC order (x fastest), exactly the
// recurrences of the sequential algorithm, run as a tile wavefront.
//
// Recurrences (A = 7-point pressure operator, -1 between liquid neighbours,
// prec = 1/sqrt(e), "lower" = the -x, -y, -z neighbours that are liquid):
//   factor:   e_i = d_i - sum_lower prec_m^2 (1 + tau * n_m),  n_m = number of
//             liquid +neighbours of m in the other two directions;
//             e_i < sigma d_i  =>  e_i = d_i
//   forward:  y_i = prec_i (r_i + sum_lower prec_m y_m)
//   backward: z_i = prec_i (y_i + prec_i sum_upper z_m)
//
// Schedule. The grid is cut into 8x8x8 tiles; a tile depends on its -x, -y, -z
// neighbour tiles (forward, factor) or its +x, +y, +z neighbours (backward).
// Tiles holding liquid are listed by tile level (tx + ty + tz). Persistent blocks
// take the next tile from an atomic counter, so every predecessor of a tile was
// taken earlier by a block that is already running: waiting on it always ends.
// A block waits (bounded spin) until each predecessor's flag reaches this
// sweep's epoch, has the tile and its one-cell halo in shared memory, walks the 22
// intra-tile diagonal levels (x + y + z = const), writes the tile, and publishes its
// flag. A spin that runs out sets an
// error word; every other wait sees it and gives up, so the launch always ends.
// Values that other blocks of the same launch wrote (halo cells of predecessor
// tiles) are read through L2 (ld.global.cg), never from a possibly stale L1 line.
#include <algorithm>
#include <vector>

#include "fs_internal.cuh"

namespace fs {
namespace {

constexpr int MT = 8;                  // tile edge
constexpr int MTH = MT * MT * MT;      // threads per block of the factorisation, one per cell
enum { MIC_FORWARD = 1, MIC_BACKWARD = 2 };

struct MicGrid {
    int ntx, nty, ntz;
    int nx, ny, nz;
    int P, PL;      // layout pitch and plane
    int origin;     // cell-space offset of cell (0, 0, 0)
};

__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(int *p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ bool liquid(const uint8_t *cf, int t) { return (cf[t] & CF_LIQ) != 0; }

// Waits until predecessor tile a (0..2: along x, y, z; DIR -1 the lower, 1 the upper
// one) of tile (ti, tj, tk) has published this sweep's epoch. False when the wait ran
// out, or another one did. No sleep between the polls: each is an L2 round trip.
template <int DIR>
__device__ __forceinline__ bool wait_tile(const MicGrid &G, int ti, int tj, int tk, int a,
                                          const uint8_t *__restrict__ tact, const int *tflag, int epoch,
                                          int spin_limit, unsigned *err)
{
    const int pi = ti + (a == 0 ? DIR : 0), pj = tj + (a == 1 ? DIR : 0), pk = tk + (a == 2 ? DIR : 0);
    if (pi < 0 || pj < 0 || pk < 0 || pi >= G.ntx || pj >= G.nty || pk >= G.ntz) return true;
    const int pt = (pk * G.nty + pj) * G.ntx + pi;
    if (!tact[pt]) return true;
    int spins = 0;
    while (ld_acquire(tflag + pt) < epoch) {
        if (++spins > spin_limit || ((spins & 15) == 1 && ld_acquire(reinterpret_cast<const int *>(err)) != 0)) {
            atomicOr(err, 1u);
            return false;
        }
    }
    return true;
}

__global__ void __launch_bounds__(MTH) k_mic_factor(MicGrid G, const uint8_t *__restrict__ cf, float *prec,
                                                    const int *__restrict__ order, int n,
                                                    const uint8_t *__restrict__ tact, int *tflag, int *next, int epoch,
                                                    int spin_limit, unsigned *err, float tau, float sigma)
{
    // prec of the tile with a one-cell lower halo: cell (x, y, z) at [z+1][y+1][x+1]
    __shared__ float sp[MT + 1][MT + 1][MT + 1];
    __shared__ int s_tile;
    __shared__ int s_abort;
    const int tid = threadIdx.x;
    const int x = tid % MT, y = (tid / MT) % MT, z = tid / (MT * MT);
    for (;;) {
        if (tid == 0) {
            const int w = atomicAdd(next, 1);
            s_tile = w < n ? order[w] : -1;
            s_abort = 0;
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int ti = tile % G.ntx, tj = (tile / G.ntx) % G.nty, tk = tile / (G.ntx * G.nty);
        if (tid < 3 && !wait_tile<-1>(G, ti, tj, tk, tid, tact, tflag, epoch, spin_limit, err)) s_abort = 1;
        __syncthreads();
        if (s_abort) {
            // give up on this sweep: publish nothing, drain the remaining tiles
            __syncthreads();
            continue;
        }
        const int gi = ti * MT + x, gj = tj * MT + y, gk = tk * MT + z;
        const bool valid = gi < G.nx && gj < G.ny && gk < G.nz;
        const int t = G.origin + gk * G.PL + gj * G.P + gi;
        const bool liq = valid && liquid(cf, t);
        sp[z + 1][y + 1][x + 1] = 0.f;
        // lower faces: x = -1, y = -1, z = -1 (cells outside the grid read as non-liquid)
        if (x == 0) {
            const bool ok = gi - 1 >= 0 && gj < G.ny && gk < G.nz && liquid(cf, t - 1);
            sp[z + 1][y + 1][0] = ok ? __ldcg(prec + (t - 1)) : 0.f;
        }
        if (y == 0) {
            const bool ok = gj - 1 >= 0 && gi < G.nx && gk < G.nz && liquid(cf, t - G.P);
            sp[z + 1][0][x + 1] = ok ? __ldcg(prec + (t - G.P)) : 0.f;
        }
        if (z == 0) {
            const bool ok = gk - 1 >= 0 && gi < G.nx && gj < G.ny && liquid(cf, t - G.PL);
            sp[0][y + 1][x + 1] = ok ? __ldcg(prec + (t - G.PL)) : 0.f;
        }
        float diag = 0.f;
        int nlow = 0;  // bit mask of liquid lower neighbours
        if (liq) {
            diag = (float)(cf[t] & CF_D);
            const int off[3] = {1, G.P, G.PL};
            const int pos[3] = {gi, gj, gk};
            for (int a = 0; a < 3; a++) {
                if (pos[a] > 0 && liquid(cf, t - off[a])) nlow |= 1 << a;
            }
        }
        __syncthreads();
        // the 22 diagonal levels of the tile
        const int lvl = x + y + z;
        for (int l = 0; l <= 3 * (MT - 1); l++) {
            if (lvl == l && liq) {
                float e = diag;
                const int off[3] = {1, G.P, G.PL};
                for (int a = 0; a < 3; a++) {
                    if (!(nlow & (1 << a))) continue;
                    const float pm = a == 0 ? sp[z + 1][y + 1][x] : (a == 1 ? sp[z + 1][y][x + 1] : sp[z][y + 1][x + 1]);
                    // n_m: liquid +neighbours of m in the other two directions
                    const int m = t - off[a];
                    int nm = 0;
                    for (int b = 0; b < 3; b++) {
                        if (b == a) continue;
                        const int mp[3] = {gi - (a == 0), gj - (a == 1), gk - (a == 2)};
                        const int qb = (b == 0 ? mp[0] : (b == 1 ? mp[1] : mp[2])) + 1;
                        if (qb < (b == 0 ? G.nx : (b == 1 ? G.ny : G.nz)) && liquid(cf, m + off[b])) nm++;
                    }
                    e -= pm * pm * (1.f + tau * (float)nm);
                }
                if (e < sigma * diag) e = diag;
                sp[z + 1][y + 1][x + 1] = diag > 0.f ? 1.f / sqrtf(e) : 0.f;
            }
            __syncthreads();
        }
        if (valid) prec[t] = liq ? sp[z + 1][y + 1][x + 1] : 0.f;
        __threadfence();
        __syncthreads();
        if (tid == 0) st_release(tflag + tile, epoch);
    }
}


// Forward or backward substitution. Its time is a chain: a small grid has few tiles
// on a wavefront, and tile after tile must see its predecessors' flags, read their
// faces, walk its diagonals and publish. So what does not depend on them (the tile's
// own values, and the flags and prec of its halo) is loaded before the wait, and one
// warp walks the 22 diagonals in registers: lane (x, y) owns the columns y and y + 4
// along z, its x and y predecessors are the values that other lanes formed a step
// before (shuffles), its z predecessor its own. With a thread per cell, a block
// barrier per diagonal and the loads after the wait, a sweep over 32^3 (ten tiles in
// a row) took 55 us forward and 47 backward; it takes 41 and 39. The backward sweep is the same walk in
// mirrored coordinates.
constexpr int MSTH = 128;          // threads: one per quad of the tile
constexpr int MPY = 40, MPZ = 384; // pitches of the padded tile: a warp's 32 cells lie in 32 banks
template <int MODE>
__global__ void __launch_bounds__(MSTH) k_mic_solve(MicGrid G, const uint8_t *__restrict__ cf,
                                                    const float *__restrict__ prec, const float *in,
                                                    float *out, const int *__restrict__ order, int n,
                                                    const uint8_t *__restrict__ tact, int *tflag, int *next, int *other,
                                                    int epoch, int spin_limit, unsigned *err)
{
    constexpr bool FWD = MODE == MIC_FORWARD;
    constexpr int DIR = FWD ? -1 : 1;
    // in the walk's coordinates: prec with its lower halo (cell (x, y, z) at x + 1, y + 1,
    // z + 1), the right-hand side (overwritten with the result), and the halo's values
    __shared__ float sp[(MT + 1) * MPZ];
    __shared__ float sr[MT * MT * MT];
    __shared__ float hx[MT * MT], hy[MT * MT], hz[MT * MT];
    __shared__ int s_tile;
    __shared__ int s_abort;
    const int tid = threadIdx.x;
    dep_wait();
    dep_go();
    if (blockIdx.x == 0 && tid == 0) *other = 0;  // the next sweep's tile counter
    const int qx = (tid & 1) * 4, qy = (tid >> 1) % MT, qz = tid / (2 * MT);
    for (;;) {
        if (tid == 0) {
            const int w = atomicAdd(next, 1);
            s_tile = w < n ? order[FWD ? w : n - 1 - w] : -1;
            s_abort = 0;
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int ti = tile % G.ntx, tj = (tile / G.ntx) % G.nty, tk = tile / (G.ntx * G.nty);
        // the quad of this thread (a quad that begins inside the grid ends inside its row's padding)
        const bool qin = ti * MT + qx < G.nx && tj * MT + qy < G.ny && tk * MT + qz < G.nz;
        const int qt = G.origin + (tk * MT + qz) * G.PL + (tj * MT + qy) * G.P + ti * MT + qx;
        float4 rv = make_float4(0.f, 0.f, 0.f, 0.f), pv = rv;
        if (qin) {
            const uchar4 f = __ldg(reinterpret_cast<const uchar4 *>(cf + qt));
            const float4 r4 = ldd4(in + qt), p4 = *reinterpret_cast<const float4 *>(prec + qt);
            rv = make_float4(f.x & CF_LIQ ? r4.x : 0.f, f.y & CF_LIQ ? r4.y : 0.f, f.z & CF_LIQ ? r4.z : 0.f,
                             f.w & CF_LIQ ? r4.w : 0.f);
            pv = make_float4(f.x & CF_LIQ ? p4.x : 0.f, f.y & CF_LIQ ? p4.y : 0.f, f.z & CF_LIQ ? p4.z : 0.f,
                             f.w & CF_LIQ ? p4.w : 0.f);
        }
        {
            const float ra[4] = {rv.x, rv.y, rv.z, rv.w}, pa[4] = {pv.x, pv.y, pv.z, pv.w};
            const int wy = FWD ? qy : MT - 1 - qy, wz = FWD ? qz : MT - 1 - qz;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int wx = FWD ? qx + e : MT - 1 - qx - e;
                sr[(wz * MT + wy) * MT + wx] = ra[e];
                sp[(wz + 1) * MPZ + (wy + 1) * MPY + wx + 1] = pa[e];
            }
        }
        // the halo: cell (u, v) of face a, two per thread at most; its element, or -1 off the liquid
        int ht[2] = {-1, -1};
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int c = tid + h * MSTH;
            if (c >= 3 * MT * MT) continue;
            const int a = c / (MT * MT), u = c % MT, v = (c / MT) % MT;
            // walk coordinates of the halo cell: face 0 at (-1, u, v), 1 at (u, -1, v), 2 at (u, v, -1)
            const int wx = a == 0 ? -1 : u, wy = a == 1 ? -1 : (a == 0 ? u : v), wz = a == 2 ? -1 : v;
            const int gi = ti * MT + (FWD ? wx : MT - 1 - wx), gj = tj * MT + (FWD ? wy : MT - 1 - wy);
            const int gk = tk * MT + (FWD ? wz : MT - 1 - wz);
            float p = 0.f;
            if (gi >= 0 && gj >= 0 && gk >= 0 && gi < G.nx && gj < G.ny && gk < G.nz) {
                const int t = G.origin + gk * G.PL + gj * G.P + gi;
                if (liquid(cf, t)) {
                    ht[h] = t;
                    if (FWD) p = prec[t];
                }
            }
            if (FWD) sp[(wz + 1) * MPZ + (wy + 1) * MPY + wx + 1] = p;
        }
        if (tid < 3 && !wait_tile<DIR>(G, ti, tj, tk, tid, tact, tflag, epoch, spin_limit, err)) s_abort = 1;
        __syncthreads();
        if (s_abort) {
            // give up on this sweep: publish nothing, drain the remaining tiles
            __syncthreads();
            continue;
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int c = tid + h * MSTH;
            if (c >= 3 * MT * MT) continue;
            const float v = ht[h] >= 0 ? __ldcg(out + ht[h]) : 0.f;
            const int a = c / (MT * MT);
            (a == 0 ? hx : a == 1 ? hy : hz)[c % (MT * MT)] = v;
        }
        __syncthreads();
        if (tid < 32) {
            const int x = tid & 7, y = tid >> 3;
            float va = 0.f, vb = 0.f;  // the last value of column (x, y) and of (x, y + 4)
            auto cell = [&](int cy, int z, float nx, float ny, float nz) {  // cell (x, cy, z) from its predecessors
                const int i = (z * MT + cy) * MT + x, j = (z + 1) * MPZ + (cy + 1) * MPY + x + 1;
                const float p = sp[j], r = sr[i];
                float v;
                if (FWD) {
                    float acc = r;
                    acc += sp[j - 1] * nx;
                    acc += sp[j - MPY] * ny;
                    acc += sp[j - MPZ] * nz;
                    v = acc * p;
                } else {
                    v = p * (r + p * ((nx + ny) + nz));
                }
                return p != 0.f ? v : 0.f;  // (zero off the liquid)
            };
#pragma unroll
            for (int l = 0; l <= 3 * (MT - 1); l++) {
                const int za = l - x - y, zb = za - 4;
                const int ca = min(max(za, 0), MT - 1), cb = min(max(zb, 0), MT - 1);
                const float ax = __shfl_up_sync(0xffffffffu, va, 1), ay = __shfl_up_sync(0xffffffffu, va, 8);
                const float bx = __shfl_up_sync(0xffffffffu, vb, 1), by = __shfl_up_sync(0xffffffffu, vb, 8);
                const float ab = __shfl_sync(0xffffffffu, va, (tid + 24) & 31);  // (x, 3) for lanes (x, 0)
                const float wa = cell(y, ca, x == 0 ? hx[ca * MT + y] : ax, y == 0 ? hy[ca * MT + x] : ay,
                                      za == 0 ? hz[y * MT + x] : va);
                const float wb = cell(y + 4, cb, x == 0 ? hx[cb * MT + y + 4] : bx, y == 0 ? ab : by,
                                      zb == 0 ? hz[(y + 4) * MT + x] : vb);
                if (za == ca) sr[(ca * MT + y) * MT + x] = va = wa;
                if (zb == cb) sr[(cb * MT + y + 4) * MT + x] = vb = wb;
            }
        }
        __syncthreads();
        if (qin) {
            float o[4];
            const int wy = FWD ? qy : MT - 1 - qy, wz = FWD ? qz : MT - 1 - qz;
#pragma unroll
            for (int e = 0; e < 4; e++) o[e] = sr[(wz * MT + wy) * MT + (FWD ? qx + e : MT - 1 - qx - e)];
            *reinterpret_cast<float4 *>(out + qt) = make_float4(o[0], o[1], o[2], o[3]);
        }
        __syncthreads();
        if (tid == 0) {
            __threadfence();  // the block's values, ordered before this by the barrier
            st_release(tflag + tile, epoch);
        }
    }
}

}  // namespace

static MicGrid mic_grid(const fs_ctx *c)
{
    MicGrid g;
    g.nx = c->L.nx;
    g.ny = c->L.ny;
    g.nz = c->L.nz;
    g.ntx = (g.nx + MT - 1) / MT;
    g.nty = (g.ny + MT - 1) / MT;
    g.ntz = (g.nz + MT - 1) / MT;
    g.P = c->L.P;
    g.PL = c->L.PL;
    g.origin = c->L.PL;
    return g;
}

// Tile order by level and the per-tile liquid flag (set-up work, on the host).
static int mic_schedule(fs_ctx *c)
{
    const MicGrid g = mic_grid(c);
    const int ntiles = g.ntx * g.nty * g.ntz;
    std::vector<uint8_t> cf((size_t)c->L.nC);
    FS_CUDA(cudaMemcpy(cf.data(), c->cflag, cf.size(), cudaMemcpyDeviceToHost));
    std::vector<uint8_t> act((size_t)ntiles, 0);
    for (int k = 0; k < g.nz; k++)
        for (int j = 0; j < g.ny; j++)
            for (int i = 0; i < g.nx; i++)
                if (cf[(size_t)g.origin + (size_t)k * g.PL + (size_t)j * g.P + i] & CF_LIQ)
                    act[(size_t)((k / MT) * g.nty + j / MT) * g.ntx + i / MT] = 1;
    std::vector<int> order;
    for (int t = 0; t < ntiles; t++)
        if (act[(size_t)t]) order.push_back(t);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        const int la = a % g.ntx + (a / g.ntx) % g.nty + a / (g.ntx * g.nty);
        const int lb = b % g.ntx + (b / g.ntx) % g.nty + b / (g.ntx * g.nty);
        return la < lb;
    });
    c->mic_n = (int)order.size();
    if (!order.empty())
        FS_CUDA(cudaMemcpy(c->mic_order, order.data(), order.size() * sizeof(int), cudaMemcpyHostToDevice));
    FS_CUDA(cudaMemcpy(c->mic_tact, act.data(), act.size(), cudaMemcpyHostToDevice));
    FS_CUDA(cudaMemset(c->mic_tflag, 0, (size_t)ntiles * sizeof(int)));
    c->mic_epoch = 0;
    c->mic_sched_ready = 1;
    return FS_OK;
}

template <int MODE>
static int mic_solve(fs_ctx *c, const float *in, float *out)
{
    // forward and backward sweeps alternate, each with its own tile counter, which the
    // other one zeroes
    int *next = c->mic_next + (MODE == MIC_FORWARD ? 0 : 1), *other = c->mic_next + (MODE == MIC_FORWARD ? 1 : 0);
    c->mic_epoch += 1;
    const int grid = std::max(1, std::min(c->mic_n, 4 * c->num_sms));
    launch_dep(k_mic_solve<MODE>, grid, MSTH, 0, c->stream, mic_grid(c), c->cflag, c->mic_prec, in, out, c->mic_order,
               c->mic_n, c->mic_tact, c->mic_tflag, next, other, c->mic_epoch, c->prm.spin_limit, c->err_word);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    return FS_OK;
}

int mic0_factor(fs_ctx *c)
{
    if (!c->mic_sched_ready) {
        int rc = mic_schedule(c);
        if (rc) return rc;
    }
    FS_CUDA(cudaMemsetAsync(c->err_word, 0, sizeof(unsigned), c->stream));
    c->mic_epoch += 1;
    FS_CUDA(cudaMemsetAsync(c->mic_next, 0, 2 * sizeof(int), c->stream));  // (the factorisation counts in the second)
    const int grid = std::max(1, std::min(c->mic_n, 2 * c->num_sms));
    k_mic_factor<<<grid, MTH, 0, c->stream>>>(mic_grid(c), c->cflag, c->mic_prec, c->mic_order, c->mic_n, c->mic_tact,
                                              c->mic_tflag, c->mic_next + 1, c->mic_epoch, c->prm.spin_limit, c->err_word,
                                              (float)c->prm.mic_tau, (float)c->prm.mic_sigma);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    c->mic_ready = 1;
    return FS_OK;
}

int mic0_apply(fs_ctx *c, const float *r, float *z)
{
    cudaEvent_t e0 = prof_mark(c);
    int rc = mic_solve<MIC_FORWARD>(c, r, c->py);
    if (rc) return rc;
    rc = mic_solve<MIC_BACKWARD>(c, c->py, z);
    if (rc) return rc;
    prof_add(c, K_MIC_APPLY, e0, prof_mark(c), 0.0);
    return FS_OK;
}

}  // namespace fs
