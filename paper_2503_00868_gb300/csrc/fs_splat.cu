// fs_splat.cu -- forward splatting of the Gaussians into an image (arXiv
// 2503.00868, Sec. 3.2.1 compositing formula, Sec. 3.5 rendering by splatting),
// into a headless device buffer.
//
// Per Gaussian (pinhole camera, x_c = R x + t): depth z, projected mean, 2D
// covariance S = J R A R^T J^T (J the projection Jacobian at the mean) and its
// inverse (the conic). At a pixel centre d = pixel - mean,
//   alpha = min(0.99, sigma exp(-d^T S^-1 d / 2)), kept inside the 3-sigma ellipse
//   (d^T S^-1 d <= 9) and when alpha >= 1/255,
// and the pixel composites front to back by depth (ties by index):
//   C = sum_i alpha_i c_i T_i + T bg,  T_i = prod_{j<i} (1 - alpha_j),
// stopping once the transmittance would fall below 1e-4. Colours are degree-0
// spherical harmonics (RGB).
//
// Pipeline: (1) project, record each Gaussian's tile rectangle (16 x 16 pixel
// tiles covering the 3-sigma ellipse's bounding box) and count entries per tile;
// (2) exclusive scan of the counts (one block); (3) write (depth bits << 32 | index)
// keys into each tile's segment; (4) one block per tile sorts a segment and
// composites, one thread per pixel, in batches of records staged in shared memory.
// The sort is a bucket sort in shared memory, linear in the keys: the tile's depths
// are nearly uniform, so SP_NB buckets over their range hold a key or two each, which
// one thread puts in order. A segment
// of more than SP_CAP keys is first dealt into coarse buckets in global memory, which
// come in groups of at most SP_CAP: most tiles saturate in the first one. Depths that
// crowd into a bucket (a plane facing the camera) take a bitonic sort, or a radix
// sort of the whole segment. Every sort orders the full 64-bit key, so equal depths
// fall back to index order whatever order the atomics filled the segment in.
//
// Bitonic sorts of every segment and a radix sort of the longest by one block took
// 407 and 126 us of a 650 us frame (835 k Gaussians at 1920 x 1080, 5.7 M pairs); this
// step takes 178 of 275. The latency of the compositing's own instructions is most of
// it now (issue on 62 % of the cycles, L1 below half its rate): a warp has a block of
// 8 x 4 pixels and walks only the records whose box meets it (208 us when it walked
// them all), which leaves the order and every sum as they were.
#include <cmath>
#include <new>

#include "fs_internal.cuh"

namespace fs {

struct __align__(16) SplatRecord {
    float mx, my;          // projected mean (pixels)
    float ca, cb;          // conic: S^-1 = [[ca, cb], [cb, cc]]
    float r, g, b;
    float opacity;
    float cc;
    float ex, ey;          // half extents of the 3-sigma ellipse's bounding box, 1 pixel added
    float pad;
};

struct SplatState {
    SplatRecord *rec = nullptr;
    int4 *rect = nullptr;            // tile rectangle [x0, x1) x [y0, y1)
    float *depth = nullptr;
    int cap_n = 0;
    unsigned *tcount = nullptr, *toff = nullptr, *tfill = nullptr;
    int cap_t = 0;
    unsigned long long *keys = nullptr, *keys2 = nullptr;
    long long cap_k = 0, cap_k2 = 0;
    unsigned long long last_entries = 0, last_max = 0;  // counters of the last render
};

namespace {

constexpr int SP_TILE = 16;
constexpr int SP_CAP = 4096;   // keys of a tile sorted in shared memory at once
constexpr int SP_NB = 2048;    // buckets of its sort (coarse and fine)
constexpr int SP_CROWD = 48;   // keys in one bucket above which the bitonic sort takes over

struct Cam {
    float R[9], t[3];
    float fx, fy, cx, cy;
    int w, h;
    float znear;
    float bg[3];
};

// Block-local table of tiles (open addressing, linear probing, no deletion): the
// (Gaussian, tile) pairs of a block's 256 Gaussians, which are usually neighbours
// in space and share tiles, are counted in shared memory and reach the global
// per-tile counters with one atomic per distinct tile. A tile that finds no slot
// within SP_PROBE probes goes to the global counter directly; since slots are
// never freed, a later lookup of that tile fails the same way.
constexpr int SP_HT = 1024;
constexpr int SP_PROBE = 16;
constexpr unsigned SP_EMPTY = 0xffffffffu;

__device__ __forceinline__ int ht_slot(unsigned *hk, unsigned t, bool insert)
{
    const unsigned h = (t * 2654435761u) >> 22;
    for (int p = 0; p < SP_PROBE; p++) {
        const unsigned sl = (h + p) & (SP_HT - 1);
        unsigned cur = hk[sl];
        if (cur == t) return (int)sl;
        if (cur == SP_EMPTY) {
            if (!insert) return -1;
            cur = atomicCAS(hk + sl, SP_EMPTY, t);
            if (cur == SP_EMPTY || cur == t) return (int)sl;
        }
    }
    return -1;
}

// View-dependent colour (Sec. 3.2.1, SH(r; F_i)): max(0, 1/2 + sum_j sh[j] Y_j(d))
// per channel, with the real spherical harmonics Y_j of degree <= 3 in the sign
// convention of the standard 3DGS evaluator and d the unit vector from the camera
// centre to the mean. The constants are the normalisations of the basis:
// sqrt(3/4pi), sqrt(15/4pi), sqrt(5/16pi), sqrt(15/16pi), sqrt(35/32pi),
// sqrt(105/4pi), sqrt(21/32pi), sqrt(7/16pi).
__device__ __forceinline__ void sh_colour(int deg, const float *__restrict__ sh, float dx, float dy, float dz,
                                          float out[3])
{
    constexpr float Y0 = 0.28209479177387814f, A1 = 0.4886025119029199f;
    constexpr float B2 = 1.0925484305920792f, C2 = 0.31539156525252005f, E2 = 0.5462742152960396f;
    constexpr float F3 = 0.5900435899266435f, G3 = 2.890611442640554f, H3 = 0.4570457994644658f,
                    K3 = 0.3731763325901154f;
    float Y[16];
    Y[0] = Y0;
    if (deg >= 1) {
        Y[1] = -A1 * dy;
        Y[2] = A1 * dz;
        Y[3] = -A1 * dx;
    }
    if (deg >= 2) {
        const float xx = dx * dx, yy = dy * dy, zz = dz * dz;
        Y[4] = B2 * dx * dy;
        Y[5] = -B2 * dy * dz;
        Y[6] = C2 * (2.f * zz - xx - yy);
        Y[7] = -B2 * dx * dz;
        Y[8] = E2 * (xx - yy);
        if (deg >= 3) {
            Y[9] = -F3 * dy * (3.f * xx - yy);
            Y[10] = G3 * dx * dy * dz;
            Y[11] = -H3 * dy * (4.f * zz - xx - yy);
            Y[12] = K3 * dz * (2.f * zz - 3.f * xx - 3.f * yy);
            Y[13] = -H3 * dx * (4.f * zz - xx - yy);
            Y[14] = 0.5f * G3 * dz * (xx - yy);
            Y[15] = -F3 * dx * (xx - 3.f * yy);
        }
    }
    const int nb = (deg + 1) * (deg + 1);
#pragma unroll
    for (int k = 0; k < 3; k++) {
        float v = 0.5f;
        for (int j = 0; j < nb; j++) v += sh[3 * j + k] * Y[j];
        out[k] = fmaxf(v, 0.f);
    }
}

// Projection, colour and tile counting of each Gaussian. The colour is col[i]
// (RGB) or, with sh non-null, the spherical-harmonic colour of degree `deg`
// seen from the camera centre.
__global__ void __launch_bounds__(256) k_sp_project(int n, const float *__restrict__ x,
                                                    const float *__restrict__ op, const float *__restrict__ A,
                                                    const float *__restrict__ col, const float *__restrict__ sh,
                                                    int deg, Cam cam, SplatRecord *rec, int4 *rect, float *depth,
                                                    unsigned *tcount, int ntx, int nty)
{
    __shared__ unsigned hk[SP_HT], hc[SP_HT];
    for (int base = blockIdx.x * 256; base < n; base += gridDim.x * 256) {  // uniform over the block
        for (int e = threadIdx.x; e < SP_HT; e += 256) {
            hk[e] = SP_EMPTY;
            hc[e] = 0;
        }
        __syncthreads();
        const int i = base + threadIdx.x;
        int4 rc = make_int4(0, 0, 0, 0);
        float xc[3];
        const int ii = min(i, n - 1);  // rows past n: read a valid row, record nothing
#pragma unroll
        for (int r = 0; r < 3; r++)
            xc[r] = cam.R[3 * r] * x[3 * ii] + cam.R[3 * r + 1] * x[3 * ii + 1] + cam.R[3 * r + 2] * x[3 * ii + 2] +
                    cam.t[r];
        const float z = xc[2];
        if (i < n && z > cam.znear) {
            const float mx = cam.fx * xc[0] / z + cam.cx, my = cam.fy * xc[1] / z + cam.cy;
            const float J[6] = {cam.fx / z, 0.f, -cam.fx * xc[0] / (z * z), 0.f, cam.fy / z, -cam.fy * xc[1] / (z * z)};
            float M[6];
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
                for (int c = 0; c < 3; c++)
                    M[3 * r + c] = J[3 * r] * cam.R[c] + J[3 * r + 1] * cam.R[3 + c] + J[3 * r + 2] * cam.R[6 + c];
            float S[4];
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
                for (int s = 0; s < 2; s++) {
                    float acc = 0.f;
#pragma unroll
                    for (int a = 0; a < 3; a++)
#pragma unroll
                        for (int b = 0; b < 3; b++) acc += M[3 * r + a] * A[9 * i + 3 * a + b] * M[3 * s + b];
                    S[2 * r + s] = acc;
                }
            const float det = S[0] * S[3] - S[1] * S[2];
            if (det > 0.f && S[0] > 0.f && S[3] > 0.f) {
                SplatRecord q;
                q.mx = mx;
                q.my = my;
                q.ca = S[3] / det;
                q.cb = -S[1] / det;
                q.cc = S[0] / det;
                q.opacity = op[i];
                if (sh) {
                    // the camera centre -R^T t and the unit direction to the mean
                    float d[3], nrm = 0.f;
#pragma unroll
                    for (int r = 0; r < 3; r++) {
                        const float cr = -(cam.R[r] * cam.t[0] + cam.R[3 + r] * cam.t[1] + cam.R[6 + r] * cam.t[2]);
                        d[r] = x[3 * i + r] - cr;
                        nrm += d[r] * d[r];
                    }
                    const float inv = nrm > 0.f ? rsqrtf(nrm) : 0.f;
                    float cv[3];
                    sh_colour(deg, sh + (size_t)i * (deg + 1) * (deg + 1) * 3, d[0] * inv, d[1] * inv, d[2] * inv, cv);
                    q.r = cv[0];
                    q.g = cv[1];
                    q.b = cv[2];
                } else {
                    q.r = col[3 * i];
                    q.g = col[3 * i + 1];
                    q.b = col[3 * i + 2];
                }
                // the 3-sigma ellipse lies in mean +- 3 sqrt(diag S); pixel centres at p + 1/2
                const float ex = 3.f * sqrtf(S[0]) + 1.f, ey = 3.f * sqrtf(S[3]) + 1.f;
                q.ex = ex;
                q.ey = ey;
                q.pad = 0.f;
                rec[i] = q;
                depth[i] = z;
                const float x0 = fmaxf(mx - ex, 0.f), x1 = fminf(mx + ex, (float)cam.w);
                const float y0 = fmaxf(my - ey, 0.f), y1 = fminf(my + ey, (float)cam.h);
                if (x0 < x1 && y0 < y1) {
                    rc.x = min((int)(x0 / SP_TILE), ntx - 1);
                    rc.y = min((int)(x1 / SP_TILE), ntx - 1) + 1;
                    rc.z = min((int)(y0 / SP_TILE), nty - 1);
                    rc.w = min((int)(y1 / SP_TILE), nty - 1) + 1;
                }
            }
        }
        if (i < n) rect[i] = rc;
        for (int ty = rc.z; ty < rc.w; ty++)
            for (int tx = rc.x; tx < rc.y; tx++) {
                const unsigned t = (unsigned)(ty * ntx + tx);
                const int sl = ht_slot(hk, t, true);
                if (sl >= 0)
                    atomicAdd(hc + sl, 1u);
                else
                    atomicAdd(tcount + t, 1u);
            }
        __syncthreads();
        for (int e = threadIdx.x; e < SP_HT; e += 256)
            if (hk[e] != SP_EMPTY) atomicAdd(tcount + hk[e], hc[e]);
        __syncthreads();
    }
}

// exclusive scan of the tile counts, one block of 1024 threads; total[0] = the
// number of entries, total[1] = the largest tile count
__global__ void __launch_bounds__(1024) k_sp_scan(const unsigned *__restrict__ cnt, unsigned *off, int nt,
                                                  unsigned long long *total)
{
    __shared__ unsigned long long part[1024];
    __shared__ unsigned pmax[1024];
    const int per = (nt + 1023) / 1024;
    const int lo = threadIdx.x * per, hi = min(lo + per, nt);
    unsigned long long s = 0;
    unsigned mx = 0;
    for (int t = lo; t < hi; t++) {
        s += cnt[t];
        mx = max(mx, cnt[t]);
    }
    part[threadIdx.x] = s;
    pmax[threadIdx.x] = mx;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {  // inclusive scan (Hillis-Steele)
        const unsigned long long v = threadIdx.x >= d ? part[threadIdx.x - d] : 0ull;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    unsigned long long run = threadIdx.x ? part[threadIdx.x - 1] : 0ull;
    for (int t = lo; t < hi; t++) {
        off[t] = (unsigned)run;
        run += cnt[t];
    }
    for (int d = 512; d > 0; d >>= 1) {
        if ((int)threadIdx.x < d) pmax[threadIdx.x] = max(pmax[threadIdx.x], pmax[threadIdx.x + d]);
        __syncthreads();
    }
    if (threadIdx.x == 1023) total[0] = part[1023];
    if (threadIdx.x == 0) total[1] = pmax[0];
}

// Writes each (Gaussian, tile) key into its tile's segment. Pass 1 counts a
// block's pairs per tile in the shared table (pairs without a slot take a global
// position at once); one global atomic per table slot then reserves a contiguous
// range of the segment; pass 2 walks the pairs again and places them in the range.
__global__ void __launch_bounds__(256) k_sp_fill(int n, const int4 *__restrict__ rect,
                                                 const float *__restrict__ depth,
                                                 const unsigned *__restrict__ off, unsigned *fill,
                                                 unsigned long long *keys, int ntx)
{
    __shared__ unsigned hk[SP_HT], hc[SP_HT], hb[SP_HT];
    for (int base = blockIdx.x * 256; base < n; base += gridDim.x * 256) {  // uniform over the block
        for (int e = threadIdx.x; e < SP_HT; e += 256) {
            hk[e] = SP_EMPTY;
            hc[e] = 0;
        }
        __syncthreads();
        const int i = base + threadIdx.x;
        const int4 rc = i < n ? rect[i] : make_int4(0, 0, 0, 0);
        const unsigned long long key =
            i < n ? ((unsigned long long)__float_as_uint(depth[i]) << 32) | (unsigned)i : 0ull;
        for (int ty = rc.z; ty < rc.w; ty++)
            for (int tx = rc.x; tx < rc.y; tx++) {
                const unsigned t = (unsigned)(ty * ntx + tx);
                const int sl = ht_slot(hk, t, true);
                if (sl >= 0) {
                    atomicAdd(hc + sl, 1u);
                } else {
                    const unsigned pos = atomicAdd(fill + t, 1u);
                    keys[off[t] + pos] = key;
                }
            }
        __syncthreads();
        for (int e = threadIdx.x; e < SP_HT; e += 256)
            if (hk[e] != SP_EMPTY) {
                hb[e] = off[hk[e]] + atomicAdd(fill + hk[e], hc[e]);
                hc[e] = 0;
            }
        __syncthreads();
        for (int ty = rc.z; ty < rc.w; ty++)
            for (int tx = rc.x; tx < rc.y; tx++) {
                const int sl = ht_slot(hk, (unsigned)(ty * ntx + tx), false);
                if (sl >= 0) keys[hb[sl] + atomicAdd(hc + sl, 1u)] = key;
            }
        __syncthreads();
    }
}

// Stable LSD radix sort (8-bit digits) of a segment of n keys by one block of 256
// threads, through `tmp`, with 17.5 KB of shared memory. Digits 0-3 are the Gaussian
// index (those above the largest index are skipped), 4-7 the depth bits; a digit that
// all keys share is skipped too. A round takes 2048 keys, warp w the 256 consecutive
// keys [w * 256, w * 256 + 256) as BS_IT slots of 32; slot by slot, a key's rank among
// the warp's keys with the same digit is the warp's running count of that digit plus
// its rank within the slot (__match_any_sync), and the warps are ordered by a
// per-digit prefix, so equal digits keep their order. The result ends in `keys`.
constexpr int BS_IT = 8;

__device__ __noinline__ void radix_segment(unsigned long long *keys, unsigned long long *tmp, unsigned n, int idx_digits,
                                           unsigned *sm)
{
    unsigned *hist = sm, *wsum = sm + 256;
    unsigned(*wcnt)[256] = reinterpret_cast<unsigned(*)[256]>(sm + 264);
    unsigned(*wpos)[256] = reinterpret_cast<unsigned(*)[256]>(sm + 264 + 8 * 256);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long *src = keys, *dst = tmp;
    for (int w = 0; w < 8; w++) wcnt[w][tid] = 0;
    for (int dgt = 0; dgt < 8; dgt++) {
        if (dgt < 4 && dgt >= idx_digits) continue;
        const int shift = 8 * dgt;
        hist[tid] = 0;
        __syncthreads();
        for (unsigned e = tid; e < n; e += 256) atomicAdd(&hist[(unsigned)(src[e] >> shift) & 255u], 1u);
        __syncthreads();
        if (__syncthreads_or(hist[tid] == n)) continue;  // one digit for all keys
        // exclusive scan of the histogram: the digits' base positions
        const unsigned v = hist[tid];
        unsigned incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        unsigned wpre = 0;
        for (int w = 0; w < warp; w++) wpre += wsum[w];
        hist[tid] = wpre + incl - v;
        __syncthreads();
        for (unsigned r0 = 0; r0 < n; r0 += 256 * BS_IT) {
            unsigned long long kv[BS_IT];
            unsigned dg[BS_IT], rk[BS_IT];
#pragma unroll
            for (int q = 0; q < BS_IT; q++) {
                const unsigned e = r0 + warp * 256 + q * 32 + lane;
                kv[q] = e < n ? src[e] : 0ull;
                dg[q] = e < n ? ((unsigned)(kv[q] >> shift) & 255u) : 256u;
            }
#pragma unroll
            for (int q = 0; q < BS_IT; q++) {
                const unsigned mask = __match_any_sync(0xffffffffu, dg[q]);
                const unsigned before = dg[q] < 256u ? wcnt[warp][dg[q]] : 0u;
                rk[q] = before + __popc(mask & ((1u << lane) - 1u));
                __syncwarp();
                if (dg[q] < 256u && lane == __ffs(mask) - 1) wcnt[warp][dg[q]] = before + __popc(mask);
                __syncwarp();
            }
            __syncthreads();
            unsigned run = hist[tid];  // thread tid owns digit tid
            for (int w = 0; w < 8; w++) {
                wpos[w][tid] = run;
                run += wcnt[w][tid];
                wcnt[w][tid] = 0;
            }
            hist[tid] = run;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < BS_IT; q++)
                if (dg[q] < 256u) dst[wpos[warp][dg[q]] + rk[q]] = kv[q];
        }
        unsigned long long *t = src;
        src = dst;
        dst = t;
        __syncthreads();
    }
    if (src != keys)
        for (unsigned e = tid; e < n; e += 256) keys[e] = src[e];
    __syncthreads();
}

__device__ __forceinline__ float key_depth(unsigned long long k) { return __uint_as_float((unsigned)(k >> 32)); }

// Monotone bucket of a depth: floor((d - dmin) * scale), clamped.
struct DepthBuckets {
    float dmin, scale;
    __device__ __forceinline__ DepthBuckets(unsigned lo, unsigned hi)
    {
        dmin = __uint_as_float(lo);
        const float range = __uint_as_float(hi) - dmin;
        scale = range > 0.f ? (float)SP_NB / range : 0.f;
    }
    __device__ __forceinline__ int of(unsigned long long k) const
    {
        return max(0, min(SP_NB - 1, (int)((key_depth(k) - dmin) * scale)));
    }
};

// smallest and largest depth bits over the block (positive floats order like integers)
__device__ __forceinline__ void block_range(unsigned &lo, unsigned &hi)
{
    __shared__ unsigned slo[8], shi[8];
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        slo[threadIdx.x >> 5] = lo;
        shi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    for (int w = 0; w < 8; w++) {
        lo = min(lo, slo[w]);
        hi = max(hi, shi[w]);
    }
}

// exclusive scan of the SP_NB counts in place; returns the largest count
__device__ __forceinline__ unsigned scan_buckets(unsigned *hist)
{
    __shared__ unsigned wsum[8], wmax[8];
    constexpr int PER = SP_NB / 256;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned c[PER], sum = 0, mx = 0;
#pragma unroll
    for (int k = 0; k < PER; k++) {
        c[k] = hist[tid * PER + k];
        sum += c[k];
        mx = max(mx, c[k]);
    }
    unsigned incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 31) wsum[warp] = incl;
    if (lane == 0) wmax[warp] = mx;
    __syncthreads();
    unsigned run = incl - sum;
    for (int w = 0; w < 8; w++) {
        if (w < warp) run += wsum[w];
        mx = max(mx, wmax[w]);
    }
#pragma unroll
    for (int k = 0; k < PER; k++) {
        hist[tid * PER + k] = run;
        run += c[k];
    }
    __syncthreads();
    return mx;
}

// Sorts the n <= SP_CAP keys at src (global memory; read three times, from L1 or L2)
// into sk. With SP_NB buckets a bucket holds one or two keys, which its thread orders
// in place.
__device__ __forceinline__ void sort_tile(const unsigned long long *src, int n, unsigned long long *sk, unsigned *hist)
{
    const int tid = threadIdx.x;
    unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
    for (int e = tid; e < n; e += 256) {
        const unsigned d = (unsigned)(src[e] >> 32);
        lo = min(lo, d);
        hi = max(hi, d);
    }
    for (int e = tid; e < SP_NB; e += 256) hist[e] = 0;
    block_range(lo, hi);
    const DepthBuckets bk(lo, hi);
#pragma unroll 4
    for (int e = tid; e < n; e += 256) atomicAdd(&hist[bk.of(src[e])], 1u);
    __syncthreads();
    const bool crowded = scan_buckets(hist) > SP_CROWD;
#pragma unroll 4
    for (int e = tid; e < n; e += 256) {
        const unsigned long long k = src[e];
        sk[atomicAdd(&hist[bk.of(k)], 1u)] = k;  // each start becomes the bucket's end
    }
    __syncthreads();
    if (!crowded) {
        for (int b = tid; b < SP_NB; b += 256) {
            const int b0 = b ? (int)hist[b - 1] : 0, b1 = (int)hist[b];
            for (int i = b0 + 1; i < b1; i++) {
                const unsigned long long k = sk[i];
                int j = i;
                for (; j > b0 && sk[j - 1] > k; j--) sk[j] = sk[j - 1];
                sk[j] = k;
            }
        }
        __syncthreads();
        return;
    }
    // crowded depths: bitonic sort (ascending: depth, then index)
    int m = 1;
    while (m < n) m <<= 1;
    for (int e = n + tid; e < m; e += 256) sk[e] = ~0ull;
    __syncthreads();
    for (int k = 2; k <= m; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int e = tid; e < m; e += 256) {
                const int p = e ^ j;
                if (p > e) {
                    const bool up = (e & k) == 0;
                    const unsigned long long a = sk[e], b = sk[p];
                    if ((a > b) == up) {
                        sk[e] = b;
                        sk[p] = a;
                    }
                }
            }
            __syncthreads();
        }
}

// shared memory of k_sp_render: keys, buckets, a batch of records
constexpr size_t SP_SMEM = (size_t)SP_CAP * 8 + SP_NB * 4 + 256 * (16 + 16 + 4 + 1);

__global__ void __launch_bounds__(256, 4) k_sp_render(unsigned long long *keys, unsigned long long *tmp, int idx_digits,
                                                   const unsigned *__restrict__ off,
                                                   const unsigned *__restrict__ cnt,
                                                   const SplatRecord *__restrict__ rec, Cam cam, int ntx,
                                                   float *rgb, float *Tout)
{
    extern __shared__ __align__(16) unsigned char sp_sm[];
    unsigned long long *sk = reinterpret_cast<unsigned long long *>(sp_sm);
    unsigned *hist = reinterpret_cast<unsigned *>(sk + SP_CAP);
    float4 *ra = reinterpret_cast<float4 *>(hist + SP_NB), *rb = ra + 256;  // mean and conic; colour and opacity
    float *rc = reinterpret_cast<float *>(rb + 256);                        // the conic's last entry
    uint8_t *rw = reinterpret_cast<uint8_t *>(rc + 256);                    // the warps a record may touch
    __shared__ int group;
    const int tile = blockIdx.x;
    const int tid = threadIdx.x;
    const unsigned n = cnt[tile];
    unsigned long long *seg = keys + off[tile];
    // a warp has 8 x 4 pixels, and walks the records of a batch whose box meets them
    const int warp = tid >> 5, lane = tid & 31;
    const int tx0 = (tile % ntx) * SP_TILE, ty0 = (tile / ntx) * SP_TILE;
    const int px = tx0 + (warp & 1) * 8 + (lane & 7), py = ty0 + (warp >> 1) * 4 + (lane >> 3);
    const bool inside = px < cam.w && py < cam.h;
    const float pu = px + 0.5f, pv = py + 0.5f;
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    bool done = !inside;
    // composites the m sorted keys in sk; true when every pixel is done
    auto composite = [&](int m) -> bool {
        for (int b0 = 0; b0 < m; b0 += 256) {
            if (__syncthreads_and(done)) return true;
            if (b0 + tid < m) {
                const float4 *r = reinterpret_cast<const float4 *>(rec + (unsigned)(sk[b0 + tid] & 0xffffffffu));
                const float4 a = __ldg(r), c = __ldg(r + 2);
                ra[tid] = a;
                rb[tid] = __ldg(r + 1);
                rc[tid] = c.x;
                // pixel centres tx0 + 1/2 .. tx0 + 15/2 in the left column of warps, and so on
                unsigned cols = 0, rows = 0;
#pragma unroll
                for (int k = 0; k < 2; k++)
                    if (a.x + c.y >= (float)(tx0 + 8 * k) && a.x - c.y <= (float)(tx0 + 8 * k + 8)) cols |= 1u << k;
#pragma unroll
                for (int k = 0; k < 4; k++)
                    if (a.y + c.z >= (float)(ty0 + 4 * k) && a.y - c.z <= (float)(ty0 + 4 * k + 4)) rows |= cols << (2 * k);
                rw[tid] = (uint8_t)rows;
            }
            __syncthreads();
            const int nb = min(256, m - b0);
            for (int q0 = 0; q0 < nb; q0 += 32) {
                unsigned hits = __ballot_sync(0xffffffffu, q0 + lane < nb && ((rw[q0 + lane] >> warp) & 1));
                if (__all_sync(0xffffffffu, done)) break;
                for (; hits && !done; hits &= hits - 1) {
                    const int q = q0 + __ffs(hits) - 1;
                    const float4 g = ra[q];
                    const float dx = pu - g.x, dy = pv - g.y;
                    const float md = g.z * dx * dx + 2.f * g.w * dx * dy + rc[q] * dy * dy;
                    if (md > 9.f) continue;
                    const float4 col = rb[q];
                    float alpha = fminf(0.99f, col.w * expf(-0.5f * md));
                    if (alpha < 1.f / 255.f) continue;
                    const float Tn = T * (1.f - alpha);
                    if (Tn < 1e-4f) {
                        done = true;
                        break;
                    }
                    c0 += alpha * T * col.x;
                    c1 += alpha * T * col.y;
                    c2 += alpha * T * col.z;
                    T = Tn;
                }
                __syncwarp();
            }
        }
        return __syncthreads_and(done);
    };
    if (n <= SP_CAP) {
        if (n > 0) {
            sort_tile(seg, (int)n, sk, hist);
            composite((int)n);
        }
    } else {
        // coarse buckets in global memory
        unsigned long long *out = tmp + off[tile];
        unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
        for (unsigned e = tid; e < n; e += 256) {
            const unsigned d = (unsigned)(seg[e] >> 32);
            lo = min(lo, d);
            hi = max(hi, d);
        }
        for (int e = tid; e < SP_NB; e += 256) hist[e] = 0;
        block_range(lo, hi);
        const DepthBuckets bk(lo, hi);
#pragma unroll 4
        for (unsigned e = tid; e < n; e += 256) atomicAdd(&hist[bk.of(seg[e])], 1u);
        __syncthreads();
        if (scan_buckets(hist) <= SP_CAP) {
#pragma unroll 4
            for (unsigned e = tid; e < n; e += 256) {
                const unsigned long long k = seg[e];
                out[atomicAdd(&hist[bk.of(k)], 1u)] = k;  // each start becomes the bucket's end
            }
            __syncthreads();
            unsigned ends[SP_NB / 256];  // the ends outlive the shared buckets, which the groups' sorts use
#pragma unroll
            for (int k = 0; k < SP_NB / 256; k++) ends[k] = hist[tid * (SP_NB / 256) + k];
            for (unsigned b0 = 0; b0 < n;) {
                if (tid == 0) group = 0;
                __syncthreads();
                int best = 0;  // the last end within SP_CAP of b0
#pragma unroll
                for (int k = 0; k < SP_NB / 256; k++)
                    if (ends[k] > b0 && ends[k] - b0 <= SP_CAP) best = max(best, (int)(ends[k] - b0));
                if (best) atomicMax(&group, best);
                __syncthreads();
                const int m = group;
                sort_tile(out + b0, m, sk, hist);
                if (composite(m)) break;
                b0 += m;
            }
        } else {  // more keys in one coarse bucket than shared memory holds
            radix_segment(seg, out, n, idx_digits, reinterpret_cast<unsigned *>(sk));
            for (unsigned b0 = 0; b0 < n; b0 += SP_CAP) {
                const int m = (int)min((unsigned)SP_CAP, n - b0);
                for (int e = tid; e < m; e += 256) sk[e] = seg[b0 + e];
                __syncthreads();
                if (composite(m)) break;
            }
        }
    }
    if (inside) {
        const long long o = (long long)py * cam.w + px;
        rgb[3 * o] = c0 + T * cam.bg[0];
        rgb[3 * o + 1] = c1 + T * cam.bg[1];
        rgb[3 * o + 2] = c2 + T * cam.bg[2];
        if (Tout) Tout[o] = T;
    }
}

template <typename T>
int grow(T **p, long long &cap, long long need)
{
    if (need <= cap && *p) return FS_OK;
    cudaFree(*p);
    *p = nullptr;
    cap = 0;
    const long long n = need > 0 ? need : 1;
    if (cudaMalloc((void **)p, (size_t)n * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        return set_error(FS_ENOMEM, "splatting scratch of %lld elements", n);
    }
    cap = n;
    return FS_OK;
}

}  // namespace

void splat_free(fs_ctx *c)
{
    SplatState *s = static_cast<SplatState *>(c->splat);
    if (!s) return;
    cudaFree(s->rec);
    cudaFree(s->rect);
    cudaFree(s->depth);
    cudaFree(s->tcount);
    cudaFree(s->toff);
    cudaFree(s->tfill);
    cudaFree(s->keys);
    cudaFree(s->keys2);
    delete s;
    c->splat = nullptr;
}

int splat_render(fs_ctx *c, int n, const float *x, const float *op, const float *A, const float *col,
                 const float *sh, int deg, const fs_camera *camh, float *rgb, float *T)
{
    SplatState *s = static_cast<SplatState *>(c->splat);
    if (!s) {
        s = new (std::nothrow) SplatState();
        if (!s) return set_error(FS_ENOMEM, "host allocation failed");
        c->splat = s;
    }
    Cam cam;
    for (int k = 0; k < 9; k++) cam.R[k] = (float)camh->R[k];
    for (int k = 0; k < 3; k++) {
        cam.t[k] = (float)camh->t[k];
        cam.bg[k] = (float)camh->bg[k];
    }
    cam.fx = (float)camh->fx;
    cam.fy = (float)camh->fy;
    cam.cx = (float)camh->cx;
    cam.cy = (float)camh->cy;
    cam.w = camh->width;
    cam.h = camh->height;
    cam.znear = (float)camh->znear;
    const int ntx = (cam.w + SP_TILE - 1) / SP_TILE, nty = (cam.h + SP_TILE - 1) / SP_TILE, nt = ntx * nty;
    int rc;
    if (n > s->cap_n || !s->rec) {  // per-Gaussian arrays, grown together
        long long c0 = 0, c1 = 0, c2 = 0;
        if ((rc = grow(&s->rec, c0, n)) || (rc = grow(&s->rect, c1, n)) || (rc = grow(&s->depth, c2, n))) return rc;
        s->cap_n = n > 0 ? n : 1;
    }
    if (nt > s->cap_t || !s->tcount) {  // per-tile arrays
        long long c0 = 0, c1 = 0, c2 = 0;
        if ((rc = grow(&s->tcount, c0, nt)) || (rc = grow(&s->toff, c1, nt)) || (rc = grow(&s->tfill, c2, nt)))
            return rc;
        s->cap_t = nt;
    }
    FS_CUDA(cudaMemsetAsync(s->tcount, 0, (size_t)nt * 4, c->stream));
    FS_CUDA(cudaMemsetAsync(s->tfill, 0, (size_t)nt * 4, c->stream));
    const int gb = grid_blocks(c, n > 0 ? n : 1, 256);
    if (n > 0)
        k_sp_project<<<gb, 256, 0, c->stream>>>(n, x, op, A, col, sh, deg, cam, s->rec, s->rect, s->depth,
                                                s->tcount, ntx, nty);
    unsigned long long *total_d = reinterpret_cast<unsigned long long *>(c->partials);
    k_sp_scan<<<1, 1024, 0, c->stream>>>(s->tcount, s->toff, nt, total_d);
    c->n_launches += 2;
    FS_CUDA(cudaGetLastError());
    unsigned long long tot[2] = {0, 0};
    FS_CUDA(cudaMemcpyAsync(tot, total_d, sizeof(tot), cudaMemcpyDeviceToHost, c->stream));
    FS_CUDA(cudaStreamSynchronize(c->stream));
    s->last_entries = tot[0];
    s->last_max = tot[1];
    if (tot[0] > 0xffffffffull) return set_error(FS_EINVAL, "more than 2^32 tile entries");
    if ((rc = grow(&s->keys, s->cap_k, (long long)tot[0]))) return rc;
    if (n > 0) {
        k_sp_fill<<<gb, 256, 0, c->stream>>>(n, s->rect, s->depth, s->toff, s->tfill, s->keys, ntx);
        c->n_launches += 1;
    }
    if (tot[1] > (unsigned long long)SP_CAP)
        if ((rc = grow(&s->keys2, s->cap_k2, (long long)tot[0]))) return rc;
    const int idx_digits = n <= (1 << 8) ? 1 : n <= (1 << 16) ? 2 : n <= (1 << 24) ? 3 : 4;
    FS_CUDA(cudaFuncSetAttribute(k_sp_render, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SP_SMEM));
    k_sp_render<<<nt, 256, SP_SMEM, c->stream>>>(s->keys, s->keys2, idx_digits, s->toff, s->tcount, s->rec, cam, ntx, rgb,
                                                 T);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    return FS_OK;
}

void splat_stats(const fs_ctx *c, unsigned long long *entries, unsigned long long *max_tile)
{
    const SplatState *s = static_cast<const SplatState *>(c->splat);
    *entries = s ? s->last_entries : 0;
    *max_tile = s ? s->last_max : 0;
}

}  // namespace fs
