// fs_net.cu -- the learned pressure preconditioner (arXiv 2503.00868, Sec. 3.4.1,
// Fig. percnn_str_fit: a convolutional network with fitted 3x3x3 kernels that
// maps a pressure right-hand side to a pressure, fitted to solver output).
//
// Network: five 3x3x3 convolutions, channels 2 -> 16 -> 16 -> 16 -> 16 -> 1, zero
// padding at the grid boundary, ReLU after the first four. Input channel 0 is
// r / s on liquid cells rounded to bf16 (s = max |r| over the liquid), channel 1
// the cell type code (liquid 1, air 0, solid -1). Output z = s * y on liquid
// cells. Weights are bf16 (FP32 master copies for training), every hidden
// activation is stored as bf16, every sum accumulates in FP32.
//
// Kernels:
//   k_conv<OUT>    layers 2-5, layer 1 of training and the backward-data pass of
//                  layers 2-4 (flipped, transposed weights, ReLU-derivative
//                  epilogue) as an implicit GEMM per 3x3x3 tap on the tensor cores
//                  (mma.sync m16n8k16 bf16 x bf16 -> f32), tiles by tensor copy,
//                  weights in registers; layer 5 uses one 8-wide n-tile and writes
//                  z = s y on liquid cells. For inference layer l visits only the
//                  tiles within 5 - l cells of the liquid (the output on liquid
//                  cells depends on nothing farther), from a list sorted by that
//                  distance;
//   k_conv1        layer 1 of inference from r itself, three taps per MMA;
//   k_conv_tc      the inference layers on tcgen05 (fs_net_kernel);
//   k_bwd_last     gradient through layer 5 to its input;
//   k_wgrad<CIN,COUT>  weight and bias gradients as contractions over the cells on
//                  the tensor cores (per-block sums, one atomicAdd per weight per
//                  block);
//   k_adam         Adam on the FP32 master weights, then the bf16 copies.
// Layout: activations are channel-last, [cell][16] bf16 (32 bytes per cell) in
// cell space; a neighbour outside the grid reads zero (the tile copies fill zeros there).
#include <cuda_bf16.h>

#include <new>

#include <algorithm>
#include <cmath>
#include <vector>

#include "fs_internal.cuh"

namespace fs {

// parameter offsets in the flat FP32 vector (PyTorch conv3d layout [co][ci][kd][kh][kw])
constexpr int NW1 = 16 * 2 * 27, NB1 = 16, NWM = 16 * 16 * 27, NBM = 16, NW5 = 16 * 27, NB5 = 1;
constexpr int OW1 = 0, OB1 = OW1 + NW1;
constexpr int OW2 = OB1 + NB1, OB2 = OW2 + NWM;
constexpr int OW3 = OB2 + NBM, OB3 = OW3 + NWM;
constexpr int OW4 = OB3 + NBM, OB4 = OW4 + NWM;
constexpr int OW5 = OB4 + NBM, OB5 = OW5 + NW5;
constexpr int NPARAM = OB5 + NB5;

struct NetState {
    float *master;        // FP32 parameters, flat
    float *grad;          // FP32 gradient accumulator, flat
    float *m, *v;         // Adam moments
    float *w1f, *w5f;     // bf16-rounded layer-1 / layer-5 weights as float
    __nv_bfloat16 *wf;    // layers 2-4 forward: [3][27 tap][16 co][16 ci]
    __nv_bfloat16 *wf1;   // layer 1 forward: [27 tap][16 co][16 ci], ci >= 2 zero
    __nv_bfloat16 *wf5;   // layer 5 forward: [27 tap][16 co][16 ci], co >= 1 zero
    int *tlist;           // 32 x 8 x 4 tiles sorted by distance to the liquid (0 .. 5 = farther)
    uint8_t *tdist;       // per 32 x 8 x 1 tile: Chebyshev distance to the nearest liquid cell, capped at 5
    int tcount[6];        // tiles within distance d of the liquid
    int *tlist_tc;        // tiles of the tensor-core layer (TC_M x TC_NY of one plane), sorted the same way
    int tcount_tc[6];
    int kernel;           // inference layers: 0 mma.sync (k_conv), 1 tcgen05 (k_conv_tc)
    long long tlist_epoch;  // mask epoch the list was built for (-1: none)
    double flops;         // of one inference on the cells that each layer must compute (net_flops)
    long long flops_epoch;  // mask epoch it was counted for (-1: none)
    __nv_bfloat16 *wt;    // layers 2-4 backward-data: [3][27 tap][16 ci][16 co], tap flipped
    __nv_bfloat16 *act;   // [6][nC][16]: x (2 ch used), a1, a2, a3, a4, spare
    __nv_bfloat16 *gact;  // [2][nC][16] gradient ping-pong
    float *y;             // [nC] network output (training) / scratch
    float *gy;            // [nC] dL/dy
    unsigned *smax;       // device max |r| (float bits)
    int loaded;
};

namespace {

constexpr int NT_X = 32, NT_Y = 8;  // conv tile: 32 x 8 cells of one plane

__device__ __forceinline__ int tap_index(int dz, int dy, int dx) { return (dz + 1) * 9 + (dy + 1) * 3 + (dx + 1); }

__device__ __forceinline__ bool in_grid(const Layout &L, int i, int j, int k)
{
    return i >= 0 && j >= 0 && k >= 0 && i < L.nx && j < L.ny && k < L.nz;
}

__device__ __forceinline__ int cell_t(const Layout &L, int i, int j, int k) { return L.PL + (k * L.R + j) * L.P + i; }

__device__ __forceinline__ float type_code(uint8_t f) { return (f & CF_LIQ) ? 1.f : ((f & CF_AIR) ? 0.f : -1.f); }

__device__ __forceinline__ float bfr(float x) { return __bfloat162float(__float2bfloat16(x)); }

// ---- the shared tile of the weight gradients -----------------------------------------
// Shared tile: 3 planes x (NT_Y + 2) rows x (NT_X + 2) cells x 16 bf16. The two
// 16-byte halves of a cell are swapped when bit 2 of its tile index is set, so
// the 8 rows of an ldmatrix phase fall in distinct banks.
constexpr int TZ3 = 3, TYH = NT_Y + 2, TXH = NT_X + 2;
constexpr int TCELLS = TZ3 * TYH * TXH;

__device__ __forceinline__ uint32_t swz_off(int cidx, int half)  // byte offset of a cell half
{
    return (uint32_t)(cidx * 32 + ((half ^ ((cidx >> 2) & 1)) << 4));
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

enum : int { IN_ACT = 0, IN_R = 1 };                  // input (tcgen05 layers): bf16 activations / built from r
enum : int { OUT_RELU = 0, OUT_BWD = 1, OUT_Z = 2 };  // epilogue
constexpr unsigned ERR_NET = 8u;  // error word: a bounded wait of a network kernel ran out

struct ConvArgs {
    const __nv_bfloat16 *in;    // IN_ACT: [cell][16]
    const float *r;             // IN_R: right-hand side (cell space)
    const uint8_t *cf;          // cell flags
    const unsigned *smax;       // max |r| over the liquid (float bits)
    const __nv_bfloat16 *wts;   // [27 tap][16 n][16 k]
    const float *bias;          // OUT_RELU: [16]; OUT_Z: [1]
    const __nv_bfloat16 *aref;  // OUT_BWD: the layer input whose ReLU derivative masks
    __nv_bfloat16 *out;         // OUT_RELU, OUT_BWD: [cell][16]
    float *y, *z;               // OUT_Z (each optional): network output; z = s y on liquid, else 0
    const int *tiles;           // optional list of conv tiles (else every tile)
    int ntiles;                 // entries of `tiles`
    const int *done;            // k_conv, k_conv1: return at once when *done != 0 (nullable)
    Layout L;
};

// ---- layers 2-5 and the backward-data pass -----------------------------------------
// OUT_RELU: out = relu(conv(in) + bias). OUT_BWD (backward data): out = conv(in) *
// [aref > 0]. OUT_Z: y = conv(in) + bias, z = s y on liquid cells. Outputs only on
// grid cells.
//
// A block computes 32 x 8 x 4 cells, a warp 16 x 8 cells of one plane: 8 M-tiles of
// 16 cells, one per row, whose sums it holds in registers with the weights of all 27
// taps (108 registers). An input row of a plane is read once per x shift and serves
// the three output rows it touches, so a warp issues 90 ldmatrix for 432 MMAs; with
// one row per warp and the weights read beside the cells it was 108 for 108 (264 us on
// a union of spheres at 256^3; now 154, and the last layer 89 from 240). The tensor pipe
// is active 68 % of the cycles there (the last layer: 53), and two warps per scheduler
// wait for it or for the latency of an MMA most of the rest; L1 moves a third of its
// rate. Per output the taps are summed in the order dz, dy, dx, one MMA each, as before. The
// next tile comes by one tensor copy (zeros off the grid) while this one is worked
// on: with 2 warps per scheduler, cp.async and its index arithmetic in the computing
// warps left the MMA pipe idle half the time. The copy's 32-byte swizzle swaps the
// two halves of a cell when bit 2 of its index is set, so that the 8 rows of an
// ldmatrix phase fall in distinct banks; rows are 36 cells apart, so the swap flips
// with the row's parity. Output channels are dealt to the MMA columns so that a lane
// holds four neighbouring ones and stores 8 bytes.
constexpr int CV_Z = 4, CV_P = 36, CV_PL = CV_P * TYH, CV_CELLS = CV_PL * (CV_Z + 2);
constexpr int CV_BUF = CV_CELLS * 32;                    // bytes of a tile, a multiple of 256
constexpr size_t CV_SMEM = 1024 + 2 * (size_t)CV_BUF;
constexpr unsigned CV_SPIN = 1u << 24;                   // try_wait rounds before a wait gives up
static_assert(CV_P >= TXH && CV_P % 4 == 0 && CV_PL % 8 == 0 && CV_BUF % 256 == 0, "the swizzle of the tile");

// 32 x 8 x 4 tiles of the grid: index (kz * nty + ty) * ntx + tx
__device__ __forceinline__ void conv_tile(int tb, const Layout &L, int &i0, int &j0, int &k0)
{
    const int ntx = (L.nx + NT_X - 1) / NT_X, nty = (L.ny + NT_Y - 1) / NT_Y;
    i0 = (tb % ntx) * NT_X;
    j0 = ((tb / ntx) % nty) * NT_Y;
    k0 = tb / (ntx * nty) * CV_Z;
}

// 16 bytes from global to shared memory, or zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// an mbarrier's phase, waited for within a bound
__device__ __forceinline__ bool bar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity)
{
    for (unsigned n = 0; n < CV_SPIN; n++)
        if (bar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void bar_init(uint32_t bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(1) : "memory");
}

// a box of cells (16 channels, from cell (x, y, z)) global -> shared, completing on `bar`
__device__ __forceinline__ void tma_cells(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar,
                                          uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// the output channel of MMA column n (0 .. 15, two n-tiles of 8)
__device__ __forceinline__ int conv_channel(int n) { return 4 * ((n & 7) >> 1) + (n & 1) + 2 * (n >> 3); }

template <int OUT>
__global__ void __launch_bounds__(256, 1) k_conv(const __grid_constant__ CUtensorMap map,
                                                 const __grid_constant__ ConvArgs a, unsigned *err)
{
    constexpr int NT = OUT == OUT_Z ? 1 : 2;  // n-tiles of 8 output channels
    dep_wait();
    dep_go();
    if (a.done && *(volatile const int *)a.done) return;  // the solve has converged
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t mbar[2];
    const Layout &L = a.L;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int xh = (warp & 1) * 16, pz = warp >> 1;
    const uint32_t sm = ((uint32_t)__cvta_generic_to_shared(smem) + 1023u) & ~1023u;
    const uint32_t bar[2] = {(uint32_t)__cvta_generic_to_shared(mbar), (uint32_t)__cvta_generic_to_shared(mbar + 1)};
    const int total = a.tiles ? a.ntiles : ((L.nx + NT_X - 1) / NT_X) * ((L.ny + NT_Y - 1) / NT_Y) *
                                               ((L.nz + CV_Z - 1) / CV_Z);
    auto tile_at = [&](int idx) { return a.tiles ? __ldg(a.tiles + idx) : idx; };
    auto stage = [&](int idx, int buf) {
        int i0, j0, k0;
        conv_tile(tile_at(idx), L, i0, j0, k0);
        tma_cells(sm + buf * CV_BUF, &map, i0 - 1, j0 - 1, k0 - 1, bar[buf], CV_BUF);
    };
    if (tid == 0) {
        bar_init(bar[0]);
        bar_init(bar[1]);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if ((int)blockIdx.x < total) stage(blockIdx.x, 0);
    }
    uint32_t wreg[27][NT][2];  // lane's B fragments: input channels 2 (lane % 4) + {0, 1} (+ 8) of column lane / 4
#pragma unroll
    for (int tp = 0; tp < 27; tp++)
#pragma unroll
        for (int n = 0; n < NT; n++) {
            const int co = OUT == OUT_Z ? lane >> 2 : conv_channel(8 * n + (lane >> 2));
            const __nv_bfloat16 *w = a.wts + (tp * 16 + co) * 16 + 2 * (lane & 3);
            wreg[tp][n][0] = __ldg(reinterpret_cast<const uint32_t *>(w));
            wreg[tp][n][1] = __ldg(reinterpret_cast<const uint32_t *>(w + 8));
        }
    float bv[4] = {0.f, 0.f, 0.f, 0.f};  // bias of the lane's four channels
    if (OUT == OUT_RELU) {
#pragma unroll
        for (int e = 0; e < 4; e++) bv[e] = a.bias[4 * (lane & 3) + e];
    } else if (OUT == OUT_Z) {
        bv[0] = a.bias[0];
    }
    const float sc = OUT == OUT_Z ? __uint_as_float(*a.smax) : 1.f;
    // the lane's ldmatrix row for each x shift (rows of odd index have the halves swapped)
    uint32_t off[3];
#pragma unroll
    for (int dx = 0; dx < 3; dx++) off[dx] = swz_off(pz * CV_PL + xh + dx + (lane & 15), lane >> 4);
    __syncthreads();
    int buf = 0;
    uint32_t phase = 0;  // bit b: parity of buffer b's next phase
    for (int idx = blockIdx.x; idx < total; idx += gridDim.x, buf ^= 1) {
        if (tid == 0 && idx + (int)gridDim.x < total) stage(idx + gridDim.x, buf ^ 1);
        int i0, j0, k0;
        conv_tile(tile_at(idx), L, i0, j0, k0);
        const bool ok = bar_wait(bar[buf], (phase >> buf) & 1u);
        phase ^= 1u << buf;
        if (__syncthreads_or(!ok)) {  // a copy that never came: note it, wait (bounded) for the one in flight, leave
            if (tid == 0) {
                atomicOr(err, ERR_NET);
                if (idx + (int)gridDim.x < total) bar_wait(bar[buf ^ 1], (phase >> (buf ^ 1)) & 1u);
            }
            __syncthreads();
            break;
        }
        const int gk = k0 + pz;
        if (gk < L.nz) {
            float acc[NT_Y][NT][4];
#pragma unroll
            for (int y = 0; y < NT_Y; y++)
#pragma unroll
                for (int n = 0; n < NT; n++)
#pragma unroll
                    for (int e = 0; e < 4; e++) acc[y][n][e] = 0.f;
            const uint32_t base = sm + buf * CV_BUF;
#pragma unroll
            for (int dz = 0; dz < 3; dz++)
#pragma unroll
                for (int r = 0; r < TYH; r++)
#pragma unroll
                    for (int dx = 0; dx < 3; dx++) {
                        uint32_t a0, a1, a2, a3;
                        ldsm_x4(base + (off[dx] ^ ((r & 1) << 4)) + (dz * CV_PL + r * CV_P) * 32, a0, a1, a2, a3);
#pragma unroll
                        for (int dy = 2; dy >= 0; dy--) {
                            const int y = r - dy, tp = dz * 9 + dy * 3 + dx;
                            if (y < 0 || y >= NT_Y) continue;
#pragma unroll
                            for (int n = 0; n < NT; n++)
                                mma_bf16(acc[y][n], a0, a1, a2, a3, wreg[tp][n][0], wreg[tp][n][1]);
                        }
                    }
            // cells lane / 4 (accumulators 0, 1) and lane / 4 + 8 (2, 3) of each row
            const int gi = i0 + xh + (lane >> 2);
            const size_t t0 = (size_t)cell_t(L, gi, j0, gk);
            if (OUT == OUT_Z) {
                // column 0 sits in one lane of four; the four share the rows (their flags are read at once)
                const int c = lane & 3;
                float y4[2][2];
                uint8_t f4[2][2];
#pragma unroll
                for (int q = 0; q < 2; q++)
#pragma unroll
                    for (int hr = 0; hr < 2; hr++) {
                        float v = 0.f;
#pragma unroll
                        for (int e = 0; e < 4; e++) {
                            const float w = __shfl_sync(0xffffffffu, acc[4 * q + e][0][hr * 2], lane & ~3);
                            if (e == c) v = w;
                        }
                        y4[q][hr] = v + bv[0];
                        const int y = 4 * q + c;
                        f4[q][hr] = gi + hr * 8 < L.nx && j0 + y < L.ny ? __ldg(a.cf + t0 + y * L.P + hr * 8) : 0;
                    }
#pragma unroll
                for (int q = 0; q < 2; q++)
#pragma unroll
                    for (int hr = 0; hr < 2; hr++) {
                        const int y = 4 * q + c;
                        if (gi + hr * 8 >= L.nx || j0 + y >= L.ny) continue;
                        const size_t t = t0 + y * L.P + hr * 8;
                        if (a.y) a.y[t] = y4[q][hr];
                        if (a.z) a.z[t] = (f4[q][hr] & CF_LIQ) ? sc * y4[q][hr] : 0.f;
                    }
            } else {
#pragma unroll
                for (int y2 = 0; y2 < NT_Y; y2 += 2) {
                    uint2 m[2][2];
                    if (OUT == OUT_BWD) {  // four rows' masks in flight before the first store
#pragma unroll
                        for (int y = 0; y < 2; y++)
#pragma unroll
                            for (int hr = 0; hr < 2; hr++)
                                m[y][hr] = gi + hr * 8 < L.nx && j0 + y2 + y < L.ny
                                               ? __ldg(reinterpret_cast<const uint2 *>(
                                                     a.aref + (t0 + (y2 + y) * L.P + hr * 8) * 16 + 4 * (lane & 3)))
                                               : make_uint2(0u, 0u);
                    }
#pragma unroll
                    for (int yy = 0; yy < 2; yy++)
#pragma unroll
                        for (int hr = 0; hr < 2; hr++) {
                            const int y = y2 + yy;
                            if (gi + hr * 8 >= L.nx || j0 + y >= L.ny) continue;
                            float v[4] = {acc[y][0][hr * 2], acc[y][0][hr * 2 + 1], acc[y][NT - 1][hr * 2],
                                          acc[y][NT - 1][hr * 2 + 1]};
                            if (OUT == OUT_RELU) {
#pragma unroll
                                for (int e = 0; e < 4; e++) v[e] = fmaxf(v[e] + bv[e], 0.f);
                            } else {
                                const __nv_bfloat162 m0 = *reinterpret_cast<const __nv_bfloat162 *>(&m[yy][hr].x);
                                const __nv_bfloat162 m1 = *reinterpret_cast<const __nv_bfloat162 *>(&m[yy][hr].y);
                                v[0] = __bfloat162float(m0.x) > 0.f ? v[0] : 0.f;
                                v[1] = __bfloat162float(m0.y) > 0.f ? v[1] : 0.f;
                                v[2] = __bfloat162float(m1.x) > 0.f ? v[2] : 0.f;
                                v[3] = __bfloat162float(m1.y) > 0.f ? v[3] : 0.f;
                            }
                            const __nv_bfloat162 o0 = __floats2bfloat162_rn(v[0], v[1]);
                            const __nv_bfloat162 o1 = __floats2bfloat162_rn(v[2], v[3]);
                            *reinterpret_cast<uint2 *>(a.out + (t0 + y * L.P + hr * 8) * 16 + 4 * (lane & 3)) =
                                make_uint2(*reinterpret_cast<const uint32_t *>(&o0),
                                           *reinterpret_cast<const uint32_t *>(&o1));
                        }
                }
            }
        }
        __syncthreads();  // this buffer is copied into again
    }
}

// ---- layer 1 of inference ------------------------------------------------------------
// The input (bf16(r / s) on liquid, cell-type code) is one 32-bit word per cell, and a
// row of three taps along x is one m16n8k8 MMA: k = 2 dx + channel, so lane l of an A
// fragment reads the word of the cell l % 4 to the right of its row's first tap (the
// fourth has weight zero). 9 MMAs pairs per 16 cells in place of 27 of K = 16 on
// channels padded from 2 to 16 (319 us on a union of spheres at 256^3, most of it the
// padded tile; now 85, with the tensor pipe active 45 % of the cycles and every memory
// below half its rate: four warps per scheduler that wait for an MMA's latency).
__device__ __forceinline__ void mma_bf16_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(b0));
}

// the input word of a cell of flags f and right-hand side r
__device__ __forceinline__ uint32_t net_input(float r, uint8_t f, float inv)
{
    const __nv_bfloat162 x = __floats2bfloat162_rn((f & CF_LIQ) ? r * inv : 0.f, type_code(f));
    return *reinterpret_cast<const uint32_t *>(&x);
}

__global__ void __launch_bounds__(256, 2) k_conv1(const __grid_constant__ ConvArgs a)
{
    dep_wait();
    dep_go();
    if (a.done && *(volatile const int *)a.done) return;  // the solve has converged
    __shared__ uint32_t sx[CV_CELLS];
    const Layout &L = a.L;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int xh = (warp & 1) * 16, pz = warp >> 1;
    uint32_t wreg[9][2];
#pragma unroll
    for (int q = 0; q < 9; q++)
#pragma unroll
        for (int n = 0; n < 2; n++)
            wreg[q][n] = (lane & 3) == 3 ? 0u
                                         : __ldg(reinterpret_cast<const uint32_t *>(
                                               a.wts + ((q * 3 + (lane & 3)) * 16 + conv_channel(8 * n + (lane >> 2))) * 16));
    float bv[4];
#pragma unroll
    for (int e = 0; e < 4; e++) bv[e] = a.bias[4 * (lane & 3) + e];
    const float sc = __uint_as_float(*a.smax);
    const float inv = sc > 0.f ? 1.f / sc : 0.f;
    for (int e = tid; e < CV_CELLS; e += 256) sx[e] = 0u;  // the padding of the rows stays zero
    // the next tile's cells are read into registers while this tile is worked on
    constexpr int PER = ((CV_Z + 2) * TYH * TXH + 255) / 256;
    float rv[PER];
    uint8_t fv[PER];
    // (r by __ldg: its writer is not the launch before, but k_absmax's predecessor, and
    // k_absmax, an ordinary launch, has waited for it)
    auto fetch = [&](int idx) {
        int i0, j0, k0;
        conv_tile(__ldg(a.tiles + idx), L, i0, j0, k0);
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int e = tid + q * 256;
            const int xx = e % TXH, yy = (e / TXH) % TYH, zz = e / (TXH * TYH);
            const int gi = i0 - 1 + xx, gj = j0 - 1 + yy, gk = k0 - 1 + zz;
            const bool in = zz < CV_Z + 2 && in_grid(L, gi, gj, gk);
            const int t = in ? cell_t(L, gi, gj, gk) : 0;
            fv[q] = in ? __ldg(a.cf + t) : 0xff;
            rv[q] = in ? __ldg(a.r + t) : 0.f;
        }
    };
    if ((int)blockIdx.x < a.ntiles) fetch(blockIdx.x);
    for (int idx = blockIdx.x; idx < a.ntiles; idx += gridDim.x) {
        int i0, j0, k0;
        conv_tile(__ldg(a.tiles + idx), L, i0, j0, k0);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int e = tid + q * 256;
            if (e < (CV_Z + 2) * TYH * TXH) {
                const int xx = e % TXH, yy = (e / TXH) % TYH, zz = e / (TXH * TYH);
                sx[zz * CV_PL + yy * CV_P + xx] = fv[q] == 0xff ? 0u : net_input(rv[q], fv[q], inv);
            }
        }
        __syncthreads();
        if (idx + (int)gridDim.x < a.ntiles) fetch(idx + gridDim.x);
        const int gk = k0 + pz;
        if (gk >= L.nz) continue;
        float acc[NT_Y][2][4];
#pragma unroll
        for (int y = 0; y < NT_Y; y++)
#pragma unroll
            for (int n = 0; n < 2; n++)
#pragma unroll
                for (int e = 0; e < 4; e++) acc[y][n][e] = 0.f;
        const uint32_t *row0 = sx + pz * CV_PL + xh + (lane >> 2) + (lane & 3);
#pragma unroll
        for (int dz = 0; dz < 3; dz++)
#pragma unroll
            for (int r = 0; r < TYH; r++) {
                const uint32_t a0 = row0[dz * CV_PL + r * CV_P], a1 = row0[dz * CV_PL + r * CV_P + 8];
#pragma unroll
                for (int dy = 2; dy >= 0; dy--) {
                    const int y = r - dy;
                    if (y < 0 || y >= NT_Y) continue;
#pragma unroll
                    for (int n = 0; n < 2; n++) mma_bf16_k8(acc[y][n], a0, a1, wreg[dz * 3 + dy][n]);
                }
            }
#pragma unroll
        for (int y = 0; y < NT_Y; y++) {
            const int gj = j0 + y;
#pragma unroll
            for (int hr = 0; hr < 2; hr++) {
                const int gi = i0 + xh + (lane >> 2) + hr * 8;
                if (gi >= L.nx || gj >= L.ny) continue;
                const __nv_bfloat162 o0 = __floats2bfloat162_rn(fmaxf(acc[y][0][hr * 2] + bv[0], 0.f),
                                                                fmaxf(acc[y][0][hr * 2 + 1] + bv[1], 0.f));
                const __nv_bfloat162 o1 = __floats2bfloat162_rn(fmaxf(acc[y][1][hr * 2] + bv[2], 0.f),
                                                                fmaxf(acc[y][1][hr * 2 + 1] + bv[3], 0.f));
                *reinterpret_cast<uint2 *>(a.out + (size_t)cell_t(L, gi, gj, gk) * 16 + 4 * (lane & 3)) =
                    make_uint2(*reinterpret_cast<const uint32_t *>(&o0), *reinterpret_cast<const uint32_t *>(&o1));
            }
        }
    }
}

// The network's input on every grid cell, 16 channels (training: layer 1 then runs as
// the others do, and its weight gradient reads it).
__global__ void k_net_x(const float *__restrict__ r, const uint8_t *__restrict__ cf, const unsigned *smax, Layout L,
                        __nv_bfloat16 *x)
{
    const float sc = __uint_as_float(*smax);
    const float inv = sc > 0.f ? 1.f / sc : 0.f;
    for (int t = L.PL + blockIdx.x * blockDim.x + threadIdx.x; t < L.PL + L.S; t += gridDim.x * blockDim.x) {
        uint4 *o = reinterpret_cast<uint4 *>(x + (size_t)t * 16);
        o[0] = make_uint4(net_input(r[t], cf[t], inv), 0u, 0u, 0u);
        o[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// ---- the same layer on the fifth-generation tensor cores (tcgen05, TMEM) ----------
// Inference only. A tile is TC_NY = 2 rows of TC_M = 128 cells along x of one
// plane; each row is one M = 128, N = 16 GEMM over K = 27 taps x 16 channels,
// issued as 27 tcgen05.mma (kind::f16, BF16 inputs, FP32 accumulators in tensor
// memory, one 16-column accumulator per row) by one thread. The input tile (3
// planes x TC_NY + 2 rows x TC_M + 2 cells, 16 channels) is staged in shared
// memory split by channel half: region [plane][row][half][x][8 channels], so that
// a tap's A operand is the same region read from a start shifted by the tap's
// offset, in the canonical K-major layout without swizzling (8-row core matrices
// of 16 bytes per row, 128 bytes apart along M; the second 8 channels TC_HALF
// bytes further along K). The weights of a tap are [half][out channel][8 in
// channels], 512 bytes. Two input buffers alternate: all threads stage the next
// tile while the tensor core works on the current one. The accumulators are read
// back with tcgen05.ld (warp w owns lanes 32 (w % 4) .. + 31 of row w / 4, one
// cell per lane) for the bias, ReLU and bf16 store. Every wait on the MMAs'
// completion is bounded: on timeout the block records an error bit, waits
// (bounded) for its MMAs in flight, frees its tensor memory and stops.
constexpr int TC_M = 128, TC_NY = 2, TC_XW = TC_M + 2, TC_ROWS = TC_NY + 2, TC_THREADS = 256;
constexpr int TC_HALF = TC_XW * 16;                          // 2080 bytes: one channel half of a row
constexpr int TC_ROWB = 2 * TC_HALF;                         // 4160 bytes per (plane, row)
constexpr int TC_A_BYTES = 3 * TC_ROWS * TC_ROWB;            // 49920 per buffer
constexpr int TC_B_BYTES = 27 * 512;                         // 13824
constexpr size_t TC_SMEM = 128 + 2 * (size_t)TC_A_BYTES + TC_B_BYTES;
constexpr unsigned TC_SPIN = 1u << 24;
static_assert(TC_THREADS == 2 * TC_M, "one thread per accumulator row lane in the epilogue");

__device__ __forceinline__ uint32_t tc_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte
// offsets in units of 16 bytes, descriptor version 1, no swizzling
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulate (bits 4-5 = 1), A and B
// BF16 (bits 7-9 = 1, 10-12 = 1), both K-major, N >> 3 at bits 17-22, M >> 4 at
// bits 24-28
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(16 >> 3) << 17) |
                              ((uint32_t)(TC_M >> 4) << 24);

__device__ __forceinline__ void tc_mma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate)
{
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(TC_IDESC), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ bool tc_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// 16 FP32 columns of the warp's lane quarter, one lane per thread
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 16; k++) v[k] = __uint_as_float(r[k]);
}

// tiles of the tensor-core layer: TC_M x TC_NY cells of one plane, index
// (k * ntyc + ty) * ntxc + tx
__device__ __forceinline__ void tc_tile(int tb, const Layout &L, int &i0, int &j0, int &k)
{
    const int ntxc = (L.nx + TC_M - 1) / TC_M, ntyc = (L.ny + TC_NY - 1) / TC_NY;
    i0 = (tb % ntxc) * TC_M;
    j0 = ((tb / ntxc) % ntyc) * TC_NY;
    k = tb / (ntxc * ntyc);
}

// stage the input tile of tile tb into sa: plane kz - 1 + pz, row j0 - 1 + ry,
// cell i0 - 1 + x, both channel halves
template <int IN>
__device__ __forceinline__ void tc_stage(const ConvArgs &a, int tb, unsigned char *sa, float inv)
{
    const Layout &L = a.L;
    int i0, j0, kz;
    tc_tile(tb, L, i0, j0, kz);
    for (int e = threadIdx.x; e < 3 * TC_ROWS * TC_XW; e += blockDim.x) {
        const int x = e % TC_XW, ry = (e / TC_XW) % TC_ROWS, pz = e / (TC_XW * TC_ROWS);
        const int gi = i0 - 1 + x, gj = j0 - 1 + ry, gk = kz - 1 + pz;
        uint4 h0 = make_uint4(0u, 0u, 0u, 0u), h1 = h0;
        if (in_grid(L, gi, gj, gk)) {
            const int t = cell_t(L, gi, gj, gk);
            if (IN == IN_ACT) {
                h0 = __ldg(reinterpret_cast<const uint4 *>(a.in + (size_t)t * 16));
                h1 = __ldg(reinterpret_cast<const uint4 *>(a.in + (size_t)t * 16) + 1);
            } else {
                const uint8_t f = a.cf[t];
                const __nv_bfloat162 xv = __floats2bfloat162_rn((f & CF_LIQ) ? a.r[t] * inv : 0.f, type_code(f));
                h0.x = *reinterpret_cast<const uint32_t *>(&xv);
            }
        }
        unsigned char *row = sa + (pz * TC_ROWS + ry) * TC_ROWB + x * 16;
        *reinterpret_cast<uint4 *>(row) = h0;
        *reinterpret_cast<uint4 *>(row + TC_HALF) = h1;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor core
}

template <int IN, int OUT>
__global__ void __launch_bounds__(TC_THREADS) k_conv_tc(ConvArgs a, unsigned *err)
{
    extern __shared__ __align__(128) unsigned char smem_tc[];
    unsigned char *base = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_tc) + 127) & ~(uintptr_t)127);
    unsigned char *sa[2] = {base, base + TC_A_BYTES};  // input tiles, alternating
    unsigned char *sb = base + 2 * TC_A_BYTES;          // weights
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int stop;
    const Layout &L = a.L;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // weights: [tap][half][co][8 ci] from [tap][co][16 ci]
    for (int e = tid; e < 27 * 16 * 2; e += blockDim.x) {
        const int tap = e >> 5, co = (e >> 1) & 15, half = e & 1;
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(a.wts) + (tap * 16 + co) * 2 + half);
        *reinterpret_cast<uint4 *>(sb + tap * 512 + half * 256 + co * 16) = v;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(&tmem_base)),
                     "r"(32)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem(&mbar)), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        stop = 0;
    }
    float bv[16];
#pragma unroll
    for (int k = 0; k < 16; k++) bv[k] = 0.f;
    if (OUT == OUT_RELU) {
#pragma unroll
        for (int k = 0; k < 16; k++) bv[k] = a.bias[k];
    } else {
        bv[0] = a.bias[0];
    }
    float sc = 1.f, inv = 0.f;
    if (IN == IN_R || OUT == OUT_Z) {
        sc = __uint_as_float(*a.smax);
        inv = sc > 0.f ? 1.f / sc : 0.f;
    }
    const int ntxc = (L.nx + TC_M - 1) / TC_M, ntyc = (L.ny + TC_NY - 1) / TC_NY;
    const int total = a.tiles ? a.ntiles : ntxc * ntyc * L.nz;
    auto tile_at = [&](int idx) { return a.tiles ? __ldg(a.tiles + idx) : idx; };
    if ((int)blockIdx.x < total) tc_stage<IN>(a, tile_at(blockIdx.x), sa[0], inv);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const uint32_t sb_u = tc_smem(sb), bar_u = tc_smem(&mbar);
    uint32_t phase = 0;
    int buf = 0;
    for (int idx = blockIdx.x; idx < total; idx += gridDim.x, buf ^= 1) {
        int i0, j0, kz;
        tc_tile(tile_at(idx), L, i0, j0, kz);
        if (tid == 0) {
            const uint32_t sa_u = tc_smem(sa[buf]);
#pragma unroll 1
            for (int yr = 0; yr < TC_NY; yr++) {
#pragma unroll 1
                for (int tap = 0; tap < 27; tap++) {
                    const int dz = tap / 9, dy = (tap / 3) % 3, dx = tap % 3;
                    const uint32_t aaddr = sa_u + (uint32_t)((dz * TC_ROWS + yr + dy) * TC_ROWB + dx * 16);
                    tc_mma(tmem + (uint32_t)(16 * yr), tc_desc(aaddr, TC_HALF, 128), tc_desc(sb_u + tap * 512, 256, 128),
                           tap > 0 ? 1u : 0u);
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_u)
                         : "memory");
        }
        // the next tile into the other buffer while the tensor core works
        if (idx + (int)gridDim.x < total) tc_stage<IN>(a, tile_at(idx + gridDim.x), sa[buf ^ 1], inv);
        bool ok = false;
        for (unsigned n = 0; n < TC_SPIN && !ok; n++) ok = tc_try_wait(bar_u, phase);
        if (!ok) {
            if (lane == 0) atomicOr(err, ERR_NET);
            stop = 1;
        }
        phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncthreads();
        if (stop) break;
        // epilogue: warp w reads lanes 32 (w % 4) .. + 31 of row w / 4
        {
            const int yr = warp >> 2, q = warp & 3;
            float acc[16];
            tc_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(16 * yr), acc);
            const int gi = i0 + 32 * q + lane, gj = j0 + yr;
            if (gi < L.nx && gj < L.ny) {
                const size_t t = (size_t)cell_t(L, gi, gj, kz);
                if (OUT == OUT_Z) {
                    const float yv = acc[0] + bv[0];
                    if (a.y) a.y[t] = yv;
                    if (a.z) a.z[t] = (a.cf[t] & CF_LIQ) ? sc * yv : 0.f;
                } else {
                    uint32_t pk[8];
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        const __nv_bfloat162 b2 = __floats2bfloat162_rn(fmaxf(acc[2 * k] + bv[2 * k], 0.f),
                                                                        fmaxf(acc[2 * k + 1] + bv[2 * k + 1], 0.f));
                        pk[k] = *reinterpret_cast<const uint32_t *>(&b2);
                    }
                    uint4 *o = reinterpret_cast<uint4 *>(a.out + t * 16);
                    o[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    o[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                }
            }
        }
        // the accumulators read and the next buffer staged before the next MMAs
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (stop) {  // the MMAs of a timed-out tile may still run: wait for them again (bounded) before freeing
        bool ok = false;
        for (unsigned n = 0; n < TC_SPIN && !ok; n++) ok = tc_try_wait(bar_u, phase ^ 1u);
    }
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(32) : "memory");
}

// Chebyshev distance from each conv tile (32 x 8 cells of one plane) to the
// nearest liquid cell, capped at 5: one block per tile scans the tile grown by 5.
__global__ void __launch_bounds__(256) k_conv_tile_dist(const uint8_t *__restrict__ cf, Layout L, uint8_t *dist)
{
    __shared__ int best;
    const int ntx = (L.nx + NT_X - 1) / NT_X, nty = (L.ny + NT_Y - 1) / NT_Y;
    const int tb = blockIdx.x;
    const int tx = tb % ntx, ty = (tb / ntx) % nty, tk = tb / (ntx * nty);
    const int i0 = tx * NT_X, j0 = ty * NT_Y;
    if (threadIdx.x == 0) best = 5;
    __syncthreads();
    const int bx = NT_X + 10, by = NT_Y + 10, bz = 11;
    int d = 5;
    for (int e = threadIdx.x; e < bx * by * bz; e += blockDim.x) {
        const int gi = i0 - 5 + e % bx, gj = j0 - 5 + (e / bx) % by, gk = tk - 5 + e / (bx * by);
        if (!in_grid(L, gi, gj, gk) || !(cf[cell_t(L, gi, gj, gk)] & CF_LIQ)) continue;
        const int dx = max(0, max(i0 - gi, gi - (i0 + NT_X - 1)));
        const int dy = max(0, max(j0 - gj, gj - (j0 + NT_Y - 1)));
        const int dz = abs(gk - tk);
        d = min(d, max(dx, max(dy, dz)));
    }
    if (d < 5) atomicMin(&best, d);
    __syncthreads();
    if (threadIdx.x == 0) dist[tb] = (uint8_t)best;
}

// The cells of the grid within Chebyshev distance d of the liquid -> count[d], d = 0 .. 4
// (once per mask, for the profiled flops).
__global__ void __launch_bounds__(256) k_net_reach(const uint8_t *__restrict__ cf, Layout L, unsigned long long *count)
{
    const int ncell = L.nx * L.ny * L.nz;
    unsigned long long near[5] = {0, 0, 0, 0, 0};
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ncell; e += gridDim.x * blockDim.x) {
        const int i = e % L.nx, j = (e / L.nx) % L.ny, k = e / (L.nx * L.ny);
        int d = cf[cell_t(L, i, j, k)] & CF_LIQ ? 0 : 5;
        for (int z = -4; z <= 4 && d > 0; z++)
            for (int y = -4; y <= 4; y++)
                for (int x = -4; x <= 4; x++) {
                    const int far = max(abs(z), max(abs(y), abs(x)));
                    if (far < d && in_grid(L, i + x, j + y, k + z) && (cf[cell_t(L, i + x, j + y, k + z)] & CF_LIQ))
                        d = far;
                }
#pragma unroll
        for (int q = 0; q < 5; q++) near[q] += d <= q;
    }
#pragma unroll
    for (int q = 0; q < 5; q++) {
        for (int o = 16; o > 0; o >>= 1) near[q] += __shfl_xor_sync(0xffffffffu, near[q], o);
        if ((threadIdx.x & 31) == 0 && near[q]) atomicAdd(count + q, near[q]);
    }
}

// max |r| over the liquid, as float bits (non-negative floats order like ints), over
// the list of quads that hold liquid (r is zero on their other cells)
__global__ void __launch_bounds__(256) k_absmax(const int *__restrict__ ql, int nq, const float *__restrict__ r,
                                                unsigned *smax, const int *done)
{
    if (done && *(volatile const int *)done) return;  // the solve has converged
    float m = 0.f;
    FS_FOR_LIST(ql, nq)
    {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(r) + q);
        m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(smax, __float_as_uint(m));
}

// s is rounded to bf16 (the oracle rounds x = r/s, not s; keep s exact)
// ---- training: loss, gradients -----------------------------------------------------

// Energy-norm loss (y - q/s)^T A (y - q/s) / ((q/s)^T A (q/s)), A the pressure
// operator. Pass 1: e = y - q/s and t = q/s on liquid cells (zero elsewhere).
__global__ void k_net_err(const float *__restrict__ y, const float *__restrict__ q, const uint8_t *__restrict__ cf,
                          const unsigned *__restrict__ smax, float *e, float *tq, int n)
{
    const float sc = __uint_as_float(*smax);
    const float inv = sc > 0.f ? 1.f / sc : 0.f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const bool liq = (cf[t] & CF_LIQ) != 0;
        const float tv = liq ? q[t] * inv : 0.f;
        tq[t] = tv;
        e[t] = liq ? y[t] - tv : 0.f;
    }
}

// Pass 2: Ae (kept for the gradient), e.Ae and t.At -> aux[0], aux[1].
__global__ void __launch_bounds__(256) k_net_energy(const float *__restrict__ e, const float *__restrict__ tq,
                                                    float *ae, const uint8_t *__restrict__ cf, Layout L,
                                                    SolveScal *s, double *partials)
{
    double num = 0.0, den = 0.0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < L.nC; t += gridDim.x * blockDim.x) {
        const uint8_t f = cf[t];
        if (!(f & CF_LIQ)) continue;
        const float d = (float)(f & CF_D);
        const float av = d * e[t] - ((e[t - 1] + e[t + 1]) + (e[t - L.P] + e[t + L.P]) + (e[t - L.PL] + e[t + L.PL]));
        const float at = d * tq[t] - ((tq[t - 1] + tq[t + 1]) + (tq[t - L.P] + tq[t + L.P]) +
                                      (tq[t - L.PL] + tq[t + L.PL]));
        ae[t] = av;
        num += (double)e[t] * av;
        den += (double)tq[t] * at;
    }
    double v[2] = {num, den}, tot[2];
    if (grid_reduce<2>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        s->aux[0] = tot[0];
        s->aux[1] = tot[1];
    }
}

// Pass 3: dloss/dy = 2 A e / den on liquid cells.
__global__ void k_net_gy(const float *__restrict__ ae, const uint8_t *__restrict__ cf, const SolveScal *s, float *gy,
                         int n)
{
    const double den = s->aux[1];
    const float g = den > 0.0 ? (float)(2.0 / den) : 0.f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
        gy[t] = (cf[t] & CF_LIQ) ? g * ae[t] : 0.f;
}

// ---- the loss of the network followed by the V-cycle (FS_PRECOND_LEARNED_MG) ----
// With y the network output (masked to the liquid), b/s and q/s the scaled pair
// and M the V-cycle: w = q/s - y - M(b/s - A y), loss = w.A w / (q/s).A (q/s).
// w = (I - M A)(q/s - y), so dloss/dy = -2 (I - A M) A w / den, M and A symmetric.

// ym = y on liquid cells, 0 elsewhere
__global__ void k_net_mask_y(const float *__restrict__ y, const uint8_t *__restrict__ cf, float *ym, int n)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
        ym[t] = (cf[t] & CF_LIQ) ? y[t] : 0.f;
}

// t1 = b/s - A ym on liquid cells (the residual the network leaves), 0 elsewhere
__global__ void __launch_bounds__(256) k_netmg_res(const float *__restrict__ b, const float *__restrict__ ym,
                                                   const uint8_t *__restrict__ cf, const unsigned *__restrict__ smax,
                                                   Layout L, float *t1)
{
    const float sc = __uint_as_float(*smax);
    const float inv = sc > 0.f ? 1.f / sc : 0.f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < L.nC; t += gridDim.x * blockDim.x) {
        const uint8_t f = cf[t];
        float v = 0.f;
        if (f & CF_LIQ) {
            const float ay = (float)(f & CF_D) * ym[t] -
                             ((ym[t - 1] + ym[t + 1]) + (ym[t - L.P] + ym[t + L.P]) + (ym[t - L.PL] + ym[t + L.PL]));
            v = b[t] * inv - ay;
        }
        t1[t] = v;
    }
}

// w = q/s - ym - m and tq = q/s on liquid cells, 0 elsewhere
__global__ void k_netmg_err(const float *__restrict__ q, const float *__restrict__ ym, const float *__restrict__ m,
                            const uint8_t *__restrict__ cf, const unsigned *__restrict__ smax, float *w, float *tq,
                            int n)
{
    const float sc = __uint_as_float(*smax);
    const float inv = sc > 0.f ? 1.f / sc : 0.f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const bool liq = (cf[t] & CF_LIQ) != 0;
        const float tv = liq ? q[t] * inv : 0.f;
        tq[t] = tv;
        w[t] = liq ? tv - ym[t] - m[t] : 0.f;
    }
}

// dloss/dy = -2 (v - A u) / den on liquid cells, v = A w, u = M v
__global__ void __launch_bounds__(256) k_netmg_gy(const float *__restrict__ v, const float *__restrict__ u,
                                                  const uint8_t *__restrict__ cf, const SolveScal *s, Layout L,
                                                  float *gy)
{
    const double den = s->aux[1];
    const float g = den > 0.0 ? (float)(-2.0 / den) : 0.f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < L.nC; t += gridDim.x * blockDim.x) {
        const uint8_t f = cf[t];
        float o = 0.f;
        if (f & CF_LIQ) {
            const float au = (float)(f & CF_D) * u[t] -
                             ((u[t - 1] + u[t + 1]) + (u[t - L.P] + u[t + L.P]) + (u[t - L.PL] + u[t + L.PL]));
            o = g * (v[t] - au);
        }
        gy[t] = o;
    }
}

// dL/d(layer-5 input) = sum_tap w5[ci][tap] gy[cell - tap], times [a4 > 0]
__global__ void __launch_bounds__(256) k_bwd_last(const float *__restrict__ gy, const float *__restrict__ w5f,
                                                  const __nv_bfloat16 *__restrict__ a4, __nv_bfloat16 *g4, Layout L)
{
    __shared__ float w[NW5];
    for (int t = threadIdx.x; t < NW5; t += blockDim.x) w[t] = w5f[t];
    __syncthreads();
    const int ncell = L.nx * L.ny * L.nz;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        const int i = c % L.nx, j = (c / L.nx) % L.ny, k = c / (L.nx * L.ny);
        float acc[16];
#pragma unroll
        for (int o = 0; o < 16; o++) acc[o] = 0.f;
        for (int dz = -1; dz <= 1; dz++)
            for (int dy = -1; dy <= 1; dy++)
                for (int dx = -1; dx <= 1; dx++) {
                    // output cell (i - d) saw this cell through tap d
                    if (!in_grid(L, i - dx, j - dy, k - dz)) continue;
                    const float g = gy[cell_t(L, i - dx, j - dy, k - dz)];
                    if (g == 0.f) continue;
                    const int tp = tap_index(dz, dy, dx);
#pragma unroll
                    for (int o = 0; o < 16; o++) acc[o] += w[o * 27 + tp] * g;
                }
        const size_t t = (size_t)cell_t(L, i, j, k);
        const __nv_bfloat162 *a = reinterpret_cast<const __nv_bfloat162 *>(a4 + t * 16);
        __nv_bfloat162 *o2 = reinterpret_cast<__nv_bfloat162 *>(g4 + t * 16);
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const float2 av = __bfloat1622float2(a[q]);
            o2[q] = __floats2bfloat162_rn(av.x > 0.f ? acc[2 * q] : 0.f, av.y > 0.f ? acc[2 * q + 1] : 0.f);
        }
    }
}

// Weight and bias gradients of one layer: gW[co][ci][tap] += sum_cells
// g[cell][co] * a[cell + tap][ci]; gB[co] += sum_cells g[cell][co]. g is bf16
// [cell][16] (COUT = 16) or FP32 [cell] (COUT = 1); a is bf16 [cell][16], of which
// the first CIN channels count.
//
// A contraction over the cells: per tap M = 16 output channels, N = 16 (or 8)
// input channels, K = cells, on mma.sync m16n8k16 (bf16 products, FP32 sums). A
// tile is 32 x 8 cells of one plane; warp w takes the taps of dz = w / 4 on rows
// 2 (w % 4) and the next, whose g operand it loads once per 16 cells for its nine
// taps. Each tile's sums start from zero and are added to FP32 totals in
// registers, as few terms in a row as before (a tile had been one chain of 256).
// An FP32 g (the last layer) enters as three bf16 rows of M whose sum it is
// exactly (8 + 8 + 8 significant bits). The next tile is copied (cp.async) while
// this one is worked on. At 64^3 a 16 x 16 layer takes 27 us (FP32 cores, one
// thread per weight walking the tile's cells: 3.09 ms), the last layer 26 (247).
// One block of 12 warps fits an SM (its registers, and its copies of the tiles with
// halo, 4 times the cells): the tensor pipe is active 25 % of the cycles, instructions
// issue on 45 %, and warps wait for ldmatrix, an MMA's latency or the barrier.
constexpr int WG_TH = 384;
constexpr int WG_A = TCELLS * 32, WG_G = NT_X * NT_Y * 32;  // bytes of a tile's two operands
constexpr size_t WG_SMEM = 2 * (size_t)(WG_A + WG_G);

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

template <int CIN, int COUT, bool GF32>
__global__ void __launch_bounds__(WG_TH, 1) k_wgrad(const void *__restrict__ gptr, const __nv_bfloat16 *__restrict__ a,
                                                    float *gW, float *gB, Layout L)
{
    constexpr int NB = CIN > 8 ? 2 : 1;  // tiles of 8 input channels
    extern __shared__ __align__(128) unsigned char wg_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int dz = warp >> 2, y0 = 2 * (warp & 3);
    const int ntx = (L.nx + NT_X - 1) / NT_X, nty = (L.ny + NT_Y - 1) / NT_Y;
    const int ntiles = ntx * nty * L.nz;
    auto stage = [&](int tb, unsigned char *buf) {
        const int tx = tb % ntx, ty = (tb / ntx) % nty, tk = tb / (ntx * nty);
        const int i0 = tx * NT_X, j0 = ty * NT_Y;
        const uint32_t sa = (uint32_t)__cvta_generic_to_shared(buf), sg = sa + WG_A;
        for (int e = tid; e < TCELLS * 2; e += WG_TH) {
            const int cidx = e >> 1, half = e & 1;
            const int xx = cidx % TXH, yy = (cidx / TXH) % TYH, zz = cidx / (TXH * TYH);
            const int gi = i0 - 1 + xx, gj = j0 - 1 + yy, gk = tk - 1 + zz;
            const bool in = in_grid(L, gi, gj, gk);
            const int t = in ? cell_t(L, gi, gj, gk) : L.PL;
            cp_async16(sa + swz_off(cidx, half), a + (size_t)t * 16 + half * 8, in);
        }
        if (!GF32) {
            for (int e = tid; e < NT_X * NT_Y * 2; e += WG_TH) {
                const int cl = e >> 1, half = e & 1;
                const int gi = i0 + cl % NT_X, gj = j0 + cl / NT_X;
                const bool in = gi < L.nx && gj < L.ny;
                const int t = in ? cell_t(L, gi, gj, tk) : L.PL;
                cp_async16(sg + swz_off(cl, half), static_cast<const __nv_bfloat16 *>(gptr) + (size_t)t * 16 + half * 8,
                           in);
            }
        } else {  // rows 0, 1, 2 of M: the leading, middle and last bf16 of g
            for (int cl = tid; cl < NT_X * NT_Y; cl += WG_TH) {
                const int gi = i0 + cl % NT_X, gj = j0 + cl / NT_X;
                const float g = gi < L.nx && gj < L.ny ? static_cast<const float *>(gptr)[cell_t(L, gi, gj, tk)] : 0.f;
                const __nv_bfloat16 h = __float2bfloat16(g);
                const float g1 = g - __bfloat162float(h);
                const __nv_bfloat16 m = __float2bfloat16(g1);
                const __nv_bfloat16 l = __float2bfloat16(g1 - __bfloat162float(m));
                __nv_bfloat162 hm, lz;
                hm.x = h;
                hm.y = m;
                lz.x = l;
                lz.y = __float2bfloat16(0.f);
                unsigned char *dst = buf + WG_A;
                *reinterpret_cast<uint4 *>(dst + swz_off(cl, 0)) =
                    make_uint4(*reinterpret_cast<uint32_t *>(&hm), *reinterpret_cast<uint32_t *>(&lz), 0u, 0u);
                *reinterpret_cast<uint4 *>(dst + swz_off(cl, 1)) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        cp_async_commit();
    };
    float tot[9][NB][4], btot[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int p = 0; p < 9; p++)
#pragma unroll
        for (int n = 0; n < NB; n++)
#pragma unroll
            for (int e = 0; e < 4; e++) tot[p][n][e] = 0.f;
    const uint32_t one2 = 0x3f803f80u;  // two bf16 ones: the bias sums g itself
    int buf = 0;
    if ((int)blockIdx.x < ntiles) stage(blockIdx.x, wg_smem);
    for (int tb = blockIdx.x; tb < ntiles; tb += gridDim.x, buf ^= 1) {
        if (tb + (int)gridDim.x < ntiles) {
            stage(tb + gridDim.x, wg_smem + (buf ^ 1) * (WG_A + WG_G));
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const uint32_t sa = (uint32_t)__cvta_generic_to_shared(wg_smem + buf * (WG_A + WG_G)), sg = sa + WG_A;
        float acc[9][NB][4], bacc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int p = 0; p < 9; p++)
#pragma unroll
            for (int n = 0; n < NB; n++)
#pragma unroll
                for (int e = 0; e < 4; e++) acc[p][n][e] = 0.f;
#pragma unroll 1
        for (int ch = 0; ch < 4; ch++) {  // two rows of two groups of 16 cells
            const int y = y0 + (ch >> 1), x = (ch & 1) * 16;
            // g transposed: matrices (cells 0-7, channels 0-7), (0-7, 8-15), (8-15, 0-7), (8-15, 8-15)
            uint32_t g0, g1, g2, g3;
            {
                const int cl = y * NT_X + x + (lane & 7) + ((lane >> 4) << 3);
                ldsm_x4_t(sg + swz_off(cl, (lane >> 3) & 1), g0, g1, g2, g3);
            }
            if (dz == 0) mma_bf16(bacc, g0, g1, g2, g3, one2, one2);
#pragma unroll
            for (int p = 0; p < 9; p++) {
                // a: matrices (cells 0-7, channels 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15)
                const int cidx = (dz * TYH + y + p / 3) * TXH + x + p % 3 + (lane & 15);
                uint32_t b0, b1, b2, b3;
                ldsm_x4_t(sa + swz_off(cidx, lane >> 4), b0, b1, b2, b3);
                mma_bf16(acc[p][0], g0, g1, g2, g3, b0, b1);
                if (NB == 2) mma_bf16(acc[p][NB - 1], g0, g1, g2, g3, b2, b3);
            }
        }
#pragma unroll
        for (int p = 0; p < 9; p++)
#pragma unroll
            for (int n = 0; n < NB; n++)
#pragma unroll
                for (int e = 0; e < 4; e++) tot[p][n][e] += acc[p][n][e];
#pragma unroll
        for (int e = 0; e < 4; e++) btot[e] += bacc[e];
        __syncthreads();  // this buffer is staged again
    }
    // the four warps of a dz added in order, then one atomic per weight and block
    constexpr int PER = 9 * NB * 4 + 4;
    float *red = reinterpret_cast<float *>(wg_smem);  // [3 dz][PER][32]
    for (int w = 0; w < 4; w++) {
        if ((warp & 3) == w) {
            float *r = red + (size_t)dz * PER * 32 + lane;
#pragma unroll
            for (int p = 0; p < 9; p++)
#pragma unroll
                for (int n = 0; n < NB; n++)
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        float &v = r[((p * NB + n) * 4 + e) * 32];
                        v = w ? v + tot[p][n][e] : tot[p][n][e];
                    }
#pragma unroll
            for (int e = 0; e < 4; e++) {
                float &v = r[(9 * NB * 4 + e) * 32];
                v = w ? v + btot[e] : btot[e];
            }
        }
        __syncthreads();
    }
    // accumulator element e of lane l: row l / 4 (+ 8 for e >= 2), column 2 (l % 4) + (e & 1)
    auto sum_at = [&](int z, int slot, int row, int col) {
        const int e = ((row >> 3) << 1) | (col & 1), l = (row & 7) * 4 + (col >> 1);
        return red[((size_t)z * PER + slot * 4 + e) * 32 + l];
    };
    for (int o = tid; o < COUT * CIN * 27; o += WG_TH) {
        const int tp = o % 27, ci = (o / 27) % CIN, co = o / (27 * CIN);
        const int slot = (tp % 9) * NB + (ci >> 3);
        float v = sum_at(tp / 9, slot, co, ci & 7);
        if (GF32) v += sum_at(tp / 9, slot, 1, ci & 7) + sum_at(tp / 9, slot, 2, ci & 7);
        atomicAdd(gW + o, v);
    }
    if (tid < COUT) {
        float v = sum_at(0, 9 * NB, tid, 0);
        if (GF32) v += sum_at(0, 9 * NB, 1, 0) + sum_at(0, 9 * NB, 2, 0);
        atomicAdd(gB + tid, v);
    }
}

// A parameter that does not depend on the residual: a bias, or a weight of the
// cell-type input channel (W1[co][1][tap]).
__device__ __forceinline__ bool offset_param(int t)
{
    if (t < OB1) return (t / 27) % 2 == 1;
    return (t >= OB1 && t < OW2) || (t >= OB2 && t < OW3) || (t >= OB3 && t < OW4) || (t >= OB4 && t < OW5) ||
           t >= OB5;
}

// Adam on the FP32 master copy; the gradient buffer is cleared. With
// `fix_offsets` the offset parameters keep their values.
__global__ void k_adam(float *p, float *g, float *m, float *v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2, float gscale, int fix_offsets)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        if (fix_offsets && offset_param(t)) {
            g[t] = 0.f;
            continue;
        }
        const float gr = g[t] * gscale;
        const float mm = b1 * m[t] + (1.f - b1) * gr;
        const float vv = b2 * v[t] + (1.f - b2) * gr * gr;
        m[t] = mm;
        v[t] = vv;
        p[t] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
        g[t] = 0.f;
    }
}

// bf16 working copies from the master copy
__global__ void k_net_refresh(const float *__restrict__ p, float *w1f, float *w5f, __nv_bfloat16 *wf,
                              __nv_bfloat16 *wt, __nv_bfloat16 *wf1, __nv_bfloat16 *wf5)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < NPARAM; t += gridDim.x * blockDim.x) {
        if (t < OB1) {
            w1f[t] = bfr(p[t]);
            const int tp = t % 27, ci = (t / 27) % 2, co = t / 54;  // [co][ci][tap]
            wf1[(tp * 16 + co) * 16 + ci] = __float2bfloat16(p[t]);
        }
        if (t >= OW5 && t < OB5) {
            w5f[t - OW5] = bfr(p[t]);
            const int tp = (t - OW5) % 27, ci = (t - OW5) / 27;    // [1][ci][tap]
            wf5[(tp * 16 + 0) * 16 + ci] = __float2bfloat16(p[t]);
        }
        const int offs[3] = {OW2, OW3, OW4};
        for (int l = 0; l < 3; l++) {
            if (t < offs[l] || t >= offs[l] + NWM) continue;
            const int e = t - offs[l];
            const int tp = e % 27, ci = (e / 27) % 16, co = e / (27 * 16);
            const __nv_bfloat16 v = __float2bfloat16(p[t]);
            wf[(size_t)l * NWM + (tp * 16 + co) * 16 + ci] = v;            // [tap][n = co][k = ci]
            wt[(size_t)l * NWM + ((26 - tp) * 16 + ci) * 16 + co] = v;     // [tap'][n = ci][k = co]
        }
    }
}

__global__ void k_fill_zero(float *p, int n)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) p[t] = 0.f;
}

}  // namespace

static NetState *net(fs_ctx *c) { return static_cast<NetState *>(c->net); }

// 32 x 8 tiles of one plane, and 32 x 8 x 4 tiles
static int plane_tiles(const Layout &L) { return ((L.nx + NT_X - 1) / NT_X) * ((L.ny + NT_Y - 1) / NT_Y) * L.nz; }
static int conv_tiles(const Layout &L)
{
    return ((L.nx + NT_X - 1) / NT_X) * ((L.ny + NT_Y - 1) / NT_Y) * ((L.nz + CV_Z - 1) / CV_Z);
}

static int conv_tiles_tc(const Layout &L)
{
    return ((L.nx + TC_M - 1) / TC_M) * ((L.ny + TC_NY - 1) / TC_NY) * L.nz;
}

int net_alloc(fs_ctx *c, bool training)
{
    if (c->net && (!training || net(c)->gact)) return FS_OK;
    NetState *n = net(c);
    if (!n) {
        n = new (std::nothrow) NetState();
        if (!n) return set_error(FS_ENOMEM, "host allocation failed");
        n->tlist_epoch = n->flops_epoch = -1;
        c->net = n;
    }
    auto alloc = [&](void **p, size_t bytes) -> int {
        if (*p) return FS_OK;
        cudaError_t e = cudaMalloc(p, bytes);
        if (e != cudaSuccess) {
            *p = nullptr;
            cudaGetLastError();
            return set_error(FS_ENOMEM, "cudaMalloc of %zu bytes failed", bytes);
        }
        return check_cuda(cudaMemset(*p, 0, bytes), "cudaMemset");
    };
    const size_t nC = (size_t)c->L.nC;
    int rc;
    if ((rc = alloc((void **)&n->master, NPARAM * 4)) || (rc = alloc((void **)&n->grad, NPARAM * 4)) ||
        (rc = alloc((void **)&n->m, NPARAM * 4)) || (rc = alloc((void **)&n->v, NPARAM * 4)) ||
        (rc = alloc((void **)&n->w1f, NW1 * 4)) || (rc = alloc((void **)&n->w5f, NW5 * 4)) ||
        (rc = alloc((void **)&n->wf, 3 * NWM * 2)) || (rc = alloc((void **)&n->wt, 3 * NWM * 2)) ||
        (rc = alloc((void **)&n->smax, 16)) || (rc = alloc((void **)&n->y, nC * 4)) ||
        (rc = alloc((void **)&n->wf1, 27 * 16 * 16 * 2)) || (rc = alloc((void **)&n->wf5, 27 * 16 * 16 * 2)) ||
        (rc = alloc((void **)&n->tdist, (size_t)plane_tiles(c->L))) ||
        (rc = alloc((void **)&n->tlist, (size_t)conv_tiles(c->L) * sizeof(int))) ||
        (rc = alloc((void **)&n->tlist_tc, (size_t)conv_tiles_tc(c->L) * sizeof(int))))
        return rc;
    // inference needs two activation buffers; training keeps all five layer inputs
    const int nact = training ? 6 : 2;
    if (training && n->act && !n->gact) {
        cudaFree(n->act);
        n->act = nullptr;
    }
    if ((rc = alloc((void **)&n->act, nact * nC * 32))) return rc;
    if (training) {
        if ((rc = alloc((void **)&n->gact, 2 * nC * 32)) || (rc = alloc((void **)&n->gy, nC * 4))) return rc;
    }
    static bool attr_done = false;
    if (!attr_done) {
        FS_CUDA(cudaFuncSetAttribute(k_conv<OUT_RELU>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CV_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_conv<OUT_Z>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CV_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_conv<OUT_BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CV_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_conv_tc<IN_R, OUT_RELU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)TC_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_conv_tc<IN_ACT, OUT_RELU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)TC_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_conv_tc<IN_ACT, OUT_Z>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)TC_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_wgrad<16, 16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)WG_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_wgrad<16, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)WG_SMEM));
        FS_CUDA(cudaFuncSetAttribute(k_wgrad<2, 16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)WG_SMEM));
        attr_done = true;
    }
    return FS_OK;
}

void net_free(fs_ctx *c)
{
    NetState *n = net(c);
    if (!n) return;
    void *ptrs[] = {n->master, n->grad, n->m, n->v, n->w1f, n->w5f, n->wf, n->wt, n->act, n->gact,
                    n->y, n->gy, n->smax, n->wf1, n->wf5, n->tdist, n->tlist, n->tlist_tc};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    delete n;
    c->net = nullptr;
}

int net_load(fs_ctx *c, const float *params, int count, bool host)
{
    if (count != NPARAM) return set_error(FS_EINVAL, "the network has %d parameters, got %d", NPARAM, count);
    int rc = net_alloc(c, false);
    if (rc) return rc;
    NetState *n = net(c);
    FS_CUDA(cudaMemcpyAsync(n->master, params, NPARAM * 4, host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice,
                            c->stream));
    k_net_refresh<<<(NPARAM + 255) / 256, 256, 0, c->stream>>>(n->master, n->w1f, n->w5f, n->wf, n->wt, n->wf1,
                                                                n->wf5);
    FS_CUDA(cudaGetLastError());
    FS_CUDA(cudaStreamSynchronize(c->stream));
    n->loaded = 1;
    return FS_OK;
}

int net_read(fs_ctx *c, float *params_host)
{
    NetState *n = net(c);
    if (!n || !n->loaded) return set_error(FS_ESTATE, "no network loaded");
    FS_CUDA(cudaMemcpyAsync(params_host, n->master, NPARAM * 4, cudaMemcpyDeviceToHost, c->stream));
    FS_CUDA(cudaStreamSynchronize(c->stream));
    return FS_OK;
}

// The conv tiles sorted by their distance to the liquid, for the current mask.
static int net_tile_list(fs_ctx *c)
{
    NetState *n = net(c);
    if (n->tlist_epoch == c->mask_epoch) return FS_OK;
    const Layout &L = c->L;
    const int nt = plane_tiles(L);
    k_conv_tile_dist<<<nt, 256, 0, c->stream>>>(c->cflag, L, n->tdist);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    std::vector<uint8_t> d((size_t)nt);
    FS_CUDA(cudaMemcpyAsync(d.data(), n->tdist, (size_t)nt, cudaMemcpyDeviceToHost, c->stream));
    FS_CUDA(cudaStreamSynchronize(c->stream));
    // a 32 x 8 x 4 tile is as near as the nearest of its four planes' tiles
    const int ntx = (L.nx + NT_X - 1) / NT_X, nty = (L.ny + NT_Y - 1) / NT_Y, nxy = ntx * nty, n4 = conv_tiles(L);
    std::vector<uint8_t> d4((size_t)n4, 5);
    for (int t = 0; t < nt; t++) {
        uint8_t &m = d4[(size_t)(t / nxy / CV_Z * nxy + t % nxy)];
        m = std::min(m, d[(size_t)t]);
    }
    std::vector<int> list;
    list.reserve((size_t)n4);
    for (int dd = 0; dd <= 5; dd++) {
        for (int t = 0; t < n4; t++)
            if (d4[(size_t)t] == dd) list.push_back(t);
        n->tcount[dd] = (int)list.size();
    }
    FS_CUDA(cudaMemcpy(n->tlist, list.data(), list.size() * sizeof(int), cudaMemcpyHostToDevice));
    // the tensor-core layer's tiles (TC_M x TC_NY of one plane, inside one row of
    // conv tiles since NT_Y is a multiple of TC_NY): the distance of the nearest
    // conv tile they overlap
    const int ntxc = (L.nx + TC_M - 1) / TC_M, ntyc = (L.ny + TC_NY - 1) / TC_NY, ntc = conv_tiles_tc(L);
    std::vector<uint8_t> dc((size_t)ntc, 5);
    for (int t = 0; t < ntc; t++) {
        const int i0 = (t % ntxc) * TC_M, j0 = ((t / ntxc) % ntyc) * TC_NY, k = t / (ntxc * ntyc);
        const int ty = j0 / NT_Y;
        uint8_t m = 5;
        for (int tx = i0 / NT_X; tx <= std::min(ntx - 1, (i0 + TC_M - 1) / NT_X); tx++)
            m = std::min(m, d[(size_t)((k * nty + ty) * ntx + tx)]);
        dc[(size_t)t] = m;
    }
    std::vector<int> lc;
    lc.reserve((size_t)ntc);
    for (int dd = 0; dd <= 5; dd++) {
        for (int t = 0; t < ntc; t++)
            if (dc[(size_t)t] == dd) lc.push_back(t);
        n->tcount_tc[dd] = (int)lc.size();
    }
    FS_CUDA(cudaMemcpy(n->tlist_tc, lc.data(), lc.size() * sizeof(int), cudaMemcpyHostToDevice));
    n->tlist_epoch = c->mask_epoch;
    return FS_OK;
}

// Persistent grids: one block of k_conv per SM (its two tiles fill the shared memory).
static int conv_launch(fs_ctx *c, int out, const ConvArgs &a, int tiles)
{
    CUtensorMap map;
    if (int rc = encode_cells16(&map, a.in, c->L, CV_P, TYH, CV_Z + 2)) return rc;
    const int g = std::max(1, std::min(tiles, c->num_sms));
    if (out == OUT_RELU)
        launch_dep(k_conv<OUT_RELU>, g, 256, CV_SMEM, c->stream, map, a, c->err_word);
    else if (out == OUT_Z)
        launch_dep(k_conv<OUT_Z>, g, 256, CV_SMEM, c->stream, map, a, c->err_word);
    else
        launch_dep(k_conv<OUT_BWD>, g, 256, CV_SMEM, c->stream, map, a, c->err_word);
    c->n_launches += 1;
    return FS_OK;
}

// The tensor-core layer: two blocks per SM (two input tiles and the weights each).
static void conv_launch_tc(fs_ctx *c, int in, int out, const ConvArgs &a, int tiles)
{
    const int g = std::max(1, std::min(tiles, c->num_sms * 2));
    if (in == IN_R)
        k_conv_tc<IN_R, OUT_RELU><<<g, TC_THREADS, TC_SMEM, c->stream>>>(a, c->err_word);
    else if (out == OUT_RELU)
        k_conv_tc<IN_ACT, OUT_RELU><<<g, TC_THREADS, TC_SMEM, c->stream>>>(a, c->err_word);
    else
        k_conv_tc<IN_ACT, OUT_Z><<<g, TC_THREADS, TC_SMEM, c->stream>>>(a, c->err_word);
    c->n_launches += 1;
}

// z = s Net(r / s) on liquid cells (cell space; z is zero elsewhere before). Training (`keep`)
// runs every layer on every tile and keeps the layer inputs in act[0..4] and the
// output in y; inference runs layer l on the tiles within 5 - l cells of the
// liquid, with activations ping-ponging in act[0..1].
static int net_forward(fs_ctx *c, const float *r, float *z, float *y, bool keep, const int *done = nullptr)
{
    NetState *n = net(c);
    const Layout &L = c->L;
    const size_t nC = (size_t)L.nC;
    int rc;
    if (!keep && (rc = net_tile_list(c))) return rc;
    FS_CUDA(cudaMemsetAsync(n->smax, 0, sizeof(unsigned), c->stream));
    const int *ql = nullptr;
    int nq = 0;
    if ((rc = cell_quads(c, &ql, &nq))) return rc;
    k_absmax<<<grid_blocks(c, nq, 256), 256, 0, c->stream>>>(ql, nq, r, n->smax, done);
    c->n_launches += 1;
    __nv_bfloat16 *A[6];
    for (int l = 0; l < 6; l++) A[l] = n->act + (keep ? (size_t)l : (size_t)(l & 1)) * nC * 16;
    const int all = conv_tiles(L);
    const bool tc = !keep && n->kernel == 1;  // inference on the tcgen05 layer
    auto tiles_for = [&](int layer) {         // layer 1 .. 5
        return keep ? all : (tc ? n->tcount_tc[5 - layer] : n->tcount[5 - layer]);
    };
    auto launch = [&](int in, int out, const ConvArgs &ca) -> int {
        if (tc) {
            conv_launch_tc(c, in, out, ca, ca.ntiles);
        } else if (in == IN_R) {
            launch_dep(k_conv1, std::max(1, std::min(ca.ntiles, c->num_sms * 2)), 256, 0, c->stream, ca);
            c->n_launches += 1;
        } else {
            return conv_launch(c, out, ca, ca.ntiles);
        }
        return FS_OK;
    };
    ConvArgs a{};
    a.cf = c->cflag;
    a.smax = n->smax;
    a.done = done;
    a.tiles = keep ? nullptr : (tc ? n->tlist_tc : n->tlist);
    a.L = L;
    // layer 1: inference builds its input from r; training stores it, x -> A[0], a1 -> A[1]
    a.wts = n->wf1;
    a.bias = n->master + OB1;
    a.out = keep ? A[1] : A[0];
    a.ntiles = tiles_for(1);
    if (keep) {
        k_net_x<<<grid_blocks(c, L.S, 256), 256, 0, c->stream>>>(r, c->cflag, n->smax, L, A[0]);
        c->n_launches += 1;
        a.in = A[0];
        if ((rc = launch(IN_ACT, OUT_RELU, a))) return rc;
    } else {
        a.r = r;
        if ((rc = launch(IN_R, OUT_RELU, a))) return rc;
        a.r = nullptr;
    }
    __nv_bfloat16 *cur = a.out;
    const int bias_off[3] = {OB2, OB3, OB4};
    for (int l = 0; l < 3; l++) {
        __nv_bfloat16 *nxt = keep ? A[2 + l] : (cur == A[0] ? A[1] : A[0]);
        a.in = cur;
        a.wts = n->wf + (size_t)l * NWM;
        a.bias = n->master + bias_off[l];
        a.out = nxt;
        a.ntiles = tiles_for(2 + l);
        if ((rc = launch(IN_ACT, OUT_RELU, a))) return rc;
        cur = nxt;
    }
    a.in = cur;
    a.wts = n->wf5;
    a.bias = n->master + OB5;
    a.out = nullptr;
    a.y = y;
    a.z = z;
    a.ntiles = tiles_for(5);
    if ((rc = launch(IN_ACT, OUT_Z, a))) return rc;
    FS_CUDA(cudaGetLastError());
    return FS_OK;
}

// The flops of one inference for the current mask: layer l must be computed on the cells
// within 5 - l of the liquid, 2 x 27 x (channels in) x (channels out) each. What a tile
// holds beside them, and the channels a kernel pads to, do not count.
static int net_flops(fs_ctx *c)
{
    NetState *n = net(c);
    if (n->flops_epoch == c->mask_epoch) return FS_OK;
    const Layout &L = c->L;
    unsigned long long *dev = reinterpret_cast<unsigned long long *>(c->partials), cells[5];
    FS_CUDA(cudaMemsetAsync(dev, 0, sizeof(cells), c->stream));
    k_net_reach<<<grid_blocks(c, (long long)L.nx * L.ny * L.nz, 256), 256, 0, c->stream>>>(c->cflag, L, dev);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    FS_CUDA(cudaMemcpyAsync(cells, dev, sizeof(cells), cudaMemcpyDeviceToHost, c->stream));
    FS_CUDA(cudaStreamSynchronize(c->stream));
    const double ch[5] = {2.0 * 16, 16.0 * 16, 16.0 * 16, 16.0 * 16, 16.0};
    n->flops = 0.0;
    for (int l = 1; l <= 5; l++) n->flops += 2.0 * 27 * ch[l - 1] * (double)cells[5 - l];
    n->flops_epoch = c->mask_epoch;
    return FS_OK;
}

int net_apply(fs_ctx *c, const float *r, float *z, const int *done)
{
    NetState *n = net(c);
    if (!n || !n->loaded) return set_error(FS_ESTATE, "the learned preconditioner has no network loaded");
    if (c->prof_on)
        if (int rc = net_flops(c)) return rc;
    cudaEvent_t e0 = prof_mark(c);
    int rc = net_forward(c, r, z, nullptr, false, done);
    prof_add(c, K_NET_APPLY, e0, prof_mark(c), n->flops);  // flops, not bytes: a tensor-core entry
    return rc;
}

int net_kernel(fs_ctx *c, int which)
{
    int rc = net_alloc(c, false);
    if (rc) return rc;
    net(c)->kernel = which;
    return FS_OK;
}

// Forward + backward for one (b, q) pair (public-layout cell arrays); adds the
// gradient to the accumulator and the loss to *loss.
int net_grad(fs_ctx *c, const float *b, const float *q, double *loss)
{
    int rc = net_alloc(c, true);
    if (rc) return rc;
    NetState *n = net(c);
    if (!n->loaded) return set_error(FS_ESTATE, "load initial network parameters first");
    const Layout &L = c->L;
    const size_t nC = (size_t)L.nC;
    const int ncell = L.nx * L.ny * L.nz;
    const int gb = std::max(1, std::min((ncell + 255) / 256, c->num_sms * 8));
    FS_CUDA(cudaMemsetAsync(c->err_word, 0, sizeof(unsigned), c->stream));
    // b, q into cell space (zero off liquid): pb <- b, px <- q
    if ((rc = cell_in(c, b, c->pb)) || (rc = cell_in(c, q, c->px))) return rc;
    if ((rc = net_forward(c, c->pb, nullptr, n->y, true))) return rc;
    __nv_bfloat16 *A[5];
    for (int l = 0; l < 5; l++) A[l] = n->act + (size_t)l * nC * 16;
    SolveScal *s = c->scal + 3;
    const int bsn = grid_blocks(c, L.nC, 256);
    if (c->prm.precond == FS_PRECOND_LEARNED_MG) {
        // the network followed by the V-cycle; scratch (no solve runs meanwhile):
        // pxh = ym, pr = b/s - A ym, pz = M pr, pp0 = w, pp1 = q/s, pq = A w, pbr = M A w
        k_net_mask_y<<<bsn, 256, 0, c->stream>>>(n->y, c->cflag, c->pxh, L.nC);
        k_netmg_res<<<bsn, 256, 0, c->stream>>>(c->pb, c->pxh, c->cflag, n->smax, L, c->pr);
        c->n_launches += 2;
        if ((rc = mg_apply(c, c->pr, c->pz, nullptr))) return rc;
        k_netmg_err<<<bsn, 256, 0, c->stream>>>(c->px, c->pxh, c->pz, c->cflag, n->smax, c->pp[0], c->pp[1], L.nC);
        k_net_energy<<<bsn, 256, 0, c->stream>>>(c->pp[0], c->pp[1], c->pq, c->cflag, L, s, c->partials);
        c->n_launches += 2;
        if ((rc = mg_apply(c, c->pq, c->pbr, nullptr))) return rc;
        k_netmg_gy<<<bsn, 256, 0, c->stream>>>(c->pq, c->pbr, c->cflag, s, L, n->gy);
        c->n_launches += 1;
    } else {
        // energy-norm loss; scratch: pr = e, pz = q/s, pq = A e (no solve runs meanwhile)
        k_net_err<<<bsn, 256, 0, c->stream>>>(n->y, c->px, c->cflag, n->smax, c->pr, c->pz, L.nC);
        k_net_energy<<<bsn, 256, 0, c->stream>>>(c->pr, c->pz, c->pq, c->cflag, L, s, c->partials);
        k_net_gy<<<bsn, 256, 0, c->stream>>>(c->pq, c->cflag, s, n->gy, L.nC);
        c->n_launches += 3;
    }
    // layer 5
    const int wg = std::max(1, std::min(((L.nx + NT_X - 1) / NT_X) * ((L.ny + NT_Y - 1) / NT_Y) * L.nz, c->num_sms));
    k_wgrad<16, 1, true><<<wg, WG_TH, WG_SMEM, c->stream>>>(n->gy, A[4], n->grad + OW5, n->grad + OB5, L);
    __nv_bfloat16 *G[2] = {n->gact, n->gact + nC * 16};
    k_bwd_last<<<gb, 256, 0, c->stream>>>(n->gy, n->w5f, A[4], G[0], L);
    // layers 4, 3, 2: weight gradient, then the gradient of the layer input
    const int woff[3] = {OW2, OW3, OW4}, boff[3] = {OB2, OB3, OB4};
    int gi = 0;
    for (int l = 2; l >= 0; l--) {
        // G[gi] = dL/d(output of layer l+2) (post-ReLU mask applied); input = A[l+1]
        k_wgrad<16, 16, false><<<wg, WG_TH, WG_SMEM, c->stream>>>(G[gi], A[l + 1], n->grad + woff[l], n->grad + boff[l], L);
        ConvArgs bw{};
        bw.in = G[gi];
        bw.wts = n->wt + (size_t)l * NWM;
        bw.aref = A[l + 1];
        bw.out = G[gi ^ 1];
        bw.L = L;
        if ((rc = conv_launch(c, OUT_BWD, bw, conv_tiles(L)))) return rc;
        gi ^= 1;
    }
    // layer 1: gradient w.r.t. W1 from the stored input x (2 channels used)
    k_wgrad<2, 16, false><<<wg, WG_TH, WG_SMEM, c->stream>>>(G[gi], A[0], n->grad + OW1, n->grad + OB1, L);
    c->n_launches += 2 + 6 + 1;
    FS_CUDA(cudaGetLastError());
    SolveScal h;
    unsigned herr = 0;
    if ((rc = read_scal(c, 3, &h, &herr))) return rc;
    if (herr & ERR_NET) return set_error(FS_ETIMEOUT, "network: a bounded wait ran out");
    if (loss) *loss += h.aux[1] > 0.0 ? h.aux[0] / h.aux[1] : 0.0;
    return FS_OK;
}

int net_adam(fs_ctx *c, double lr, double beta1, double beta2, double eps, int step, double gscale, int fix_offsets)
{
    NetState *n = net(c);
    if (!n || !n->loaded || !n->gact) return set_error(FS_ESTATE, "no gradients accumulated");
    if (step < 1) return set_error(FS_EINVAL, "step must be >= 1");
    const float c1 = (float)(1.0 - std::pow(beta1, step)), c2 = (float)(1.0 - std::pow(beta2, step));
    k_adam<<<(NPARAM + 255) / 256, 256, 0, c->stream>>>(n->master, n->grad, n->m, n->v, NPARAM, (float)lr,
                                                        (float)beta1, (float)beta2, (float)eps, c1, c2,
                                                        (float)gscale, fix_offsets);
    k_net_refresh<<<(NPARAM + 255) / 256, 256, 0, c->stream>>>(n->master, n->w1f, n->w5f, n->wf, n->wt, n->wf1,
                                                                n->wf5);
    c->n_launches += 2;
    FS_CUDA(cudaGetLastError());
    FS_CUDA(cudaStreamSynchronize(c->stream));
    return FS_OK;
}

int net_grad_read(fs_ctx *c, float *grad_host)
{
    NetState *n = net(c);
    if (!n || !n->gact) return set_error(FS_ESTATE, "no gradients accumulated");
    FS_CUDA(cudaMemcpyAsync(grad_host, n->grad, NPARAM * 4, cudaMemcpyDeviceToHost, c->stream));
    FS_CUDA(cudaStreamSynchronize(c->stream));
    return FS_OK;
}

int net_grad_clear(fs_ctx *c)
{
    NetState *n = net(c);
    if (!n) return FS_OK;
    k_fill_zero<<<(NPARAM + 255) / 256, 256, 0, c->stream>>>(n->grad, NPARAM);
    c->n_launches += 1;
    FS_CUDA(cudaGetLastError());
    return FS_OK;
}

int net_param_count() { return NPARAM; }

bool net_loaded(const fs_ctx *c) { return c->net && static_cast<const NetState *>(c->net)->loaded; }

}  // namespace fs
