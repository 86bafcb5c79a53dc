// fs_percnn.cu -- recurrent convolutional pressure solver (arXiv 2503.00868,
// Sec. 3.4.1: the PeRCNN layer that replaces the implicit pressure solve during
// the optimisation, with a fitted convolution kernel and ~100 recurrent
// sub-steps per simulation step).
//
// Reading: the physics operator is the scheme's own 7-point L_p with the
// cell-type boundary conditions (air p = 0, solid walls zero flux), the fitted
// part a 3x3x3 kernel W on the residual, and the recurrent layer emulates an
// implicit solver's iteration:
//   p_0 = 0,  r_k = m (b - L_p p_k),  p_{k+1} = p_k + m (W * r_k),  k < K,
// m the liquid mask, * the 27-tap correlation (taps [dz][dy][dx]). Fixed points
// solve L_p p = b. The kernel is stored point-symmetric (W[t] = W[26 - t]), which
// makes the map b -> p_K symmetric and the projection built on it self-adjoint,
// so the step's adjoint applies the same projection to the cotangent.
// Per sub-step: one residual pass and one 27-point correlation pass over the list of
// quads that hold liquid. At 128^3 (a blob, 40 %) the dense passes, with 27 scalar
// loads per cell, took 5.6 and 21 us, these 3.6 and 6.2; both stay in L2. The launches'
// gaps (2 x 2.4 us) went with dependent launches: 12 us per sub-step for the two.
//
// Training (fs_percnn_grad): the energy-norm loss of Sec. 3.4.1's fit,
//   e = p_K - q, loss = e^T L_p e / q^T L_p q,
// and dloss/dW by the backward recurrence over the stored residuals:
//   g_K = 2 L_p e / q^T L_p q;  for k = K-1 .. 0:
//   dW[t] += sum_i g_{k+1,i} r_k(i + t);  g_k = g_{k+1} - L_p (m W^T * g_{k+1}).
#include <cmath>
#include <new>

#include "fs_internal.cuh"

namespace fs {

struct PercnnW {
    float w[27];
};

struct PercnnState {
    PercnnW w;
    int K = 0;
    int loaded = 0;
    float *rstack = nullptr;  // K residuals (training)
    int rstack_k = 0;
    long long epoch = -1;  // mask the stack and t1 are zero off the liquid of
    float *gk = nullptr, *t1 = nullptr;  // cell space
    double *dw = nullptr;     // device [27]
};

namespace {

constexpr int TH = 256;

__device__ __forceinline__ int tap_offset(const Layout &L, int t)
{
    return (t / 9 - 1) * L.PL + ((t / 3) % 3 - 1) * L.P + (t % 3 - 1);
}

// The passes of a sub-step walk the list of quads that hold a liquid cell, four
// cells per thread; r, p and every other vector are zero off the liquid and are
// neither read nor written on the other quads.

// r = m (b - L_p p)
__global__ void __launch_bounds__(TH) k_pc_res(const int *__restrict__ ql, int nq, const float *__restrict__ b,
                                               const float *__restrict__ p, float *__restrict__ r,
                                               const uint8_t *__restrict__ cf, int P, int PL)
{
    dep_wait();
    dep_go();
    FS_FOR_LIST(ql, nq)
    {
        const int t = 4 * q;
        const uchar4 f = __ldg(reinterpret_cast<const uchar4 *>(cf + t));
        auto p4 = [&](int u) { return ldd4(p + u); };
        const float4 c = p4(t), dn = p4(t - P), up = p4(t + P), bk = p4(t - PL), fw = p4(t + PL);
        const float4 bv = ldd4(b + t);
        const float lf = ldd1(p + t - 1), rt = ldd1(p + t + 4);
        auto one = [&](uint8_t fe, float ce, float nb, float be) {
            return (fe & CF_LIQ) ? be - ((float)(fe & CF_D) * ce - nb) : 0.f;
        };
        float4 v;
        v.x = one(f.x, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x), bv.x);
        v.y = one(f.y, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y), bv.y);
        v.z = one(f.z, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z), bv.z);
        v.w = one(f.w, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w), bv.w);
        *reinterpret_cast<float4 *>(r + t) = v;
    }
}

// out = m (W * x) (+ base when base != null): 27-tap correlation on liquid cells. A
// row of three taps is formed from one float4 and its two neighbours. One guard plane
// stands before the cells, so for quads in the first two rows of the first plane some of
// these taps lie before the vector: off the grid, they count zero without a load.
__global__ void __launch_bounds__(TH) k_pc_conv(const int *__restrict__ ql, int nq, const float *__restrict__ x,
                                                const float *base, float *out, const uint8_t *__restrict__ cf, int P,
                                                int PL, const __grid_constant__ PercnnW W)
{
    dep_wait();
    dep_go();
    FS_FOR_LIST(ql, nq)
    {
        const int t = 4 * q;
        const uchar4 f = __ldg(reinterpret_cast<const uchar4 *>(cf + t));
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int row = 0; row < 9; row++) {
            const int u = t + (row / 3 - 1) * PL + (row % 3 - 1) * P;
            const bool in = row > 1 || u >= 0, lin = row > 1 || u > 0;
            const float4 c = in ? ldd4(x + u) : make_float4(0.f, 0.f, 0.f, 0.f);
            const float lf = lin ? ldd1(x + u - 1) : 0.f, rt = in ? ldd1(x + u + 4) : 0.f;
            const float w0 = W.w[3 * row], w1 = W.w[3 * row + 1], w2 = W.w[3 * row + 2];
            v.x += w0 * lf; v.y += w0 * c.x; v.z += w0 * c.y; v.w += w0 * c.z;
            v.x += w1 * c.x; v.y += w1 * c.y; v.z += w1 * c.z; v.w += w1 * c.w;
            v.x += w2 * c.y; v.y += w2 * c.z; v.z += w2 * c.w; v.w += w2 * rt;
        }
        float4 o = base ? ldd4(base + t) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (f.x & CF_LIQ) o.x += v.x;
        if (f.y & CF_LIQ) o.y += v.y;
        if (f.z & CF_LIQ) o.z += v.z;
        if (f.w & CF_LIQ) o.w += v.w;
        *reinterpret_cast<float4 *>(out + t) = o;
    }
}

// g = m (g - L_p s)
__global__ void __launch_bounds__(TH) k_pc_lapsub(float *g, const float *__restrict__ s,
                                                  const uint8_t *__restrict__ cf, int n, int P, int PL)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const uint8_t f = cf[t];
        if (f & CF_LIQ) {
            const float nb = (s[t - 1] + s[t + 1]) + (s[t - P] + s[t + P]) + (s[t - PL] + s[t + PL]);
            g[t] -= (float)(f & CF_D) * s[t] - nb;
        } else {
            g[t] = 0.f;
        }
    }
}

// dw[q] += sum over liquid cells of g_i r(i + o_q); a tap before the vector (k_pc_conv)
// is off the grid and adds nothing
__global__ void __launch_bounds__(TH) k_pc_wgrad(const float *__restrict__ g, const float *__restrict__ r,
                                                 const uint8_t *__restrict__ cf, Layout L, double *dw)
{
    __shared__ double sh[TH / 32][27];
    int off[27];
#pragma unroll
    for (int q = 0; q < 27; q++) off[q] = tap_offset(L, q);
    double acc[27];
#pragma unroll
    for (int q = 0; q < 27; q++) acc[q] = 0.0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < L.nC; t += gridDim.x * blockDim.x) {
        if (!(cf[t] & CF_LIQ)) continue;
        const float gv = g[t];
        if (gv == 0.f) continue;
#pragma unroll
        for (int q = 0; q < 27; q++)
            if (q > 3 || t + off[q] >= 0) acc[q] += (double)(gv * r[t + off[q]]);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 27; q++) {
        const double v = warp_sum(acc[q]);
        if (lane == 0) sh[wid][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < 27) {
        double s = 0.0;
        for (int w = 0; w < TH / 32; w++) s += sh[w][threadIdx.x];
        atomicAdd(dw + threadIdx.x, s);
    }
}

// e = m (p - q)
__global__ void __launch_bounds__(TH) k_pc_energy(const float *__restrict__ p, const float *__restrict__ q,
                                                  float *e, const uint8_t *__restrict__ cf, int n)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
        e[t] = (cf[t] & CF_LIQ) ? p[t] - q[t] : 0.f;
}

// e.Ae and q.Aq over the liquid -> aux[0], aux[1]; Ae kept in ae
__global__ void __launch_bounds__(TH) k_pc_quad(const float *__restrict__ e, const float *__restrict__ q,
                                                float *ae, const uint8_t *__restrict__ cf, int n, int P, int PL,
                                                SolveScal *s, double *partials)
{
    KSum ee, qq;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const uint8_t f = cf[t];
        float a = 0.f;
        if (f & CF_LIQ) {
            const float d = (float)(f & CF_D);
            a = d * e[t] - ((e[t - 1] + e[t + 1]) + (e[t - P] + e[t + P]) + (e[t - PL] + e[t + PL]));
            const float aq = d * q[t] - ((q[t - 1] + q[t + 1]) + (q[t - P] + q[t + P]) + (q[t - PL] + q[t + PL]));
            ee.add(e[t] * a);
            qq.add(q[t] * aq);
        }
        ae[t] = a;
    }
    double v[2] = {ee.value(), qq.value()}, tot[2];
    if (grid_reduce<2>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        s->aux[0] = tot[0];
        s->aux[1] = tot[1];
    }
}

__global__ void k_pc_scale(float *g, const SolveScal *s, int n)
{
    const double den = s->aux[1];
    const float sc = den > 0.0 ? (float)(2.0 / den) : 0.f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) g[t] *= sc;
}

// |r|^2 and |b|^2 over the liquid into the scalars of a finished solve of K sub-steps
__global__ void __launch_bounds__(TH) k_pc_finish(const float *__restrict__ b, const float *__restrict__ r,
                                                  const uint8_t *__restrict__ cf, int n, int K, SolveScal *s,
                                                  double *partials)
{
    KSum rr, bb;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
        if (cf[t] & CF_LIQ) {
            rr.add(r[t] * r[t]);
            bb.add(b[t] * b[t]);
        }
    double v[2] = {rr.value(), bb.value()}, tot[2];
    if (grid_reduce<2>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        s->rr = tot[0];
        s->bb = tot[1];
        s->iter = K;
        s->done = 1;
        s->status = (isfinite(tot[0]) && isfinite(tot[1])) ? FS_OK : FS_ENONFINITE;
    }
}

PercnnState *pcs(fs_ctx *c) { return static_cast<PercnnState *>(c->percnn); }

int res_resident()
{
    static const int r = resident_blocks((const void *)k_pc_res, 0);
    return r;
}
int conv_resident()
{
    static const int r = resident_blocks((const void *)k_pc_conv, 0);
    return r;
}

}  // namespace

void percnn_free(fs_ctx *c)
{
    PercnnState *s = pcs(c);
    if (!s) return;
    cudaFree(s->rstack);
    cudaFree(s->gk);
    cudaFree(s->t1);
    cudaFree(s->dw);
    delete s;
    c->percnn = nullptr;
}

bool percnn_loaded(const fs_ctx *c) { return c->percnn && static_cast<const PercnnState *>(c->percnn)->loaded; }

int percnn_load(fs_ctx *c, const float *w27, int K)
{
    if (!w27) return set_error(FS_EINVAL, "the kernel is NULL");
    if (K < 1 || K > 100000) return set_error(FS_EINVAL, "substeps must be in [1, 100000]");
    for (int t = 0; t < 27; t++)
        if (!std::isfinite(w27[t])) return set_error(FS_EINVAL, "kernel tap %d is not finite", t);
    PercnnState *s = pcs(c);
    if (!s) {
        s = new (std::nothrow) PercnnState();
        if (!s) return set_error(FS_ENOMEM, "host allocation failed");
        c->percnn = s;
    }
    for (int t = 0; t < 27; t++) s->w.w[t] = 0.5f * (w27[t] + w27[26 - t]);  // point-symmetric
    s->K = K;
    s->loaded = 1;
    return FS_OK;
}

int percnn_read(fs_ctx *c, float *w27, int *K)
{
    PercnnState *s = pcs(c);
    if (!s || !s->loaded) return set_error(FS_ESTATE, "no recurrent-solver kernel loaded");
    for (int t = 0; t < 27; t++) w27[t] = s->w.w[t];
    if (K) *K = s->K;
    return FS_OK;
}

// pb -> px by K sub-steps (pr scratch); h gets K and the scalars of the true residual
int solve_pressure_percnn(fs_ctx *c, SolveScal *h)
{
    PercnnState *s = pcs(c);
    if (!s || !s->loaded) return set_error(FS_ESTATE, "the recurrent pressure solver has no kernel loaded");
    const Layout &L = c->L;
    const int bs = grid_blocks(c, L.nC, TH);
    const int *ql = nullptr;
    int nq = 0;
    if (int rc = cell_quads(c, &ql, &nq)) return rc;
    const int br = wave_blocks(c, nq, res_resident()), bv = wave_blocks(c, nq, conv_resident());
    FS_CUDA(cudaMemsetAsync(c->px, 0, (size_t)L.nC * sizeof(float), c->stream));
    FS_CUDA(cudaMemsetAsync(c->pr, 0, (size_t)L.nC * sizeof(float), c->stream));
    for (int k = 0; k < s->K; k++) {
        launch_dep(k_pc_res, br, TH, 0, c->stream, ql, nq, c->pb, c->px, c->pr, c->cflag, L.P, L.PL);
        launch_dep(k_pc_conv, bv, TH, 0, c->stream, ql, nq, c->pr, c->px, c->px, c->cflag, L.P, L.PL, s->w);
        c->n_launches += 2;
    }
    FS_CUDA(cudaGetLastError());
    if (c->singular) {
        int rc = remove_null_mode(c, c->px);
        if (rc) return rc;
    }
    k_pc_res<<<br, TH, 0, c->stream>>>(ql, nq, c->pb, c->px, c->pr, c->cflag, L.P, L.PL);
    k_pc_finish<<<bs, TH, 0, c->stream>>>(c->pb, c->pr, c->cflag, L.nC, s->K, c->scal + 0, c->partials);
    c->n_launches += 2;
    FS_CUDA(cudaGetLastError());
    return read_scal(c, 0, h);
}

int percnn_grad(fs_ctx *c, const float *b, const float *q, double *loss, float *dw_host)
{
    PercnnState *s = pcs(c);
    if (!s || !s->loaded) return set_error(FS_ESTATE, "no recurrent-solver kernel loaded");
    const Layout &L = c->L;
    const size_t nC = (size_t)L.nC;
    const int K = s->K;
    if ((double)K * nC * 4.0 > 8e9) return set_error(FS_EINVAL, "K x grid too large for the residual stack");
    if (s->rstack_k < K) {
        cudaFree(s->rstack);
        s->rstack = nullptr;
        s->rstack_k = 0;
        if (cudaMalloc(&s->rstack, (size_t)K * nC * sizeof(float)) != cudaSuccess) {
            cudaGetLastError();
            return set_error(FS_ENOMEM, "residual stack of %d x %zu floats", K, nC);
        }
        s->rstack_k = K;
        s->epoch = -1;
    }
    if (!s->gk) {
        if (cudaMalloc(&s->gk, nC * 4) != cudaSuccess || cudaMalloc(&s->t1, nC * 4) != cudaSuccess ||
            cudaMalloc(&s->dw, 27 * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            return set_error(FS_ENOMEM, "recurrent-solver training buffers");
        }
        FS_CUDA(cudaMemset(s->gk, 0, nC * 4));
        FS_CUDA(cudaMemset(s->t1, 0, nC * 4));
    }
    int rc;
    if ((rc = cell_in(c, b, c->pb)) || (rc = cell_in(c, q, c->pz))) return rc;
    const int bs = grid_blocks(c, L.nC, TH);
    const int *ql = nullptr;
    int nq = 0;
    if ((rc = cell_quads(c, &ql, &nq))) return rc;
    const int br = wave_blocks(c, nq, res_resident()), bv = wave_blocks(c, nq, conv_resident());
    if (s->epoch != c->mask_epoch) {  // a new mask: its passes write the stack and t1 on its active quads only
        FS_CUDA(cudaMemsetAsync(s->rstack, 0, (size_t)s->rstack_k * nC * 4, c->stream));
        FS_CUDA(cudaMemsetAsync(s->t1, 0, nC * 4, c->stream));
        s->epoch = c->mask_epoch;
    }
    FS_CUDA(cudaMemsetAsync(c->px, 0, nC * 4, c->stream));
    for (int k = 0; k < K; k++) {
        float *r = s->rstack + (size_t)k * nC;
        k_pc_res<<<br, TH, 0, c->stream>>>(ql, nq, c->pb, c->px, r, c->cflag, L.P, L.PL);
        k_pc_conv<<<bv, TH, 0, c->stream>>>(ql, nq, r, c->px, c->px, c->cflag, L.P, L.PL, s->w);
    }
    // loss and g_K = 2 L e / q.Lq
    SolveScal *sc = c->scal + 3;
    k_pc_energy<<<bs, TH, 0, c->stream>>>(c->px, c->pz, c->pr, c->cflag, L.nC);
    k_pc_quad<<<bs, TH, 0, c->stream>>>(c->pr, c->pz, s->gk, c->cflag, L.nC, L.P, L.PL, sc, c->partials);
    k_pc_scale<<<bs, TH, 0, c->stream>>>(s->gk, sc, L.nC);
    FS_CUDA(cudaMemsetAsync(s->dw, 0, 27 * sizeof(double), c->stream));
    for (int k = K - 1; k >= 0; k--) {
        const float *r = s->rstack + (size_t)k * nC;
        k_pc_wgrad<<<bs, TH, 0, c->stream>>>(s->gk, r, c->cflag, L, s->dw);
        k_pc_conv<<<bv, TH, 0, c->stream>>>(ql, nq, s->gk, nullptr, s->t1, c->cflag, L.P, L.PL, s->w);  // W^T = W
        k_pc_lapsub<<<bs, TH, 0, c->stream>>>(s->gk, s->t1, c->cflag, L.nC, L.P, L.PL);
    }
    c->n_launches += 2 * K + 3 + 3 * K;
    FS_CUDA(cudaGetLastError());
    double dw[27];
    FS_CUDA(cudaMemcpyAsync(dw, s->dw, sizeof(dw), cudaMemcpyDeviceToHost, c->stream));
    SolveScal h;
    if ((rc = read_scal(c, 3, &h))) return rc;
    if (loss) *loss += h.aux[1] > 0.0 ? h.aux[0] / h.aux[1] : 0.0;
    if (dw_host)
        for (int t = 0; t < 27; t++) dw_host[t] += (float)dw[t];
    return FS_OK;
}

}  // namespace fs
