// fs_fcg.cu -- truncated flexible CG for the pressure solve with the learned
// (nonlinear) preconditioner (the network that stands in for the implicit
// pressure solve, Sec. 3.4.1).
//
// With a preconditioner that changes from one application to the next, plain
// CG loses the conjugacy of its directions. Flexible CG (Notay, "Flexible
// conjugate gradients", SIAM J. Sci. Comput. 22(4), 2000) restores it by
// A-orthogonalising each new direction explicitly against the last M ones:
//   z_k = Net(r_k)
//   p_k = z_k - sum_{j=1..min(k,M)} (z_k . A p_{k-j} / p_{k-j} . A p_{k-j}) p_{k-j}
//   alpha_k = r_k . z_k / p_k . A p_k,   x += alpha_k p_k,   r -= alpha_k A p_k.
// The M most recent (p, A p, p.Ap) triples live in a ring of cell-space vectors.
// Per iteration: the network, then four HBM-bound kernels (dots, direction,
// operator + p.Ap, update); every decision is taken on the device, the host
// reads the scalars every check_every iterations. The kernels walk the list of
// quads that hold liquid (every vector is zero elsewhere): dense passes over a
// union of spheres that fills a fifth of 256^3 took up to 82, 61, 41 and 68 us,
// these 28, 15, 11 and 14.
#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "fs_internal.cuh"

namespace fs {
namespace {

constexpr int TH = 256;
constexpr int FCG_M = 4;

// The j-th most recent direction (j = 0 newest), its A p and its p.Ap.
struct Ring {
    const float *p[FCG_M];
    const float *q[FCG_M];
    const double *pq[FCG_M];
};

// beta_j = -z . A p_j / p_j . A p_j (j < nvalid) and r.z -> s->rz; with e, z += e first
__global__ void __launch_bounds__(TH) k_fcg_dots(const int *__restrict__ ql, int nq, float *z, const float *__restrict__ e,
                                                 const float *__restrict__ r, Ring ring, int nvalid, SolveScal *s,
                                                 double *beta, double *partials)
{
    dep_wait();
    dep_go();
    if (s->done) return;
    KSum acc[FCG_M + 1];
    float4 *z4 = reinterpret_cast<float4 *>(z);
    FS_FOR_LIST(ql, nq)
    {
        float4 a = ldd4(z + 4 * q);
        const float4 b = ldd4(r + 4 * q);
        if (e) {
            const float4 w = ldd4(e + 4 * q);
            a.x += w.x; a.y += w.y; a.z += w.z; a.w += w.w;
            z4[q] = a;
        }
        acc[FCG_M].add(a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w);
#pragma unroll
        for (int j = 0; j < FCG_M; j++) {
            if (j < nvalid) {
                const float4 c = ldd4(ring.q[j] + 4 * q);
                acc[j].add(a.x * c.x + a.y * c.y + a.z * c.z + a.w * c.w);
            }
        }
    }
    KSum v[FCG_M + 1];
    double tot[FCG_M + 1];
#pragma unroll
    for (int j = 0; j <= FCG_M; j++) v[j] = acc[j];
    if (grid_reduce<FCG_M + 1>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        bool ok = isfinite(tot[FCG_M]);
        for (int j = 0; j < FCG_M; j++) {
            const double pq = j < nvalid ? *ring.pq[j] : 0.0;
            beta[j] = (j < nvalid && pq > 0.0) ? -tot[j] / pq : 0.0;
            ok = ok && isfinite(beta[j]);
        }
        if (!ok) { s->done = 1; s->status = FS_ENONFINITE; return; }
        s->rz = tot[FCG_M];
    }
}

// p = z + sum_j beta_j p_j (beta_j: written by the launch before, so read as the
// vectors are, after dep_wait and not by the non-coherent path)
__global__ void __launch_bounds__(TH) k_fcg_dir(const int *__restrict__ ql, int nq, const float *__restrict__ z, Ring ring,
                                                int nvalid, float *__restrict__ p, const SolveScal *s,
                                                const double *beta)
{
    dep_wait();
    dep_go();
    if (s->done) return;
    float b[FCG_M];
#pragma unroll
    for (int j = 0; j < FCG_M; j++) b[j] = j < nvalid ? (float)*(const volatile double *)(beta + j) : 0.f;
    float4 *p4 = reinterpret_cast<float4 *>(p);
    FS_FOR_LIST(ql, nq)
    {
        float4 v = ldd4(z + 4 * q);
#pragma unroll
        for (int j = 0; j < FCG_M; j++) {
            if (j < nvalid) {
                const float4 w = ldd4(ring.p[j] + 4 * q);
                v.x += b[j] * w.x; v.y += b[j] * w.y; v.z += b[j] * w.z; v.w += b[j] * w.w;
            }
        }
        p4[q] = v;
    }
}

// q = L_p p (7-point pressure operator on liquid cells), p.q -> *pq_out,
// alpha = r.z / p.q
__global__ void __launch_bounds__(TH) k_fcg_apply(const int *__restrict__ ql, int nq, const float *__restrict__ p,
                                                  float *__restrict__ qo, const uint8_t *__restrict__ cf, int P, int PL,
                                                  SolveScal *s, double *pq_out, double *partials)
{
    dep_wait();
    dep_go();
    if (s->done) return;
    KSum acc;
    FS_FOR_LIST(ql, nq)
    {
        const int t = 4 * q;
        const uchar4 f = __ldg(reinterpret_cast<const uchar4 *>(cf + t));
        auto p4 = [&](int u) { return ldd4(p + u); };
        const float4 c = p4(t), dn = p4(t - P), up = p4(t + P), bk = p4(t - PL), fw = p4(t + PL);
        const float lf = ldd1(p + t - 1), rt = ldd1(p + t + 4);
        auto one = [&](uint8_t fe, float ce, float nb) { return (fe & CF_LIQ) ? (float)(fe & CF_D) * ce - nb : 0.f; };
        float4 v;
        v.x = one(f.x, c.x, (lf + c.y) + (dn.x + up.x) + (bk.x + fw.x));
        v.y = one(f.y, c.y, (c.x + c.z) + (dn.y + up.y) + (bk.y + fw.y));
        v.z = one(f.z, c.z, (c.y + c.w) + (dn.z + up.z) + (bk.z + fw.z));
        v.w = one(f.w, c.w, (c.z + rt) + (dn.w + up.w) + (bk.w + fw.w));
        acc.add(c.x * v.x + c.y * v.y + c.z * v.z + c.w * v.w);
        *reinterpret_cast<float4 *>(qo + t) = v;
    }
    KSum v[1] = {acc};
    double tot[1];
    if (grid_reduce<1>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        const double pq = tot[0];
        *pq_out = pq;
        s->pq = pq;
        if (!isfinite(pq)) { s->done = 1; s->status = FS_ENONFINITE; }
        else if (!(pq > 0.0)) { s->done = 1; s->status = FS_EBREAKDOWN; }
        else s->alpha = s->rz / pq;
    }
}

// x += alpha p, r -= alpha q; r.r and the convergence decision
__global__ void __launch_bounds__(TH) k_fcg_update(const int *__restrict__ ql, int nq, float *__restrict__ x,
                                                   float *__restrict__ r, const float *__restrict__ p,
                                                   const float *__restrict__ ap, SolveScal *s, double *partials)
{
    dep_wait();
    dep_go();
    if (s->done) return;
    const float alpha = (float)s->alpha;
    KSum rr;
    float4 *x4 = reinterpret_cast<float4 *>(x);
    float4 *r4 = reinterpret_cast<float4 *>(r);
    FS_FOR_LIST(ql, nq)
    {
        const float4 pv = ldd4(p + 4 * q);
        const float4 qv = ldd4(ap + 4 * q);
        float4 xv = ldd4(x + 4 * q), rv = ldd4(r + 4 * q);
        xv.x += alpha * pv.x; xv.y += alpha * pv.y; xv.z += alpha * pv.z; xv.w += alpha * pv.w;
        rv.x -= alpha * qv.x; rv.y -= alpha * qv.y; rv.z -= alpha * qv.z; rv.w -= alpha * qv.w;
        x4[q] = xv;
        r4[q] = rv;
        rr.add(rv.x * rv.x + rv.y * rv.y + rv.z * rv.z + rv.w * rv.w);
    }
    KSum v[1] = {rr};
    double tot[1];
    if (grid_reduce<1>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        s->iter += 1;
        s->rr = tot[0];
        if (!isfinite(tot[0])) { s->done = 1; s->status = FS_ENONFINITE; }
        else if (tot[0] <= s->tol2 * s->bb) { s->done = 1; s->status = FS_OK; }
        else if (s->iter >= s->maxit) { s->done = 1; s->status = FS_ENOCONV; }
    }
}

// x = 0, r = b; b.b and the scalars of a fresh solve
__global__ void __launch_bounds__(TH) k_fcg_init(const float *__restrict__ b, float *__restrict__ x,
                                                 float *__restrict__ r, int n4, double tol2, int maxit, SolveScal *s,
                                                 double *partials)
{
    KSum bb;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n4; t += gridDim.x * blockDim.x) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(b) + t);
        reinterpret_cast<float4 *>(r)[t] = v;
        reinterpret_cast<float4 *>(x)[t] = zero;
        bb.add(v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w);
    }
    KSum v[1] = {bb};
    double tot[1];
    if (grid_reduce<1>(v, partials, &s->ticket, tot) && threadIdx.x == 0) {
        s->bb = tot[0];
        s->rr = tot[0];
        s->rz = 0.0;
        s->pq = 0.0;
        s->alpha = 0.0;
        s->beta = 0.0;
        s->tol2 = tol2;
        s->iter = 0;
        s->maxit = maxit;
        s->status = FS_OK;
        s->done = 0;
        if (!isfinite(tot[0])) { s->done = 1; s->status = FS_ENONFINITE; }
        else if (tot[0] == 0.0) s->done = 1;
    }
}

struct FcgState {
    float *p[FCG_M] = {};
    float *q[FCG_M] = {};
    double *beta = nullptr;  // device [FCG_M]
    double *pq = nullptr;    // device [FCG_M], per ring slot
    long long epoch = -1;    // mask the ring vectors are zero off the liquid of
};

void fcg_free_state(FcgState *f)
{
    if (!f) return;
    for (int j = 0; j < FCG_M; j++) {
        cudaFree(f->p[j]);
        cudaFree(f->q[j]);
    }
    cudaFree(f->beta);
    cudaFree(f->pq);
    delete f;
}

int fcg_alloc(fs_ctx *c)
{
    if (c->fcg) return FS_OK;
    FcgState *f = new (std::nothrow) FcgState();
    if (!f) return set_error(FS_ENOMEM, "flexible CG: host allocation failed");
    const size_t cb = (size_t)c->L.nC * sizeof(float);
    bool ok = true;
    for (int j = 0; j < FCG_M && ok; j++)
        ok = cudaMalloc(&f->p[j], cb) == cudaSuccess && cudaMalloc(&f->q[j], cb) == cudaSuccess;
    ok = ok && cudaMalloc(&f->beta, FCG_M * sizeof(double)) == cudaSuccess &&
         cudaMalloc(&f->pq, FCG_M * sizeof(double)) == cudaSuccess &&
         cudaMemset(f->pq, 0, FCG_M * sizeof(double)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        fcg_free_state(f);
        return set_error(FS_ENOMEM, "flexible CG: device allocation of %d direction pairs failed", FCG_M);
    }
    c->fcg = f;
    return FS_OK;
}

}  // namespace

void fcg_release(fs_ctx *c)
{
    fcg_free_state(static_cast<FcgState *>(c->fcg));
    c->fcg = nullptr;
}

// Flexible CG on pb -> px with the loaded network, from x = 0 or (warm) from
// the current x with the true residual. Leaves the final scalars in *h (status
// FS_ENOCONV also when |r| stagnates: no tenfold drop over 200 iterations); the
// caller computes the true residual.
int solve_pressure_fcg(fs_ctx *c, SolveScal *h, bool warm)
{
    int rc = fcg_alloc(c);
    if (rc) return rc;
    FcgState *f = static_cast<FcgState *>(c->fcg);
    const Layout &L = c->L;
    SolveScal *s = c->scal + 0;
    const int n4 = L.nC / 4;
    const int b4 = grid_blocks(c, n4, TH);
    if (f->epoch != c->mask_epoch) {  // a new mask: its kernels write the ring on its active quads only
        for (int j = 0; j < FCG_M; j++) {
            FS_CUDA(cudaMemsetAsync(f->p[j], 0, (size_t)L.nC * sizeof(float), c->stream));
            FS_CUDA(cudaMemsetAsync(f->q[j], 0, (size_t)L.nC * sizeof(float), c->stream));
        }
        f->epoch = c->mask_epoch;
    }
    const int *ql = nullptr;
    int nq = 0;
    if ((rc = learned_begin(c)) || (rc = cell_quads(c, &ql, &nq))) return rc;
    static const int rd = resident_blocks((const void *)k_fcg_dots, 0), ri = resident_blocks((const void *)k_fcg_dir, 0);
    static const int ra = resident_blocks((const void *)k_fcg_apply, 0);
    static const int ru = resident_blocks((const void *)k_fcg_update, 0);
    const double tol2 = c->prm.tol_p * c->prm.tol_p * (c->tol2_scale > 0.0 ? c->tol2_scale : 1.0);
    const double by_vec = (double)nq * 16.0;
    if (warm) {
        if ((rc = pressure_restart(c))) return rc;  // r = b - A x, iteration count kept
    } else {
        k_fcg_init<<<b4, TH, 0, c->stream>>>(c->pb, c->px, c->pr, n4, tol2, c->prm.maxit_p, s, c->partials);
        c->n_launches += 1;
    }
    FS_CUDA(cudaGetLastError());
    long long k = 0;
    unsigned herr = 0;
    std::vector<std::pair<int, double>> hist;  // (iteration, r.r) at the host checks
    ProfIteration iteration(c);
    for (;;) {
        if ((rc = read_scal(c, 0, h, &herr))) return rc;
        if (h->done) break;
        if (k > (long long)c->prm.maxit_p + c->prm.check_every)
            return set_error(FS_ECUDA, "flexible CG: iteration flag never set");
        hist.push_back({h->iter, h->rr});
        size_t m = hist.size();
        while (m > 0 && hist[m - 1].first > h->iter - 200) m--;
        if (m > 0 && h->iter >= 200 && h->rr > 1e-2 * hist[m - 1].second) {
            h->status = FS_ENOCONV;
            break;
        }
        for (int b = 0; b < c->prm.check_every; b++, k++) {
            iteration(k);
            const int slot = (int)(k % FCG_M);
            const int nvalid = (int)std::min<long long>(k, FCG_M);
            Ring ring;
            for (int j = 0; j < FCG_M; j++) {
                const int sj = (int)(((k - 1 - j) % FCG_M + FCG_M) % FCG_M);
                ring.p[j] = f->p[sj];
                ring.q[j] = f->q[sj];
                ring.pq[j] = f->pq + sj;
            }
            // z = M r; where no null mode is removed from z, the network's part is added by the dots
            const float *e = nullptr;
            if ((rc = learned_apply(c, c->pr, c->pz, &s->done, c->singular ? nullptr : &e))) return rc;
            if ((rc = remove_null_mode(c, c->pz))) return rc;
            const bool samp = c->prof_on && (b % c->prof_period) == 0;
            cudaEvent_t e0 = samp ? prof_mark(c) : nullptr;
            launch_dep(k_fcg_dots, wave_blocks(c, nq, rd), TH, 0, c->stream, ql, nq, c->pz, e, c->pr, ring, nvalid, s, f->beta,
                                                                     c->partials);
            launch_dep(k_fcg_dir, wave_blocks(c, nq, ri), TH, 0, c->stream, ql, nq, c->pz, ring, nvalid, f->p[slot], s, f->beta);
            launch_dep(k_fcg_apply, wave_blocks(c, nq, ra), TH, 0, c->stream, ql, nq, f->p[slot], f->q[slot], c->cflag, L.P,
                                                                      L.PL, s, f->pq + slot, c->partials);
            launch_dep(k_fcg_update, wave_blocks(c, nq, ru), TH, 0, c->stream, ql, nq, c->px, c->pr, f->p[slot], f->q[slot], s,
                                                                       c->partials);
            cudaEvent_t e1 = samp ? prof_mark(c) : nullptr;
            // vectors streamed: dots 2 + nvalid, direction 2 + nvalid, operator ~3, update 6
            prof_add(c, K_FCG_VEC, e0, e1, by_vec * (13.0 + 2.0 * nvalid));
            c->n_launches += 4;
        }
        FS_CUDA(cudaGetLastError());
    }
    return check_wait_error(c, "flexible CG", herr);
}

}  // namespace fs
