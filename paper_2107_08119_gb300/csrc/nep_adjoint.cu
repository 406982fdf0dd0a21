// nep_adjoint.cu -- gradient of the force loss with respect to the network
// parameters, by a hand-written adjoint of the force path.
//
// The paper fits without gradients (SNES, Sec. II.D); this is the
// differentiable route to the same force term of the loss.  With residuals
// e_i = F_i - F_tar_i over the N atoms of the training set and
// L_f = sqrt(sum_i |e_i|^2 / (3N)) (Eq. 30), and F_i = sum_j (dU_i/dr_ij -
// dU_j/dr_ji) (Eqs. 4-5):
//   dL_f/dz = sum_i sum_j d/dz(dU_i/dr_ij) . (delta_i - delta_j),
//   delta_i = e_i / (3N L_f).
// dU_i/dr_ij = sum_nu G_i,nu dq_i,nu/dr_ij (Eq. 23) and q does not depend on
// z, so
//   dL_f/dz = sum_i sum_nu dG_i,nu/dz lambda_i,nu,
//   lambda_i,nu = sum_j dq_i,nu/dr_ij . (delta_i - delta_j).
// For the network of Eqs. 21-22, G_nu = sum_mu w2_mu (1 - x_mu^2) w1_mu,nu;
// with s_mu = sum_nu w1_mu,nu lambda_nu and t_mu = 1 - x_mu^2, per atom:
//   d/dw2_mu    t_mu s_mu
//   d/db1_mu    2 w2_mu x_mu t_mu s_mu
//   d/dw1_mu,k  w2_mu t_mu lambda_k - 2 w2_mu x_mu t_mu s_mu q_k
//   d/db2       0
// The angular pair derivative follows the harmonic form of the force path:
// dq_nl/dr . d = sum_m 2 c_lm S_nlm (g_n' Z_lm (rhat . d) + g_n grad_u Z_lm . d_t),
// d_t = (d - (rhat . d) rhat) / r.
//
// Both passes recompute descriptors and pair derivatives from the positions;
// the only per-pair array is the forward's partial forces, which define F.
// Kernels (the first, second and fourth with 128 threads on 8, 16 or 32 atoms,
// as the site pass, nep_site_block.cuh):
//   k_adj_site    q, network, dU_i/dr_ij for every CSR pair of the atom
//   k_adj_force   F_i = sum_p (pf[p] - pf[rev[p]]), e_i, block sums of |e|^2
//   k_adj_loss    L_f from the block sums (one block, fixed order)
//   k_adj_lambda  q and S again, lambda_i, the network terms; the block sums
//                 every parameter's terms over its atoms in FP32
//   k_adj_grad    per parameter, the block sums in FP64 in a fixed order
// Every sum has a fixed order: the gradient is bitwise reproducible.
#include <cmath>
#include <type_traits>

#include "nep_dataset.cuh"
#include "nep_site_block.cuh"

namespace nep {
namespace {

constexpr int kMostPar = (kNdes + 2) * kMaxNeu + 1;  // parameters of the largest network
constexpr int kAdjWords = 2;  // own-slot words per thread: 256 pairs per atom at 32 atoms per block
static_assert(kDsCap <= 32 * kAdjWords * kSiteWarps, "a training set's pairs of an atom have own-slot bits");

inline int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }

// floats per atom row of the backward's block reduction: lambda[32], q[32],
// then a, c, t*s per neuron; odd so a warp writing one column of its rows
// hits 32 different banks
__host__ __device__ __forceinline__ int adj_row_stride(int nn) { return (kNdes * 2 + 3 * nn) | 1; }

// The site pass over the CSR pairs.  One thread per atom (255 registers, 650
// warps for a 200-structure set) ran its ~30k instructions in series: 68 us,
// now 46.
template <int AT>
__global__ void __launch_bounds__(kSiteThreads, 5) k_adj_site(int N, const int* __restrict__ sid,
                                                              const Box* __restrict__ boxes,
                                                              const float* __restrict__ xr,
                                                              const long long* __restrict__ pstart,
                                                              const int* __restrict__ pj, const float* __restrict__ z,
                                                              int n_par, SiteParams P, float* __restrict__ pf,
                                                              unsigned* err)
{
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * AT + lane % AT;
    const bool active = i < N;
    const int ia = active ? i : 0;
    const long long p0 = pstart[ia];
    const int cnt = active ? (int)(pstart[ia + 1] - p0) : 0;
    const Box box = boxes[sid[ia]];
    float uh = 0.f, ul = 0.f;
    site_block<DescSi, AT, kAdjWords>(CsrPairs{pj + p0, pf + 3 * p0}, i, active, N, cnt, xr, box, z, n_par, P, nullptr,
                                      uh, ul);
    if (threadIdx.x < AT && active && !isfinite(uh)) atomicOr(err, kErrNonFinite);
}

// F_i, e_i and the block sums of |e|^2: the block's threads gather the terms
// of 16 or more pairs per atom at a time into shared memory, and one thread per
// atom and component adds them in pair order (14.7 -> 9.6 us).
template <int AT>
__global__ void __launch_bounds__(kSiteThreads) k_adj_force(int N, const long long* __restrict__ pstart,
                                                            const long long* __restrict__ rev,
                                                            const float* __restrict__ pf,
                                                            const float* __restrict__ f_tar, float4* __restrict__ res,
                                                            double* __restrict__ part, unsigned* err)
{
    constexpr int WAYS = SiteSplit<AT>::WAYS, PER = 4, CH = WAYS * PER;
    __shared__ float s_t[3][CH][AT];
    __shared__ float s_F[3][AT];
    const int at = threadIdx.x % AT, way = threadIdx.x / AT;
    const int i = blockIdx.x * AT + at;
    const bool active = i < N;
    const long long p0 = active ? pstart[i] : 0;
    const int cnt = active ? (int)(pstart[i + 1] - p0) : 0;
    const int kmax = __reduce_max_sync(0xffffffffu, cnt);
    float F = 0.f;  // component `way` (way < 3)
    for (int k0 = 0; k0 < kmax; k0 += CH) {
        long long r[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int k = k0 + WAYS * u + way;
            r[u] = k < cnt ? rev[p0 + k] : 0;
        }
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int s = WAYS * u + way, k = k0 + s;
            if (k < cnt)
#pragma unroll
                for (int c = 0; c < 3; ++c) s_t[c][s][at] = pf[3 * (p0 + k) + c] - pf[3 * r[u] + c];
        }
        __syncthreads();
        if (way < 3) {
            const int m = min(CH, cnt - k0);
            for (int s = 0; s < m; ++s) F += s_t[way][s][at];
        }
        __syncthreads();
    }
    if (way < 3) s_F[way][at] = F;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double sq = 0.0;
    if (active && threadIdx.x < AT) {
        const float ex = s_F[0][at] - f_tar[(size_t)3 * i], ey = s_F[1][at] - f_tar[(size_t)3 * i + 1],
                    ez = s_F[2][at] - f_tar[(size_t)3 * i + 2];
        res[i] = make_float4(ex, ey, ez, 0.f);
        if (!(isfinite(ex) && isfinite(ey) && isfinite(ez))) atomicOr(err, kErrNonFinite);
        sq = (double)ex * ex + (double)ey * ey + (double)ez * ez;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (threadIdx.x == 0) part[blockIdx.x] = sq;
}

// sums[0] = sum |e|^2, sums[1] = L_f; loss (optional) = L_f.
__global__ void k_adj_loss(int nblocks, int N, const double* __restrict__ part, double* __restrict__ sums,
                           double* __restrict__ loss)
{
    double v[1] = {0.0};
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) v[0] += part[b];
    __shared__ double tot;
    block_sum_store<1>(v, &tot);
    __syncthreads();
    if (threadIdx.x == 0) {
        const double L = sqrt(tot / (3.0 * (double)N));
        sums[0] = tot;
        sums[1] = L;
        if (loss) loss[0] = L;
    }
}

// One harmonic's share of lambda for a pair: with alpha = Z (rhat . d) and
// beta = grad_u Z . d_t, lambda_nl += A_nlm (g_n' alpha + g_n beta); s_A the
// atom's column of A.
template <int AT, int LM>
__device__ __forceinline__ void adj_terms(const float* s_A, const ShFast& sh, const float (&g)[kNA],
                                          const float (&dg)[kNA], float e, float tx, float ty, float tz,
                                          float (&lam)[kNdes])
{
    if constexpr (LM < kLM) {
        float alpha = 0.f, beta = 0.f;
        float d[3] = {0.f, 0.f, 0.f};
        sh_add<LM>(sh, 1.f, 1.f, alpha, d);
        alpha *= e;
        beta = fmaf(d[0], tx, fmaf(d[1], ty, d[2] * tz));
#pragma unroll
        for (int n = 0; n < kNA; ++n)
            lam[kNR + n * kLmax + sh_l(LM)] = fmaf(s_A[site_block_at<DescSi, AT>(n, LM)],
                                                   fmaf(dg[n], alpha, g[n] * beta),
                                                   lam[kNR + n * kLmax + sh_l(LM)]);
        adj_terms<AT, LM + 1>(s_A, sh, g, dg, e, tx, ty, tz, lam);
    }
}

// Shared memory of k_adj_lambda: that of the site pass, the partial lambdas
// ([WAYS][32 v][AT]) from the coefficients on, and after both a row per atom,
// at this float offset.
template <int AT>
__host__ __device__ inline size_t adj_rows_at(int n_par, int nn)
{
    const size_t site = site_block_smem<DescSi, AT>(n_par, nn) / sizeof(float);
    const size_t lam = (size_t)(n_par + 31) / 32 * 32 + (size_t)SiteSplit<AT>::WAYS * kNdes * AT;
    return site > lam ? site : lam;
}
template <int AT>
size_t adj_lambda_smem(int n_par, int nn)
{
    return sizeof(float) * (adj_rows_at<AT>(n_par, nn) + AT * adj_row_stride(nn));
}

// lambda and the network terms.  Each thread sums its own pairs' shares of
// lambda against the coefficients in shared memory; the WAYS partial lambdas
// are added in order.  One thread per atom: 83 us for a 200-structure set, now
// 66.
template <int AT>
__global__ void __launch_bounds__(kSiteThreads, 4) k_adj_lambda(int N, const int* __restrict__ sid,
                                                                const Box* __restrict__ boxes,
                                                                const float* __restrict__ xr,
                                                                const long long* __restrict__ pstart,
                                                                const int* __restrict__ pj,
                                                                const float4* __restrict__ res,
                                                                const double* __restrict__ sums,
                                                                const float* __restrict__ z, int n_par, SiteParams P,
                                                                float* __restrict__ part)
{
    constexpr int SUB = SiteSplit<AT>::SUB, WAYS = SiteSplit<AT>::WAYS;
    extern __shared__ __align__(16) float s_site[];
    const int nn = P.n_neu;
    const int stride = adj_row_stride(nn);
    const SiteShared<DescSi, AT> sh(s_site, n_par, nn);
    float* rows = s_site + adj_rows_at<AT>(n_par, nn);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int at = lane % AT, way = SUB * warp + lane / AT;
    const int i = blockIdx.x * AT + at;
    const bool active = i < N;
    const int ia = active ? i : 0;
    const long long p0 = pstart[ia];
    const int cnt = active ? (int)(pstart[ia + 1] - p0) : 0;
    const Box box = boxes[sid[ia]];
    const double L = sums[1];
    const float scale = L > 0.0 ? (float)(1.0 / (3.0 * (double)N * L)) : 0.f;
    const CsrPairs pairs{pj + p0, nullptr};
    float* row = rows + at * stride;

    float hi[3], li[3], zi;
    load_pos(xr, ia, hi, li, zi);
    unsigned kept[kAdjWords], ang[kAdjWords];
    site_block_sums<DescSi, AT, kAdjWords>(pairs, cnt, xr, box, z, n_par, P, sh, hi, li, zi, kept, ang);
    for (int v = way; v < kNdes; v += WAYS) row[kNdes + v] = active ? sh.q[v * AT + at] : 0.f;
    // A_nlm = 2 c_lm S_nlm
    for (int n = way; n < kNA; n += WAYS)
#pragma unroll
        for (int m = 0; m < kLM; ++m) {
            const int f = 2 * ((m >> 1) * kNA + n) + (m & 1);  // site_block_at
            sh.A[(f >> 2) * 4 * AT + 4 * at + (f & 3)] *= 2.f * sh_c(m);
        }
    __syncthreads();
    float lam[kNdes];
#pragma unroll
    for (int v = 0; v < kNdes; ++v) lam[v] = 0.f;
    const float4 ei = res[ia];
    const float di[3] = {ei.x * scale, ei.y * scale, ei.z * scale};
#pragma unroll
    for (int w = 0; w < kAdjWords; ++w) {
#pragma unroll 1
        for (unsigned rest = kept[w]; rest; rest &= rest - 1) {
            const int b = __ffs((int)rest) - 1;
            const int v = pairs.value(WAYS * (32 * w + b) + way);
            const int j = v & 0xFFFFFF;
            float hj[3], lj[3], zj;
            load_pos(xr, j, hj, lj, zj);
            const float4 ej = res[j];
            float r[3];
            pair_vector(v >> 24, hi, li, hj, lj, box, r[0], r[1], r[2]);
            const float d2 = fmaf(r[0], r[0], fmaf(r[1], r[1], r[2] * r[2]));
            const float dd[3] = {fmaf(-ej.x, scale, di[0]), fmaf(-ej.y, scale, di[1]), fmaf(-ej.z, scale, di[2])};
            const float d = sqrtf(d2);
            const float inv = 1.f / d;
            const float u[3] = {r[0] * inv, r[1] * inv, r[2] * inv};
            const float e = fmaf(u[0], dd[0], fmaf(u[1], dd[1], u[2] * dd[2]));
            const float wz = pair_weight(P, zi, zj);
            if (d2 < P.rcR2) {
                float g[kNR], dg[kNR];
                radial_g_dg<kNR>(d, P.rcR, P.inv_rcR, g, dg, wz);
#pragma unroll
                for (int a = 0; a < kNR; ++a) lam[a] = fmaf(dg[a], e, lam[a]);
            }
            if ((ang[w] >> b) & 1u) {
                float g[kNA], dg[kNA];
                radial_g_dg<kNA>(d, P.rcA, P.inv_rcA, g, dg, wz);
                const float tx = fmaf(-e, u[0], dd[0]) * inv, ty = fmaf(-e, u[1], dd[1]) * inv,
                            tz = fmaf(-e, u[2], dd[2]) * inv;
                ShFast s;
                s.set(u[0], u[1], u[2]);
                adj_terms<AT, 0>(sh.A + 4 * at, s, g, dg, e, tx, ty, tz, lam);
            }
        }
    }
    __syncthreads();  // A and q are read
    float* s_lam = sh.A;
#pragma unroll
    for (int v = 0; v < kNdes; ++v) s_lam[(way * kNdes + v) * AT + at] = lam[v];
    __syncthreads();
    for (int v = way; v < kNdes; v += WAYS) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < WAYS; ++w) t += s_lam[(w * kNdes + v) * AT + at];
        row[v] = active ? t : 0.f;
    }
    __syncthreads();

    // network terms: x_mu again from q (row), s_mu = w1_mu . lambda
    const float* b1 = sh.w + nn * kNdes;
    const float* w2 = b1 + nn;
    float q[kNdes];
#pragma unroll
    for (int v = 0; v < kNdes; ++v) {
        q[v] = row[kNdes + v];
        lam[v] = row[v];
    }
    for (int mu = way; mu < nn; mu += WAYS) {
        const float* w = sh.w + mu * kNdes;
        float a = -b1[mu], s = 0.f;
#pragma unroll
        for (int v = 0; v < kNdes; ++v) {
            a = fmaf(w[v], q[v], a);
            s = fmaf(w[v], lam[v], s);
        }
        const float x = tanhf(a);
        const float t = fmaf(-x, x, 1.f);
        const float ts = active ? t * s : 0.f;
        row[2 * kNdes + mu] = active ? w2[mu] * t : 0.f;             // multiplies lambda_k in d/dw1
        row[2 * kNdes + nn + mu] = -2.f * w2[mu] * x * ts;            // multiplies q_k in d/dw1; -d/db1
        row[2 * kNdes + 2 * nn + mu] = ts;                            // d/dw2
    }
    __syncthreads();

    // block sums of every parameter's per-atom terms
    const int nw1 = nn * kNdes;
    for (int o = threadIdx.x; o < n_par; o += kSiteThreads) {
        float s = 0.f;
        if (o < nw1) {
            const int mu = o / kNdes, k = o % kNdes;
#pragma unroll 4
            for (int r = 0; r < AT; ++r) {
                const float* R = rows + r * stride;
                s = fmaf(R[2 * kNdes + mu], R[k], fmaf(R[2 * kNdes + nn + mu], R[kNdes + k], s));
            }
        } else if (o < nw1 + nn) {
            for (int r = 0; r < AT; ++r) s -= rows[r * stride + 2 * kNdes + nn + o - nw1];
        } else if (o < n_par - 1) {
            for (int r = 0; r < AT; ++r) s += rows[r * stride + 2 * kNdes + 2 * nn + o - nw1 - nn];
        }
        part[(size_t)blockIdx.x * n_par + o] = s;
    }
}

// grad[o]: the block sums of 32 parameters per block, eight warps each adding
// every eighth row in order, then the warps in order (12 us; one thread per
// parameter walking a quarter of these rows took 17 us).
constexpr int kAdjGradWarps = 8;
__global__ void __launch_bounds__(32 * kAdjGradWarps) k_adj_grad(int nblocks, int n_par,
                                                                 const float* __restrict__ part,
                                                                 const double* __restrict__ seed,
                                                                 double* __restrict__ grad)
{
    __shared__ double s_sum[kAdjGradWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (o < n_par)
#pragma unroll 8
        for (int b = warp; b < nblocks; b += kAdjGradWarps) s += (double)part[(size_t)b * n_par + o];
    s_sum[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || o >= n_par) return;
    s = 0.0;
#pragma unroll
    for (int w = 0; w < kAdjGradWarps; ++w) s += s_sum[w][lane];
    grad[o] = seed ? s * seed[0] : s;
}

template <class T>
int adj_alloc(T** p, size_t count)
{
    if (count == 0) count = 1;
    cudaError_t e = cudaMalloc((void**)p, count * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        set_error("cudaMalloc of %zu bytes failed: %s", count * sizeof(T), cudaGetErrorString(e));
        return NEP_ERR_OOM;
    }
    return NEP_OK;
}

int ensure_adjoint(nep_model* m, nep_dataset* ds)
{
    AdjointScratch& a = ds->adj;
    if (a.pf) return NEP_OK;
    const int nb = site_blocks(ds->N);
    int rc;
    if ((rc = adj_alloc(&a.pf, (size_t)3 * ds->n_pairs)) || (rc = adj_alloc(&a.res, (size_t)4 * ds->N)) ||
        (rc = adj_alloc(&a.z, (size_t)m->n_par)) || (rc = adj_alloc(&a.part, (size_t)nb * (m->n_par + 1) / 2)) ||
        (rc = adj_alloc(&a.sums, 2))) {
        free_adjoint(a);
        return rc;
    }
    a.n_blocks = nb;
    a.ready = false;
    return NEP_OK;
}

// more than the default shared memory, where needed (an attribute call costs as
// much host time as a launch): `most` bytes, what the largest network takes, as
// the limit is the kernel's and not the model's
template <class K>
int allow_shared(K kern, size_t bytes, size_t most)
{
    if (bytes <= kDefaultShared) return NEP_OK;
    return cuda_fail(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most),
                     "adjoint kernel shared memory");
}

// f(std::integral_constant<int, AT>) for the atoms per block of N atoms
template <class F>
int by_atoms_per_block(int N, F f)
{
    switch (site_atoms_per_block(N)) {
    case 8: return f(std::integral_constant<int, 8>());
    case 16: return f(std::integral_constant<int, 16>());
    default: return f(std::integral_constant<int, 32>());
    }
}

SiteParams site_params(const nep_model* m, int typed)
{
    SiteParams P;
    P.typed = typed;
    P.w = nullptr;
    P.n_neu = m->hp.n_neu;
    P.rcR = (float)m->hp.rc_R;
    P.rcA = (float)m->hp.rc_A;
    P.rcR2 = P.rcR * P.rcR;
    P.rcA2 = P.rcA * P.rcA;
    P.inv_rcR = 1.f / P.rcR;
    P.inv_rcA = 1.f / P.rcA;
    return P;
}

}  // namespace

void free_adjoint(AdjointScratch& a)
{
    if (a.pf) cudaFree(a.pf);
    if (a.res) cudaFree(a.res);
    if (a.z) cudaFree(a.z);
    if (a.part) cudaFree(a.part);
    if (a.sums) cudaFree(a.sums);
    a = AdjointScratch();
}

}  // namespace nep

using namespace nep;

extern "C" {

int nep_force_loss(nep_model* m, nep_dataset* ds, const float* z, double* loss_f, void* stream)
{
    if (!m || !ds || ds->m != m || !z) {
        set_error("nep_force_loss: NULL argument or dataset of another model");
        return NEP_ERR_ARG;
    }
    int rc = ensure_adjoint(m, ds);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    AdjointScratch& a = ds->adj;
    const int N = ds->N, n_par = m->n_par, nb = a.n_blocks;
    rc = cuda_fail(cudaMemcpyAsync(a.z, z, sizeof(float) * n_par, cudaMemcpyDeviceToDevice, st),
                   "nep_force_loss: parameter copy");
    if (rc) return rc;
    rc = by_atoms_per_block(N, [&](auto tag) {
        constexpr int AT = decltype(tag)::value;
        const size_t smem = site_block_smem<DescSi, AT>(n_par, m->hp.n_neu);
        const int r = allow_shared(k_adj_site<AT>, smem, site_block_smem<DescSi, AT>(kMostPar, kMaxNeu));
        if (r) return r;
        k_adj_site<AT><<<nb, kSiteThreads, smem, st>>>(N, ds->sid, ds->boxes, ds->xr, ds->pstart, ds->pj, a.z, n_par,
                                                       site_params(m, ds->typed), a.pf, m->d_err);
        k_adj_force<AT><<<nb, kSiteThreads, 0, st>>>(N, ds->pstart, ds->rev, a.pf, ds->f_tar,
                                                     reinterpret_cast<float4*>(a.res), a.part, m->d_err);
        return (int)NEP_OK;
    });
    if (rc) return rc;
    k_adj_loss<<<1, 256, 0, st>>>(nb, N, a.part, a.sums, loss_f);
    rc = cuda_fail(cudaGetLastError(), "force-loss forward kernels");
    if (rc) return rc;
    a.ready = true;
    return NEP_OK;
}

int nep_force_loss_backward(nep_model* m, nep_dataset* ds, const double* seed, double* grad, void* stream)
{
    if (!m || !ds || ds->m != m || !grad) {
        set_error("nep_force_loss_backward: NULL argument or dataset of another model");
        return NEP_ERR_ARG;
    }
    if (!ds->adj.ready) {
        set_error("nep_force_loss_backward: no nep_force_loss on this dataset before it");
        return NEP_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    AdjointScratch& a = ds->adj;
    const int N = ds->N, n_par = m->n_par, nb = a.n_blocks;
    const int rc = by_atoms_per_block(N, [&](auto tag) {
        constexpr int AT = decltype(tag)::value;
        const size_t smem = adj_lambda_smem<AT>(n_par, m->hp.n_neu);
        const int r = allow_shared(k_adj_lambda<AT>, smem, adj_lambda_smem<AT>(kMostPar, kMaxNeu));
        if (r) return r;
        k_adj_lambda<AT><<<nb, kSiteThreads, smem, st>>>(N, ds->sid, ds->boxes, ds->xr, ds->pstart, ds->pj,
                                                         reinterpret_cast<const float4*>(a.res), a.sums, a.z, n_par,
                                                         site_params(m, ds->typed), reinterpret_cast<float*>(a.part));
        return (int)NEP_OK;
    });
    if (rc) return rc;
    k_adj_grad<<<blocks_for(n_par, 32), 32 * kAdjGradWarps, 0, st>>>(nb, n_par, reinterpret_cast<float*>(a.part), seed,
                                                                     grad);
    return cuda_fail(cudaGetLastError(), "force-loss adjoint kernels");
}

}  // extern "C"
