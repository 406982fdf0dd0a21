// nep_force.cu -- the FP32 force path: site energies + partial forces, then
// force / per-atom virial assembly, and deterministic FP64 reductions.
//
// Pass A (k_site, nep_site_block.cuh): four warps per 32 atoms run the
// descriptor sums, the network and the partial forces dU_i/dr_ij of all their
// pairs.  Partial forces go to pf[k][i] as float4 records.
// Pass B (k_assemble): one thread per atom gathers its own p_ij and the
// neighbours' p_ji through the reverse-pair index: F_i = sum_j (p_ij - p_ji)
// and W_i = sum_j r_ij (x) p_ji (Eqs. 4-6).  In MD mode the same pass applies
// the second velocity-Verlet half kick and accumulates E_kin and the heat
// current J = sum_i W_i . v_i (Eq. 7) without storing W.
// Totals are summed per block in FP64 and then by one block in a fixed order,
// so every result is bitwise reproducible run to run.
#include <cstdio>

#include "nep_site_block.cuh"

namespace nep {

namespace {

constexpr int kAsmThreads = 128;
constexpr int kMaskSlots = 96;  // slots per atom covered by the in-cutoff mask words

// D: descriptor sizes of the model (DescSi: 32 descriptors, DescPbTe: 41).
// WORDS: 32-slot words of own-slot bits per thread (1 covers 128 slots per
// atom, 3 the largest capacity).
template <class D, int WORDS>
__global__ void __launch_bounds__(kSiteThreads, 5) k_site(int n, int m_cap, const int* __restrict__ count,
                                                          const int* __restrict__ nbr, const float* __restrict__ xr, Box box,
                                                          const float* __restrict__ z, int n_par, SiteParams P,
                                                          float* __restrict__ pf, double* __restrict__ e_atom,
                                                          double* __restrict__ e_partials, unsigned* err,
                                                          unsigned* __restrict__ mask)
{
    const int i0 = blockIdx.x * kSiteAtoms;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = i0 + lane;
    const bool active = i < n;
    const int cnt = active ? min(count[i], m_cap) : 0;
    float uh, ul;
    site_block<D, WORDS>(i, active, n, cnt, nbr, xr, box, z, n_par, P, pf, mask, uh, ul);
    if (warp != 0) return;  // warp 0 holds the site energies
    double e = 0.0;
    if (active) {
        e = (double)uh + (double)ul;
        if (e_atom) e_atom[i] = e;
        if (!isfinite(uh)) atomicOr(err, kErrNonFinite);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane == 0) e_partials[blockIdx.x] = e;
}

// Totals per block: [0..8] virial, and in MD mode [9] E_kin, [10..12] J.
template <bool MD>
__global__ void __launch_bounds__(kAsmThreads) k_assemble(int n, int m_cap, float rc2max, const int* __restrict__ count,
                                                          const int* __restrict__ nbr, const int* __restrict__ rev,
                                                          const float* __restrict__ xr,
                                                          Box box, const float* __restrict__ pf,
                                                          float* __restrict__ force, float* __restrict__ virial_atom,
                                                          double* __restrict__ partials, unsigned* err,
                                                          double* __restrict__ vel, double hdtm, double kef,
                                                          const unsigned* __restrict__ mask)
{
    constexpr int K = MD ? 13 : 9;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    if (i < n) {
        // the list is read straight from global memory: staging it in shared
        // memory (as the site pass does) cost this pass occupancy and time
        const SlotTable T{nbr, n, i};
        float F[3], W[9];
        assemble_atom(i, n, m_cap, rc2max, count, T, rev, xr, box, pf, F, W, mask);
        if (!(isfinite(F[0]) && isfinite(F[1]) && isfinite(F[2]))) atomicOr(err, kErrNonFinite);
        if (force) {
            force[i] = F[0];
            force[(size_t)n + i] = F[1];
            force[(size_t)2 * n + i] = F[2];
        }
        if (virial_atom)
#pragma unroll
            for (int c = 0; c < 9; ++c) virial_atom[(size_t)c * n + i] = W[c];
#pragma unroll
        for (int c = 0; c < 9; ++c) acc[c] = (double)W[c];
        if constexpr (MD) {
            double v[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[c] = vel[(size_t)c * n + i] + hdtm * (double)F[c];
                vel[(size_t)c * n + i] = v[c];
            }
            acc[9] = kef * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
            // J^a = sum_b W^{ab} v^b, FP32 products accumulated in FP64
#pragma unroll
            for (int a = 0; a < 3; ++a)
                acc[10 + a] = (double)(W[3 * a] * (float)v[0]) + (double)(W[3 * a + 1] * (float)v[1]) +
                              (double)(W[3 * a + 2] * (float)v[2]);
        }
    }
    block_sum_store<K>(acc, partials + (size_t)blockIdx.x * K);
}

// out[k] = sum_b partials[b * ncomp + k]: one warp per component, each lane
// summing a fixed stride of blocks, then a fixed shuffle tree (deterministic).
__global__ void k_reduce(const double* __restrict__ partials, int nblocks, int ncomp, double* __restrict__ out)
{
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k >= ncomp) return;
    double s = 0.0;
    // unrolled so that eight loads are in flight ahead of the (ordered) adds
#pragma unroll 8
    for (int b = lane; b < nblocks; b += 32) s += partials[(size_t)b * ncomp + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[k] = s;
}

inline int blocks_for(int n, int t) { return (n + t - 1) / t; }

template <class D>
int launch_site(const ForceArgs& a, NeighborList& nl, int n, double* e_atom, double* e_partials, unsigned* d_err,
                cudaStream_t st, int& nblocks)
{
    SiteParams P;
    P.w = nullptr;
    P.n_neu = a.n_neu;
    P.rcR = a.rcR;
    P.rcA = a.rcA;
    P.rcR2 = a.rcR * a.rcR;
    P.rcA2 = a.rcA * a.rcA;
    P.inv_rcR = 1.f / a.rcR;
    P.inv_rcA = 1.f / a.rcA;
    P.typed = a.typed;
    const int n_par = (D::Ndes + 2) * a.n_neu + 1;
    nblocks = site_blocks(n);
    const size_t smem = site_block_smem<D>(n_par, a.n_neu);
    auto kern = nl.m_cap <= 128 ? k_site<D, 1> : k_site<D, 3>;
    int rc = cuda_fail(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                       "site kernel shared memory");
    if (!rc)
        rc = cuda_fail(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            cudaSharedmemCarveoutMaxShared), "site kernel shared memory");
    if (rc) return rc;
    nl.mask_set = nl.m_cap <= kMaskSlots && nl.mask != nullptr;
    kern<<<nblocks, kSiteThreads, smem, st>>>(n, nl.m_cap, nl.count, nl.nbr, nl.xr, a.box, a.z, n_par, P, nl.pf,
                                              e_atom, e_partials, d_err, nl.mask_set ? nl.mask : nullptr);
    return cuda_fail(cudaGetLastError(), "site kernel");
}

}  // namespace

int launch_site_partial_forces(const ForceArgs& a, NeighborList& nl, int n, double* e_atom, double* e_partials,
                               unsigned* d_err, cudaStream_t st, int& nblocks)
{
    if (a.nr == DescPbTe::NR && a.na == DescPbTe::NA)
        return launch_site<DescPbTe>(a, nl, n, e_atom, e_partials, d_err, st, nblocks);
    if (a.nr != DescSi::NR || a.na != DescSi::NA) {
        set_error("no site kernel for %d radial and %d angular orders", a.nr, a.na);
        return NEP_ERR_UNSUPPORTED;
    }
    return launch_site<DescSi>(a, nl, n, e_atom, e_partials, d_err, st, nblocks);
}

int launch_assemble(const AssembleArgs& a, NeighborList& nl, int n, float* force, float* virial_atom,
                    double* partials, unsigned* d_err, cudaStream_t st, int& nblocks, int& ncomp)
{
    nblocks = blocks_for(n, kAsmThreads);
    const float rc2 = a.rc_max * a.rc_max;
    const bool md = a.vel != nullptr;
    ncomp = md ? 13 : 9;
    auto kern = md ? k_assemble<true> : k_assemble<false>;
    kern<<<nblocks, kAsmThreads, 0, st>>>(n, nl.m_cap, rc2, nl.count, nl.nbr, nl.rev, nl.xr, a.box, nl.pf,
                                          force, virial_atom, partials, d_err, md ? a.vel : nullptr,
                                          md ? a.half_dt_over_m : 0.0, md ? a.ke_factor : 0.0,
                                          nl.mask_set ? nl.mask : nullptr);
    return cuda_fail(cudaGetLastError(), "assemble kernel");
}

int launch_reduce(const double* partials, int nblocks, int ncomp, double* out, cudaStream_t st)
{
    k_reduce<<<1, 32 * ncomp, 0, st>>>(partials, nblocks, ncomp, out);
    return cuda_fail(cudaGetLastError(), "reduce kernel");
}

}  // namespace nep
