// nep_force.cu -- the FP32 force path: site energies + partial forces, then
// force / per-atom virial assembly, and deterministic FP64 reductions.
//
// Pass A (k_site, nep_site_block.cuh): four warps per 32 atoms run the
// descriptor sums, the network and the partial forces dU_i/dr_ij of all their
// pairs.  Partial forces go to pf[k][i] as float4 records.
// Pass B (k_assemble): the block's threads gather the slots of its atoms, own
// p_ij and the neighbours' p_ji through the reverse-pair index, into a shared
// tile, and then sum F_i = sum_j (p_ij - p_ji) and W_i = sum_j r_ij (x) p_ji
// (Eqs. 4-6), each sum in one thread in slot order.  In MD mode the same pass
// applies the second velocity-Verlet half kick and accumulates E_kin and the
// heat current J = sum_i W_i . v_i (Eq. 7) without storing W.
// Totals are summed per block in FP64 and then by one block per total in a
// fixed order, so every result is bitwise reproducible run to run.
#include <cstdio>

#include "nep_site_block.cuh"

namespace nep {

namespace {

constexpr int kAsmThreads = 128;
constexpr int kAsmPer = 2;  // slots of a tile per thread, gathered together
constexpr int kMaskSlots = 96;  // slots per atom covered by the in-cutoff mask words

// D: descriptor sizes of the model (DescSi: 32 descriptors, DescPbTe: 41).
// AT: atoms per block.  WORDS: 32-bit words of own-slot bits per thread.
template <class D, int AT, int WORDS>
__global__ void __launch_bounds__(kSiteThreads, 5) k_site(int n, int m_cap, const int* count,
                                                          const int* nbr, const float* xr,
                                                          Box box, const float* z, int n_par,
                                                          SiteParams P, float* pf,
                                                          double* e_atom,
                                                          double* e_partials, unsigned* err,
                                                          unsigned* mask)
{
    const int block = block_after();
    const int lane = threadIdx.x & 31;
    const int i = block * AT + lane % AT;
    const bool active = i < n;
    const int cnt = active ? min(count[i], m_cap) : 0;
    float uh, ul;
    const SlotMajorPairs pairs{nbr, reinterpret_cast<float4*>(pf), (size_t)n, active ? i : 0};
    site_block<D, AT, WORDS>(pairs, i, active, n, cnt, xr, box, z, n_par, P, mask, uh, ul);
    if (threadIdx.x >= 32) return;  // the first AT lanes hold the site energies
    double e = 0.0;
    if (active && lane < AT) {
        e = (double)uh + (double)ul;
        if (e_atom) e_atom[i] = e;
        if (!isfinite(uh)) atomicOr(err, kErrNonFinite);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane == 0) e_partials[block] = e;
}

// Totals of block b, [component][gridDim.x]: components 0..8 the virial, and
// in MD mode 9 E_kin, 10..12 J.
//
// What bounds it: the latency of two dependent loads per slot (list value and
// reverse slot, then the neighbour's position and p_ji) at small sizes, L2
// gathers (88 bytes per slot) at large ones.  A thread per atom walks its ~28
// kept slots one after the other: 23-26 us at any size below 40k atoms, 60 us
// with the 64 slots of the split model.  Here a tile holds 256 (slot, atom)
// entries, two per thread with all their loads in flight, and the 12 sums of an
// atom are spread over its threads.  Measured (thread per atom -> this): 512
// atoms 22.5 -> 6.4 us, 4096 26 -> 7.0, 13824 24 -> 9.9, 32768 25 -> 16.1, 46656
// 26.3 -> 22.3, 125000 39.6 -> 51.8; split model 18928 62 -> 24, 64000 97 -> 72.
// Four entries per thread (16 warps per SM): 66 us at 125000, 89 at 64000 of
// the split model; one entry: 50 and 78.
template <bool MD, int AT>
__global__ void __launch_bounds__(kAsmThreads, 8) k_assemble(int n, int m_cap, float rc2max, const int* count,
                                                          const int* nbr, const int* rev,
                                                          const float* xr, Box box,
                                                          const float* pf, float* force,
                                                          float* virial_atom,
                                                          double* partials, unsigned* err,
                                                          double* vel, double hdtm, double kef,
                                                          const unsigned* mask)
{
    constexpr int WAYS = kAsmThreads / AT;       // threads per atom
    constexpr int CH = WAYS * kAsmPer;           // slots per tile
    constexpr int ROWS = 9;                      // r_ij, p_ji, p_ij - p_ji
    constexpr int NC = (12 + WAYS - 1) / WAYS;   // sums per thread: F (0..2), W (3..11)
    constexpr float kNone = 1e30f;               // r_x of an entry that is not a pair within the cutoff
    __shared__ float s_t[ROWS][CH][AT];
    __shared__ float s_sum[12][AT];
    __shared__ float s_v[3][AT];
    const int block = block_after();
    const int at = threadIdx.x % AT, way = threadIdx.x / AT;
    const int i = block * AT + at;
    const bool active = i < n;
    const int ia = active ? i : 0;
    float hi[3], li[3];
    load_pos(xr, ia, hi, li);
    int cnt = active ? min(count[ia], m_cap) : 0;
    // the in-cutoff bits of the first 96 slots (the lists end there when they are given)
    unsigned mb[3] = {~0u, ~0u, ~0u};
    if (mask) {
#pragma unroll
        for (int w = 0; w < 3; ++w) mb[w] = active ? mask[(size_t)w * n + ia] : 0u;
        cnt = mb[2] ? 96 - __clz((int)mb[2]) : mb[1] ? 64 - __clz((int)mb[1]) : mb[0] ? 32 - __clz((int)mb[0]) : 0;
    }
    // the velocities that row 0 kicks at the end, loaded ahead of the slots
    double w[3] = {0.0, 0.0, 0.0};
    if (MD && way == 0 && active)
#pragma unroll
        for (int c = 0; c < 3; ++c) w[c] = vel[(size_t)c * n + i];
    const int kmax = __reduce_max_sync(0xffffffffu, cnt);  // the same in every warp
    const float4* pf4 = reinterpret_cast<const float4*>(pf);
    float acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.f;
    int v[kAsmPer], kr[kAsmPer];
    auto load_idx = [&](int k0) {
#pragma unroll
        for (int u = 0; u < kAsmPer; ++u) {
            const int k = k0 + WAYS * u + way;
            const unsigned word = k < 32 ? mb[0] : k < 64 ? mb[1] : mb[2];
            v[u] = -1;
            if (k < cnt && (!mask || ((word >> (k & 31)) & 1u))) {
                v[u] = nbr[(size_t)k * n + ia];
                kr[u] = rev[(size_t)k * n + ia];
            }
        }
    };
    load_idx(0);
#pragma unroll 1
    for (int k0 = 0; k0 < kmax; k0 += CH) {
        float hj[kAsmPer][3], lj[kAsmPer][3];
        float4 po[kAsmPer], pq[kAsmPer];
        int code[kAsmPer];
#pragma unroll
        for (int u = 0; u < kAsmPer; ++u) {
            code[u] = v[u] < 0 ? -1 : v[u] >> 24;
            if (v[u] >= 0) {
                const int j = v[u] & 0xFFFFFF;
                load_pos(xr, j, hj[u], lj[u]);
                pq[u] = pf4[(size_t)kr[u] * n + j];
                po[u] = pf4[(size_t)(k0 + WAYS * u + way) * n + ia];
            }
        }
        load_idx(k0 + CH);
#pragma unroll
        for (int u = 0; u < kAsmPer; ++u) {
            const int s = WAYS * u + way;
            float rx = kNone;
            if (code[u] >= 0) {
                float ry, rz;
                pair_vector(code[u], hi, li, hj[u], lj[u], box, rx, ry, rz);
                const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
                if (d2 < rc2max) {
                    s_t[1][s][at] = ry;
                    s_t[2][s][at] = rz;
                    s_t[3][s][at] = pq[u].x;
                    s_t[4][s][at] = pq[u].y;
                    s_t[5][s][at] = pq[u].z;
                    s_t[6][s][at] = po[u].x - pq[u].x;
                    s_t[7][s][at] = po[u].y - pq[u].y;
                    s_t[8][s][at] = po[u].z - pq[u].z;
                } else {
                    rx = kNone;
                }
            }
            s_t[0][s][at] = rx;
        }
        __syncthreads();
        const int smax = min(CH, kmax - k0);
        for (int s = 0; s < smax; ++s) {
            const float rx = s_t[0][s][at];
            if (rx < 0.5f * kNone) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const int o = way * NC + c;  // F: 0..2, W^{ab}: 3 + 3 a + b
                    if (o < 3)
                        acc[c] += s_t[6 + o][s][at];
                    else if (o < 12)
                        acc[c] = fmaf(s_t[o / 3 - 1][s][at], s_t[3 + o % 3][s][at], acc[c]);
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
        if (way * NC + c < 12) s_sum[way * NC + c][at] = acc[c];
    __syncthreads();

    // four rows of threads per atom finish: row 0 the force (and the kick),
    // row 1 + a the virial components (a, .) and J^a
    const int row = threadIdx.x / AT;
    double t[4] = {0.0, 0.0, 0.0, 0.0};  // row 0: E_kin; row 1 + a: W^{a.}, J^a
    float x[3] = {0.f, 0.f, 0.f};
    if (row < 4 && active) {
#pragma unroll
        for (int c = 0; c < 3; ++c) x[c] = s_sum[3 * row + c][at];
        if (row == 0) {
            if (!(isfinite(x[0]) && isfinite(x[1]) && isfinite(x[2]))) atomicOr(err, kErrNonFinite);
            if (force)
#pragma unroll
                for (int c = 0; c < 3; ++c) force[(size_t)c * n + i] = x[c];
            if constexpr (MD) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    w[c] += hdtm * (double)x[c];
                    vel[(size_t)c * n + i] = w[c];
                    s_v[c][at] = (float)w[c];
                }
                t[0] = kef * (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
            }
        } else {
            if (virial_atom)
#pragma unroll
                for (int c = 0; c < 3; ++c) virial_atom[(size_t)(3 * (row - 1) + c) * n + i] = x[c];
#pragma unroll
            for (int c = 0; c < 3; ++c) t[c] = (double)x[c];
        }
    }
    if constexpr (MD) {
        __syncthreads();
        // J^a = sum_b W^{ab} v^b, FP32 products accumulated in FP64
        if (row >= 1 && row < 4 && active)
            t[3] = (double)(x[0] * s_v[0][at]) + (double)(x[1] * s_v[1][at]) + (double)(x[2] * s_v[2][at]);
    }
    if (row >= 4) return;  // whole warps
    // sums over the AT lanes of a row: two butterfly levels that halve the
    // components (lane bits AT/2 and AT/4), then whole sums; lane bits
    // (AT/2, AT/4) give the component that a lane ends with
    const bool b1 = (at & (AT / 2)) != 0, b0 = (at & (AT / 4)) != 0;
    const double u0 = (b1 ? t[2] : t[0]) + __shfl_xor_sync(0xffffffffu, b1 ? t[0] : t[2], AT / 2);
    const double u1 = (b1 ? t[3] : t[1]) + __shfl_xor_sync(0xffffffffu, b1 ? t[1] : t[3], AT / 2);
    double sum = (b0 ? u1 : u0) + __shfl_xor_sync(0xffffffffu, b0 ? u0 : u1, AT / 4);
#pragma unroll
    for (int o = AT / 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const int c = 2 * (b1 ? 1 : 0) + (b0 ? 1 : 0);
    if (at % (AT / 4) == 0) {
        const int k = row == 0 ? (MD && c == 0 ? 9 : -1) : c < 3 ? 3 * (row - 1) + c : MD ? 9 + row : -1;
        if (k >= 0) partials[(size_t)k * gridDim.x + block] = sum;
    }
}

// The same with one thread per atom: no tile and no barriers, so it wins once
// the atoms fill the GPU and their lists are short (asm_by_atoms below).
template <bool MD>
__global__ void __launch_bounds__(kAsmThreads) k_assemble_atoms(int n, int m_cap, float rc2max, const int* count,
                                                          const int* nbr, const int* rev,
                                                          const float* xr,
                                                          Box box, const float* pf,
                                                          float* force, float* virial_atom,
                                                          double* partials, unsigned* err,
                                                          double* vel, double hdtm, double kef,
                                                          const unsigned* mask)
{
    constexpr int K = MD ? 13 : 9;
    const int block = block_after();
    const int i = block * blockDim.x + threadIdx.x;
    double acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    if (i < n) {
        // the list is read straight from global memory: staging it in shared
        // memory (as the site pass does) cost this pass occupancy and time
        const SlotTable T{nbr, n, i};
        float F[3], W[9];
        assemble_atom(i, n, m_cap, rc2max, count, T, rev, xr, box, pf, F, W, mask);
        double v[3];  // loaded ahead of the stores
        if constexpr (MD)
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] = vel[(size_t)c * n + i];
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
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[c] += hdtm * (double)F[c];
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
    block_sum_store<K>(acc, partials + block, gridDim.x);
}

// One total per block, the totals of `a` and then those of `b`: several SMs
// share the FP64 adds, which are slow on this part.
constexpr int kSumThreads = 512;
__global__ void __launch_bounds__(kSumThreads) k_sum(SumSet a, SumSet b)
{
    const int block = block_after();
    const bool first = block < a.ncomp;
    const SumSet s = first ? a : b;
    const int w = first ? block : block - a.ncomp;
    if (!s.out) return;
    const double t = sum_partials<kSumThreads>(s.src + (size_t)w * s.cstride, s.nb, s.bstride);
    if (threadIdx.x == 0) s.out[w] = t;
}

inline int blocks_for(int n, int t) { return (n + t - 1) / t; }

template <class D, int AT>
int launch_site(const ForceArgs& a, NeighborList& nl, int n, double* e_atom, double* e_partials, unsigned* d_err,
                cudaStream_t st, int& nblocks, bool after)
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
    nblocks = blocks_for(n, AT);
    const size_t smem = site_block_smem<D, AT>(n_par, a.n_neu);
    constexpr int kWide = (384 / SiteSplit<AT>::WAYS + 31) / 32;  // words that hold any capacity
    auto kern = nl.m_cap <= 32 * SiteSplit<AT>::WAYS ? k_site<D, AT, 1> : k_site<D, AT, kWide>;
    // only large networks of the split model need more than the default: an
    // attribute call costs as much host time as a launch.  The limit is the
    // kernel's, whatever model is launched: always that of the largest network
    if (smem > kDefaultShared) {
        constexpr int kMost = (int)site_block_smem<D, AT>((D::Ndes + 2) * kMaxNeu + 1, kMaxNeu);
        const int rc = cuda_fail(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost),
                                 "site kernel shared memory");
        if (rc) return rc;
    }
    nl.mask_set = nl.m_cap <= kMaskSlots && nl.mask != nullptr;
    return cuda_fail(launch_after(after, kern, nblocks, kSiteThreads, smem, st, n, nl.m_cap, nl.count,
                                  nl.nbr, nl.xr, a.box, a.z, n_par, P, nl.pf, e_atom, e_partials, d_err,
                                  nl.mask_set ? nl.mask : nullptr), "site kernel");
}

}  // namespace

int launch_site_partial_forces(const ForceArgs& a, NeighborList& nl, int n, double* e_atom, double* e_partials,
                               unsigned* d_err, cudaStream_t st, int& nblocks, bool after)
{
    const int at = site_atoms_per_block(n);
    if (a.nr == DescPbTe::NR && a.na == DescPbTe::NA)
        return (at == 8 ? launch_site<DescPbTe, 8> : at == 16 ? launch_site<DescPbTe, 16> : launch_site<DescPbTe, 32>)(
            a, nl, n, e_atom, e_partials, d_err, st, nblocks, after);
    if (a.nr != DescSi::NR || a.na != DescSi::NA) {
        set_error("no site kernel for %d radial and %d angular orders", a.nr, a.na);
        return NEP_ERR_UNSUPPORTED;
    }
    return (at == 8 ? launch_site<DescSi, 8> : at == 16 ? launch_site<DescSi, 16> : launch_site<DescSi, 32>)(
        a, nl, n, e_atom, e_partials, d_err, st, nblocks, after);
}

// One thread per atom in the assembly, by the number of atoms and the mean
// number of slots (from the density): from about 60,000 atoms with lists of
// ~26 slots (28 against 29 us at 64,000, 39.6 against 51.8 at 125,000), while
// the 64-slot lists of the split model stay faster tiled (64,000 atoms: 72
// against 97 us).
static bool asm_by_atoms(int n, double rc, const Box& b)
{
    const double slots = 4.18879 * rc * rc * rc * n / (b.L[0] * b.L[1] * b.L[2]);
    return n > 60000 && slots < 45.0;
}

int launch_assemble(const AssembleArgs& a, NeighborList& nl, int n, float* force, float* virial_atom,
                    double* partials, unsigned* d_err, cudaStream_t st, int& nblocks, int& ncomp)
{
    const bool atoms = asm_by_atoms(n, a.rc_max, a.box);
    const int at = atoms ? kAsmThreads : site_atoms_per_block(n);
    nblocks = blocks_for(n, at);
    const float rc2 = a.rc_max * a.rc_max;
    const bool md = a.vel != nullptr;
    ncomp = md ? 13 : 9;
    auto kern = atoms      ? (md ? k_assemble_atoms<true> : k_assemble_atoms<false>)
                : at == 8  ? (md ? k_assemble<true, 8> : k_assemble<false, 8>)
                : at == 16 ? (md ? k_assemble<true, 16> : k_assemble<false, 16>)
                           : (md ? k_assemble<true, 32> : k_assemble<false, 32>);
    return cuda_fail(launch_after(true, kern, nblocks, kAsmThreads, 0, st, n, nl.m_cap, rc2,
                                  nl.count, nl.nbr, nl.rev, nl.xr, a.box, nl.pf, force, virial_atom, partials, d_err,
                                  md ? a.vel : nullptr, md ? a.half_dt_over_m : 0.0, md ? a.ke_factor : 0.0,
                                  nl.mask_set ? nl.mask : nullptr), "assemble kernel");
}

int launch_sum(const SumSet& a, const SumSet& b, cudaStream_t st, bool after)
{
    if (a.ncomp + b.ncomp == 0) return NEP_OK;
    return cuda_fail(launch_after(after, k_sum, a.ncomp + b.ncomp, kSumThreads, 0, st, a, b), "sum kernel");
}

}  // namespace nep
