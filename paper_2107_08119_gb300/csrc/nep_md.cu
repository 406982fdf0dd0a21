// nep_md.cu -- NVE velocity-Verlet molecular dynamics on the NEP force path.
//
// One step is a fixed sequence of kernels on the caller's stream, with no
// host round trip:
//   k_kick_drift   v += dt/2 F/m; x += dt v (FP64); FP32 hi/lo split of x;
//                  largest squared displacement since the last list build;
//                  its last block sets the gate = (max displacement >
//                  skin/2)
//   list build     wrap, bin, Verlet list, reverse index (gated: the kernels
//                  return at once when the gate is zero)
//   k_site         site energies and partial forces
//   k_assemble     forces, second half kick, E_kin, virial and heat current
//                  J = sum_i W_i . v_i (Eq. 7), per-block FP64 sums
//   k_md_finish    block sums in a fixed order (one block per sum), thermo
//                  row and J of this step, Berendsen factor; where another
//                  step of the same graph follows, its k_kick_drift does the
//                  sums instead, or with a thermostat the scaling
// Optional extensions (nep_md_set_thermostat, nep_md_set_hnemd):
//   HNEMD          the assembly writes F and W_i; after the virial sum,
//                  k_hnemd_kick adds F_i^ext = F_e . W_i - F_e . W / N
//                  (Sec. II.B; the mean removed so the momentum is kept) and
//                  does the second half kick, E_kin and J
//   thermostat     Berendsen: after J, v *= lambda with lambda^2 = 1 +
//                  (dt/tau)(T0/T - 1), T from E_kin with 3N - 3 degrees of
//                  freedom (k_scale_v)
//   spectral heat current (nep_md_set_shc): on every `every`-th step the
//                  assembly writes W_i into a ring of n_lags samples and,
//                  next to J, k_shc_corr / k_shc_reduce add
//                  sum_i W_i(s - tau) . v_i(s) to K[tau] for every lag tau
//                  already in the ring (Sec. II.B)
#include <algorithm>
#include <cmath>
#include <new>

#include "nep_internal.cuh"

// 1 amu A^2 / fs^2 expressed in eV (CODATA 2018 atomic mass constant and
// elementary charge).
static constexpr double kAmuA2Fs2InEv = 1.66053906660e-27 * 1.0e-20 / 1.0e-30 / 1.602176634e-19;
// Boltzmann constant in eV/K (CODATA 2018)
static constexpr double kBoltzmannEv = 8.617333262e-5;
// reduced Planck constant in eV fs (CODATA 2018)
static constexpr double kHbarEvFs = 0.6582119569;
static constexpr double kPi = 3.14159265358979323846;
// 1 eV / (A fs K) in W / (m K): 1.602176634e-19 J / (1e-10 m 1e-15 s K)
static constexpr double kEvPerAFsK_WPerMK = 1.602176634e6;

namespace nep {
namespace {

// Control words on the device.  Where a call's rows go and its thermostat's
// numbers stand here and not in the launches, so that the step graphs outlive
// them: a block of five steps of 512 atoms with rows of its own took 355 us with
// new graphs, the same block again 178.
struct StepCtl {
    unsigned gate;            // 1: the list is rebuilt in this step
    unsigned step;            // steps of the call so far
    unsigned long long kick;  // blocks of k_kick_drift (see there)
    double *thermo, *heat;    // the call's rows, or NULL
    double t0, tau;           // thermostat
};

// The start of a call; `init`: of the first one on a new state too
__global__ void k_md_begin(StepCtl* ctl, int init, double* thermo, double* heat, double t0, double tau)
{
    if (init) {
        ctl->gate = 0u;
        ctl->kick = 0ull;
    }
    ctl->step = 0u;
    ctl->thermo = thermo;
    ctl->heat = heat;
    ctl->t0 = t0;
    ctl->tau = tau;
}

// A step's sums, one block each: block 0 the site-energy block partials, block
// 1 + c component c of the other block partials (each thread a fixed stride of
// the partials in order, then a fixed tree: deterministic).  Several SMs share
// the FP64 adds (slow on this part).  No sum needs another one, so each block
// writes its own place of the thermo row or of J, and that of E_kin the
// Berendsen factor; a last block that collected all sums cost a fence, an atomic
// and a second round of loads.  This and the one atomic of k_kick_drift: step of
// 4,096 atoms 45.4 -> 41.9 us, driven step of 13,824 80.1 -> 75.7.
// Without a thermostat nothing in the next step's kick needs them, so within a
// graph they are extra blocks of that kernel, not a launch of their own: step of
// 4,096 atoms 40.1 -> 37.7 us, of 125,000 294.2 -> 288.9.
struct StepSums {
    int nsum = 0;  // blocks
    const double* part_e = nullptr;
    int nb_e = 0;
    const double* part_x = nullptr;
    int nb_x = 0, bstride_x = 0;
    size_t cstride_x = 0;
    int off_x = 0;
    double* red = nullptr;
    const StepCtl* ctl = nullptr;
    int row = 0;  // row of the step, from the step counter
    bool thermostat = false;
    double dt = 0.0, dof_kb = 0.0;
};

template <int THREADS>
__device__ __forceinline__ void step_sum(const StepSums& S, int w)
{
    // sums: 0 E_pot, 1..9 W (row-major), 10 E_kin, 11..13 J; red: [1..9] W with
    // HNEMD (summed before the kick), [14] lambda
    double t = sum_partials<THREADS>(w == 0 ? S.part_e : S.part_x + (w - 1) * S.cstride_x, w == 0 ? S.nb_e : S.nb_x,
                                     w == 0 ? 1 : S.bstride_x);
    if (threadIdx.x != 0) return;
    const int k = w == 0 ? 0 : S.off_x + w - 1;
    const StepCtl& C = *S.ctl;  // (read ahead of the sum: 0.6 us more per step of 125,000 atoms)
    const size_t s = (size_t)((int)C.step + S.row);
    if (k == 10 && S.thermostat) {
        const double T = 2.0 * t / S.dof_kb;
        const double lam = T > 0.0 ? sqrt(1.0 + S.dt / C.tau * (C.t0 / T - 1.0)) : 1.0;
        S.red[14] = lam;
        t *= lam * lam;
    }
    if (C.thermo) {
        double* row = C.thermo + s * NEP_THERMO_COLS;  // E_pot, E_kin, W xx yy zz xy yz zx
        const int col = k == 0 ? 0 : k == 10 ? 1 : k == 1 ? 2 : k == 5 ? 3 : k == 9 ? 4 : k == 2 ? 5 : k == 6 ? 6
                      : k == 7 ? 7 : -1;
        if (col >= 0) row[col] = t;
        if (k == 0 && S.off_x == 10) {
            row[2] = S.red[1];
            row[3] = S.red[5];
            row[4] = S.red[9];
            row[5] = S.red[2];
            row[6] = S.red[6];
            row[7] = S.red[7];
        }
    }
    if (C.heat && k >= 11) C.heat[s * 3 + k - 11] = t;
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_md_finish(StepSums S)
{
    step_sum<THREADS>(S, block_after());
}

// The rebuild decision: gate = `far`, an atom beyond the threshold since the
// last build; `count` steps are counted.
// use_cond: the step runs from a CUDA graph whose list rebuild sits behind the
// conditional node `cond`, which this sets.
__device__ void decide(StepCtl* ctl, bool far, int count, unsigned long long* rebuilds,
                       cudaGraphConditionalHandle cond, int use_cond)
{
    ctl->gate = far ? 1u : 0u;
    if (count) ctl->step += (unsigned)count;
    if (far) *rebuilds += 1ull;
    if (use_cond) cudaGraphSetConditional(cond, far ? 1u : 0u);
}

// The first S.nsum blocks add up the previous step; SCALE: its
// Berendsen factor red[14] is applied here, to velocities that were left unscaled
// (driven step of 13,824 atoms with a thermostat 71.8 -> 70.7 us).
template <int THREADS, bool SCALE>
__global__ void __launch_bounds__(THREADS) k_kick_drift(StepSums S, const double* red, int n, double* x, double* v,
                                                        const float* F, double hdtm, double dt,
                                                        float* xr, const double* x_ref,
                                                        StepCtl* ctl, float thresh2, int count,
                                                        unsigned long long* rebuilds,
                                                        cudaGraphConditionalHandle cond, int use_cond)
{
    const int block = block_after() - S.nsum;
    if (block < 0) {
        step_sum<THREADS>(S, blockIdx.x);
        return;
    }
    const int i = block * THREADS + threadIdx.x;
    double lam = 1.0;
    if constexpr (SCALE) lam = red[14];
    float d2 = 0.f;
    if (i < n) {
        // all loads ahead of the stores
        double dd = 0.0, xn[3], xo[3], vo[3], xf[3];
        float f[3];
        const float z = load_z(xr, i);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t o = (size_t)c * n + i;
            vo[c] = v[o];
            f[c] = F[o];
            xo[c] = x[o];
            xf[c] = x_ref[o];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t o = (size_t)c * n + i;
            const double vc = (SCALE ? __dmul_rn(vo[c], lam) : vo[c]) + hdtm * to_double(f[c]);
            const double xc = xo[c] + dt * vc;
            v[o] = vc;
            x[o] = xc;
            xn[c] = xc;
            const double d = xc - xf[c];
            dd += d * d;
        }
        store_pos(xr, i, xn, z);  // the species number stays
        d2 = (float)dd;
    }
    // the blocks with an atom beyond the threshold (high half) and those that
    // are done (low half) are counted by one atomic per block; the last one
    // clears the count and takes the rebuild decision from it
    const bool far = __syncthreads_or(d2 > thresh2);
    if (threadIdx.x != 0) return;
    const unsigned long long mine = far ? (1ull << 32) + 1 : 1ull;
    const unsigned long long all = atomicAdd(&ctl->kick, mine) + mine;
    if ((unsigned)all != gridDim.x - S.nsum) return;
    ctl->kick = 0ull;
    decide(ctl, (all >> 32) != 0, count, rebuilds, cond, use_cond);
}

// Second half kick with the HNEMD driving force, E_kin and J per block.
// W is the per-atom virial [9][n]; wtot the total virial (row-major).
__global__ void k_hnemd_kick(int n, float* F, const float* W, double* vel,
                             double fe0, double fe1, double fe2, const double* wtot, double inv_n,
                             double hdtm, double kef, double* partials, unsigned* err)
{
    const int i = block_after() * blockDim.x + threadIdx.x;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const double fe[3] = {fe0, fe1, fe2};
    __shared__ double s_fm[3];
    if (threadIdx.x < 3) {
        double fm = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) fm += fe[a] * wtot[3 * a + threadIdx.x];
        s_fm[threadIdx.x] = fm;
    }
    __syncthreads();
    if (i < n) {
        float w[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) w[c] = W[(size_t)c * n + i];
        double v[3];
        float f[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {  // loaded ahead of the stores
            f[b] = F[(size_t)b * n + i];
            v[b] = vel[(size_t)b * n + i];
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double fm = s_fm[b];
            double fx = 0.0;
#pragma unroll
            for (int a = 0; a < 3; ++a) fx += fe[a] * (double)w[3 * a + b];
            const float ft = (float)((double)f[b] + fx - fm * inv_n);
            F[(size_t)b * n + i] = ft;
            v[b] += hdtm * (double)ft;
            vel[(size_t)b * n + i] = v[b];
        }
        if (!isfinite(v[0] + v[1] + v[2])) atomicOr(err, kErrNonFinite);
        acc[0] = kef * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            acc[1 + a] = (double)(w[3 * a] * (float)v[0]) + (double)(w[3 * a + 1] * (float)v[1]) +
                         (double)(w[3 * a + 2] * (float)v[2]);
    }
    block_sum_store<4>(acc, partials + (size_t)blockIdx.x * 4);
}

// Virial-velocity correlation of one sample s (the ring holds W of the last
// `avail` samples, sample s in slot `slot0`): warp w of block (bx, by) takes
// lag tau = 8 bx + w and the atoms of chunk by, and writes
// sum_i (W_i(s - tau) . v_i(s))^a for its chunk, in a fixed order (lane
// strides, then a butterfly), to part[by][tau][a].  The products are FP32
// and the sums FP64, as in the heat current of the assembly.
constexpr int kShcChunk = 4096;
constexpr int kShcLagsPerBlock = 8;

__global__ void __launch_bounds__(32 * kShcLagsPerBlock) k_shc_corr(int n, int n_lags, int avail, int slot0,
                                                                      const float* __restrict__ ring,
                                                                      const double* __restrict__ vel,
                                                                      double* __restrict__ part)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tau = blockIdx.x * kShcLagsPerBlock + warp;
    if (tau >= avail) return;  // warp-uniform
    const int slot = (slot0 - tau + n_lags) % n_lags;
    const float* W = ring + (size_t)slot * 9 * n;
    const int c0 = blockIdx.y * kShcChunk, c1 = min(n, c0 + kShcChunk);
    double acc[3] = {0.0, 0.0, 0.0};
    for (int i = c0 + lane; i < c1; i += 32) {
        const float v0 = (float)vel[i], v1 = (float)vel[(size_t)n + i], v2 = (float)vel[2 * (size_t)n + i];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            acc[a] += (double)(W[(size_t)(3 * a) * n + i] * v0) + (double)(W[(size_t)(3 * a + 1) * n + i] * v1) +
                      (double)(W[(size_t)(3 * a + 2) * n + i] * v2);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], o);
    if (lane == 0)
#pragma unroll
        for (int a = 0; a < 3; ++a) part[((size_t)blockIdx.y * n_lags + tau) * 3 + a] = acc[a];
}

// sum[tau][a] += the chunk partials of this sample, chunks in order
__global__ void k_shc_reduce(int n_lags, int avail, int n_chunks, const double* __restrict__ part,
                             double* __restrict__ sum)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= avail * 3) return;
    const int tau = e / 3, a = e % 3;
    double t = 0.0;
    for (int c = 0; c < n_chunks; ++c) t += part[((size_t)c * n_lags + tau) * 3 + a];
    sum[(size_t)tau * 3 + a] += t;
}

// K[tau] = sum[tau] / (number of origins), 0 without any
__global__ void k_shc_average(int n_lags, long long n_samples, const double* __restrict__ sum, double* __restrict__ K)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_lags * 3) return;
    const long long origins = n_samples - e / 3;
    K[e] = origins > 0 ? sum[e] / (double)origins : 0.0;
}

// out[k][a] = scale * 2 * trapezoid of K[tau][a] cos(omega_k tau dt) over the
// lags (K even in t), optionally Hann-windowed (Sec. II.B transform)
// omega_k = omega_per_x * x[k] (1 when x holds the angular frequencies).
__global__ void k_shc_spectrum(int n_lags, const double* __restrict__ K, double dt, int n_omega,
                               const double* __restrict__ omega, double omega_per_x, double scale, int window,
                               double* __restrict__ out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_omega * 3) return;
    const int k = e / 3, a = e % 3;
    const double w0 = omega_per_x * omega[k];
    double s = 0.0;
    for (int t = 0; t < n_lags; ++t) {
        double w = (t == 0 || t == n_lags - 1) ? 0.5 : 1.0;
        if (window && n_lags > 1) w *= 0.5 * (1.0 + cospi((double)t / (n_lags - 1)));
        s += w * K[(size_t)t * 3 + a] * cos(w0 * t * dt);
    }
    out[e] = scale * 2.0 * dt * s;
}

// spec[k][.] *= (h / sinh h)^2 with h = x/2, x = x_per_omega omega[k]: the
// quantum-correction factor x^2 e^x / (e^x - 1)^2 of Sec. IV.C in a form with
// no cancellation at small x (1 - h^2/3 below h = 1e-4, where FP64 sinh(h)/h
// has nothing left to resolve) and none at large x (sinh overflows to inf and
// the factor to 0).
__global__ void k_shc_quantum(int n_omega, const double* __restrict__ omega, double x_per_omega,
                              double* __restrict__ spec)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_omega) return;
    const double h = fabs(0.5 * (x_per_omega * omega[k]));
    double f;
    if (h < 1e-4) {
        f = 1.0 - h * h / 3.0;
    } else {
        const double r = h / sinh(h);
        f = r * r;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) spec[(size_t)k * 3 + a] *= f;
}

// Running mean of J times scale: thread t of one block owns a contiguous
// segment of steps; the segment sums are prefixed in order by thread 0, and
// each thread then walks its segment again from its offset.
constexpr int kKappaThreads = 256;
__global__ void __launch_bounds__(kKappaThreads) k_hnemd_kappa(int n, const double* __restrict__ J, double scale,
                                                               double* __restrict__ out)
{
    __shared__ double seg[kKappaThreads][3];
    const int t = threadIdx.x;
    const int per = (n + kKappaThreads - 1) / kKappaThreads;
    const int a = min(n, t * per), b = min(n, a + per);
    double s[3] = {0.0, 0.0, 0.0};
    for (int i = a; i < b; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) s[c] += J[(size_t)i * 3 + c];
#pragma unroll
    for (int c = 0; c < 3; ++c) seg[t][c] = s[c];
    __syncthreads();
    if (t == 0) {
        double run[3] = {0.0, 0.0, 0.0};
        for (int u = 0; u < kKappaThreads; ++u)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double x = seg[u][c];
                seg[u][c] = run[c];
                run[c] += x;
            }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) s[c] = seg[t][c];
    for (int i = a; i < b; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            s[c] += J[(size_t)i * 3 + c];
            out[(size_t)i * 3 + c] = scale * s[c] / (double)(i + 1);
        }
}

// v *= lambda (the Berendsen factor k_md_finish left in red[14])
__global__ void k_scale_v(int n, double* vel, const double* red)
{
    const int i = block_after() * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double lam = red[14];
    double v[3];  // loaded ahead of the stores
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = vel[(size_t)c * n + i];
#pragma unroll
    for (int c = 0; c < 3; ++c) vel[(size_t)c * n + i] = v[c] * lam;
}

inline int blocks_for(int n, int t) { return (n + t - 1) / t; }

}  // namespace
}  // namespace nep

using namespace nep;

// Steps per graph launch where a call has that many left: the gap between two
// graphs costs more than the one between their kernels (4,096 atoms 49.4 -> 46.1
// us per step; 10 steps per graph 45.5).
constexpr int kGraphSteps = 5;

// Steps with one capture key at which the graph of kGraphSteps steps pays for its
// capture: about 200 us of the host against 75 for one step (in part behind the
// five single steps that run meanwhile), and 4 us saved per step.  Calls with a new
// time step each, graphs of one step only -> of five whenever they fit: 512 atoms,
// 5 steps 256 -> 308 us, 10 steps 455 -> 480, 20 steps 844 -> 815; driven 13,824
// atoms 439 -> 500, 847 -> 896, 1615 -> 1647, 40 steps 3237 -> 3187.  In a large box
// five steps outlast the capture, which then is nearly free: 125,000 atoms, 5 steps
// 2020 -> 2080 us, 10 steps 4335 -> 4355, 15 steps 6710 -> 6690, and 20 steps
// that follow a call of 5 steps 5240 -> 5192.
constexpr int graph_pays(int n) { return n < 60000 ? 20 : kGraphSteps; }

// Atoms from which the starting forces of a new state hide the capture of that
// graph.  20 steps of a new state, the graph behind five single steps -> at once:
// 13,824 atoms 1213 -> 1260 us, 21,952 1535 -> 1550, 27,000 1828 -> 1821, 32,768 1966
// -> 1938, 39,304 2384 -> 2339, 125,000 5810 -> 5763.
constexpr int kHiddenCapture = 30000;

// Threads per block of the per-atom step kernels: two FP64 lanes per SM and
// clock bound them, so up to one block of 256 per SM the atoms go to more SMs
// (driven step of 13,824 atoms 73.9 -> 71.4 us, step of 4,096 39.8 -> 39.4; 128
// threads the same).  The partial sums of k_hnemd_kick, four per block, need the
// room that 64 leaves: 14 of 16 words per block of the site pass, two more here.
inline int step_threads(int n) { return n <= 152 * 256 ? 64 : 256; }

struct nep_md {
    nep_model* m = nullptr;
    int n = 0;
    Box box;
    double mass = 0.0;
    float r_list = 0.f;
    float skin = 0.f;
    Workspace ws;
    double* x_ref = nullptr;
    StepCtl* ctl = nullptr;
    // what a call set in ctl; as created, tau is one that no thermostat has
    struct CtlValues {
        double *thermo = nullptr, *heat = nullptr;
        double t0 = 0.0, tau = NAN;
        bool operator==(const CtlValues& o) const
        {
            return thermo == o.thermo && heat == o.heat && t0 == o.t0 && tau == o.tau;
        }
    } ctl_values;
    bool captured = false;  // a call ran under stream capture
    unsigned long long* rebuilds = nullptr;
    double* red = nullptr;
    bool need_init = true;
    // Berendsen thermostat (tau <= 0: off) and HNEMD driving force
    double t0 = 0.0, tau = 0.0;
    double fe[3] = {0.0, 0.0, 0.0};
    bool drive = false;
    bool plain = false;       // force pass by the plain FP32 comparator (nep_md_set_force_form)
    float* w_atom = nullptr;  // [9][n] per-atom virials (HNEMD only)
    // spectral heat current: ring of per-atom virials, lag sums, chunk partials
    int shc_lags = 0, shc_every = 1;
    long long shc_step = 0, shc_samples = 0;
    float* shc_ring = nullptr;   // [n_lags][9][n]
    double* shc_sum = nullptr;   // [n_lags][3]
    double* shc_part = nullptr;  // [chunks][n_lags][3]
    // steps captured as CUDA graphs (the list rebuild behind conditional nodes),
    // kept while everything they bake in is unchanged
    cudaStream_t gcap = nullptr, gcap2 = nullptr;
    cudaGraphExec_t gexec[2] = {nullptr, nullptr};  // one step, kGraphSteps steps
    int gsteps = 0;                                 // steps run with this key, up to graph_pays
    struct GraphKey {
        const double *pos, *vel;
        double dt, fe[3];
        bool thermostat, drive;
        const float* zatom;
        bool plain;
        bool operator==(const GraphKey& o) const
        {
            return pos == o.pos && vel == o.vel && dt == o.dt && fe[0] == o.fe[0] && fe[1] == o.fe[1] &&
                   fe[2] == o.fe[2] && thermostat == o.thermostat && drive == o.drive && zatom == o.zatom && plain == o.plain;
        }
    } gkey{};
};

namespace {
// the model's species numbers when they were set for this many atoms
const float* md_zatom(const nep_md* md)
{
    return md->m->zatom && md->m->zatom_n == md->n ? md->m->zatom : nullptr;
}

void free_shc(nep_md* md)
{
    if (md->shc_ring) cudaFree(md->shc_ring);
    if (md->shc_sum) cudaFree(md->shc_sum);
    if (md->shc_part) cudaFree(md->shc_part);
    md->shc_ring = nullptr;
    md->shc_sum = nullptr;
    md->shc_part = nullptr;
    md->shc_lags = 0;
    md->shc_step = md->shc_samples = 0;
}
}  // namespace

extern "C" {

int nep_md_create(nep_model* m, int n, const double* box9, double mass, nep_md** out)
{
    if (!m || !out || n < 1 || n > kMaxAtoms || !(mass > 0.0)) {
        set_error("nep_md_create: bad arguments");
        return NEP_ERR_ARG;
    }
    *out = nullptr;
    const double rmax = (m->hp.rc_R > m->hp.rc_A ? m->hp.rc_R : m->hp.rc_A) + m->hp.skin;
    nep_md* md = new (std::nothrow) nep_md();
    if (!md) {
        set_error("nep_md_create: host allocation failed");
        return NEP_ERR_OOM;
    }
    int rc = setup_box(box9, rmax, md->box);
    if (rc) {
        delete md;
        return rc;
    }
    md->m = m;
    md->n = n;
    md->mass = mass;
    md->r_list = (float)rmax;
    md->skin = (float)m->hp.skin;
    const int ncell = md->box.nc[0] * md->box.nc[1] * md->box.nc[2];
    const int nb = site_blocks(n);
    if ((rc = ensure_workspace(md->ws, n, m->hp.max_neighbors, ncell, nb))) {
        nep_md_destroy(md);
        return rc;
    }
    cudaError_t e = cudaMalloc((void**)&md->x_ref, sizeof(double) * 3 * (size_t)n);
    if (e == cudaSuccess) e = cudaMalloc((void**)&md->ctl, sizeof(StepCtl));
    if (e == cudaSuccess) e = cudaMalloc((void**)&md->rebuilds, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMalloc((void**)&md->red, sizeof(double) * 32);
    if (e == cudaSuccess) e = cudaMemset(md->ctl, 0, sizeof(StepCtl));
    if (e == cudaSuccess) e = cudaMemset(md->rebuilds, 0, sizeof(unsigned long long));
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("nep_md_create: %s", cudaGetErrorString(e));
        nep_md_destroy(md);
        return NEP_ERR_OOM;
    }
    *out = md;
    return NEP_OK;
}

int nep_md_destroy(nep_md* md)
{
    if (!md) return NEP_OK;
    cudaDeviceSynchronize();
    free_workspace(md->ws);
    if (md->x_ref) cudaFree(md->x_ref);
    if (md->ctl) cudaFree(md->ctl);
    if (md->rebuilds) cudaFree(md->rebuilds);
    if (md->red) cudaFree(md->red);
    if (md->w_atom) cudaFree(md->w_atom);
    free_shc(md);
    for (auto e : md->gexec)
        if (e) cudaGraphExecDestroy(e);
    if (md->gcap) cudaStreamDestroy(md->gcap);
    if (md->gcap2) cudaStreamDestroy(md->gcap2);
    delete md;
    return NEP_OK;
}

int nep_md_set_thermostat(nep_md* md, double t0, double tau)
{
    if (!md || (tau > 0.0 && !(t0 >= 0.0))) {
        set_error("nep_md_set_thermostat: NULL handle or negative target temperature");
        return NEP_ERR_ARG;
    }
    md->t0 = t0;
    md->tau = tau > 0.0 ? tau : 0.0;
    return NEP_OK;
}

int nep_md_set_force_form(nep_md* md, int form)
{
    if (!md || (form != NEP_FORCE_OPTIMISED && form != NEP_FORCE_PLAIN_FP32)) {
        set_error("nep_md_set_force_form: NULL handle or unknown form %d", form);
        return NEP_ERR_ARG;
    }
    if (form == NEP_FORCE_PLAIN_FP32 && !sizes_default(md->m->hp)) {
        set_error("nep_md_set_force_form: the plain comparator has kernels for the 32-descriptor model only");
        return NEP_ERR_UNSUPPORTED;
    }
    if (form == NEP_FORCE_PLAIN_FP32 && md->ws.plain_cap < md->n) {
        if (md->ws.plain) cudaFree(md->ws.plain);
        md->ws.plain = nullptr;
        md->ws.plain_cap = 0;
        const cudaError_t e = cudaMalloc((void**)&md->ws.plain, sizeof(float) * 2 * kNdes * (size_t)md->n);
        if (e != cudaSuccess) {
            cudaGetLastError();
            set_error("nep_md_set_force_form: %s", cudaGetErrorString(e));
            return NEP_ERR_OOM;
        }
        md->ws.plain_cap = md->n;
    }
    md->plain = form == NEP_FORCE_PLAIN_FP32;
    md->need_init = true;  // the next step recomputes the starting forces with the selected form
    return NEP_OK;
}

int nep_md_set_hnemd(nep_md* md, const double* fe)
{
    if (!md) {
        set_error("nep_md_set_hnemd: NULL handle");
        return NEP_ERR_ARG;
    }
    for (int c = 0; c < 3; ++c) md->fe[c] = fe ? fe[c] : 0.0;
    md->drive = md->fe[0] != 0.0 || md->fe[1] != 0.0 || md->fe[2] != 0.0;
    if (md->drive && !md->w_atom) {
        cudaError_t e = cudaMalloc((void**)&md->w_atom, sizeof(float) * 9 * (size_t)md->n);
        if (e != cudaSuccess) {
            cudaGetLastError();
            md->w_atom = nullptr;
            md->drive = false;
            set_error("nep_md_set_hnemd: %s", cudaGetErrorString(e));
            return NEP_ERR_OOM;
        }
    }
    md->need_init = true;  // the next step recomputes the starting forces with (or without) the drive
    return NEP_OK;
}

int nep_md_set_shc(nep_md* md, int n_lags, int every)
{
    if (!md || n_lags < 0 || n_lags > 100000 || (n_lags > 0 && every < 1)) {
        set_error("nep_md_set_shc: bad arguments (0 <= n_lags <= 100000, every >= 1)");
        return NEP_ERR_ARG;
    }
    cudaDeviceSynchronize();
    free_shc(md);
    if (n_lags == 0) return NEP_OK;
    const int chunks = (md->n + kShcChunk - 1) / kShcChunk;
    cudaError_t e = cudaMalloc((void**)&md->shc_ring, sizeof(float) * 9 * (size_t)md->n * n_lags);
    if (e == cudaSuccess) e = cudaMalloc((void**)&md->shc_sum, sizeof(double) * 3 * (size_t)n_lags);
    if (e == cudaSuccess) e = cudaMalloc((void**)&md->shc_part, sizeof(double) * 3 * (size_t)n_lags * chunks);
    if (e == cudaSuccess) e = cudaMemset(md->shc_sum, 0, sizeof(double) * 3 * (size_t)n_lags);
    if (e != cudaSuccess) {
        cudaGetLastError();
        free_shc(md);
        set_error("nep_md_set_shc: %s", cudaGetErrorString(e));
        return NEP_ERR_OOM;
    }
    md->shc_lags = n_lags;
    md->shc_every = every;
    return NEP_OK;
}

int nep_md_get_shc(nep_md* md, double* K, long long* n_samples, void* stream)
{
    if (!md || md->shc_lags == 0) {
        set_error("nep_md_get_shc: NULL handle or no correlation switched on (nep_md_set_shc)");
        return NEP_ERR_ARG;
    }
    if (n_samples) *n_samples = md->shc_samples;
    if (K) {
        const int e = md->shc_lags * 3;
        k_shc_average<<<(e + 255) / 256, 256, 0, (cudaStream_t)stream>>>(md->shc_lags, md->shc_samples, md->shc_sum,
                                                                        K);
        return cuda_fail(cudaGetLastError(), "nep_md_get_shc");
    }
    return NEP_OK;
}

int nep_shc_spectrum(const double* K, int n_lags, double dt_lag, int n_omega, const double* omega, double scale,
                     int window, double* out, void* stream)
{
    if (!K || !omega || !out || n_lags < 1 || n_omega < 1 || !(dt_lag > 0.0)) {
        set_error("nep_shc_spectrum: bad arguments");
        return NEP_ERR_ARG;
    }
    const int e = n_omega * 3;
    k_shc_spectrum<<<(e + 127) / 128, 128, 0, (cudaStream_t)stream>>>(n_lags, K, dt_lag, n_omega, omega, 1.0,
                                                                      scale, window ? 1 : 0, out);
    return cuda_fail(cudaGetLastError(), "nep_shc_spectrum");
}

int nep_shc_quantum(const double* omega, int n_omega, double x_per_omega, double* spec, void* stream)
{
    if (!omega || !spec || n_omega < 1 || !std::isfinite(x_per_omega)) {
        set_error("nep_shc_quantum: bad arguments");
        return NEP_ERR_ARG;
    }
    k_shc_quantum<<<(n_omega + 127) / 128, 128, 0, (cudaStream_t)stream>>>(n_omega, omega, x_per_omega, spec);
    return cuda_fail(cudaGetLastError(), "nep_shc_quantum");
}

int nep_hnemd_kappa(const double* J, int n, double scale, double* out, void* stream)
{
    if (!J || !out || n < 1) {
        set_error("nep_hnemd_kappa: bad arguments");
        return NEP_ERR_ARG;
    }
    k_hnemd_kappa<<<1, kKappaThreads, 0, (cudaStream_t)stream>>>(n, J, scale, out);
    return cuda_fail(cudaGetLastError(), "nep_hnemd_kappa");
}

int nep_hnemd_kappa_si(const double* J, int n, double temperature, double volume, double fe, double* out,
                       void* stream)
{
    if (!J || !out || n < 1 || !(temperature > 0.0) || !(volume > 0.0) || !(fe != 0.0) ||
        !std::isfinite(temperature * volume * fe)) {
        set_error("nep_hnemd_kappa_si: bad arguments (T > 0, V > 0, F_e != 0, all finite)");
        return NEP_ERR_ARG;
    }
    // <J> / (T V F_e) in eV / (A fs K) = kEvPerAFsK_WPerMK W / (m K)
    const double scale = kEvPerAFsK_WPerMK / (temperature * volume * fe);
    k_hnemd_kappa<<<1, kKappaThreads, 0, (cudaStream_t)stream>>>(n, J, scale, out);
    return cuda_fail(cudaGetLastError(), "nep_hnemd_kappa_si");
}

int nep_kappa_spectrum(const double* K, int n_lags, double dt_lag_fs, const double* nu_thz, int n_nu,
                       double temperature, double volume, double fe, int window, int quantum, double* out,
                       void* stream)
{
    if (!K || !nu_thz || !out || n_lags < 1 || n_nu < 1 || !(dt_lag_fs > 0.0) || !(temperature > 0.0) ||
        !(volume > 0.0) || !(fe != 0.0) || !std::isfinite(temperature * volume * fe * dt_lag_fs)) {
        set_error("nep_kappa_spectrum: bad arguments (lags, frequencies >= 1; dt, T, V > 0; F_e != 0)");
        return NEP_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    // omega = 2 pi nu, in rad/fs for nu in THz; kappa per THz of nu: the
    // W / (m K) of <J>/(T V F_e) times 1e-3 (the fs of dt over the ps of 1/nu)
    const double omega_per_nu = 2.0 * kPi * 1e-3;
    const double scale = 2.0 / (temperature * volume * fe) * kEvPerAFsK_WPerMK * 1e-3;
    const int e = n_nu * 3;
    k_shc_spectrum<<<(e + 127) / 128, 128, 0, st>>>(n_lags, K, dt_lag_fs, n_nu, nu_thz, omega_per_nu, scale,
                                                    window ? 1 : 0, out);
    // x = hbar omega / (k_B T) = (hbar / (k_B T)) (2 pi 1e-3) nu
    if (quantum)
        k_shc_quantum<<<(n_nu + 127) / 128, 128, 0, st>>>(
            n_nu, nu_thz, kHbarEvFs / (kBoltzmannEv * temperature) * omega_per_nu, out);
    return cuda_fail(cudaGetLastError(), "nep_kappa_spectrum");
}

int nep_md_invalidate(nep_md* md)
{
    if (!md) {
        set_error("nep_md_invalidate: NULL handle");
        return NEP_ERR_ARG;
    }
    md->need_init = true;
    return NEP_OK;
}

int nep_md_rebuild_count(nep_md* md, long long* count, void* stream)
{
    if (!md || !count) {
        set_error("nep_md_rebuild_count: NULL argument");
        return NEP_ERR_ARG;
    }
    int rc = cuda_fail(cudaStreamSynchronize((cudaStream_t)stream), "stream synchronise");
    if (rc) return rc;
    unsigned long long c = 0;
    rc = cuda_fail(cudaMemcpy(&c, md->rebuilds, sizeof(c), cudaMemcpyDeviceToHost), "read rebuild count");
    *count = (long long)c;
    return rc;
}

const float* nep_md_forces(const nep_md* md) { return md ? md->ws.force : nullptr; }

int nep_md_step(nep_md* md, double* pos, double* vel, int n_steps, double dt, double* thermo, double* heat,
                void* stream)
{
    if (!md || !pos || !vel || n_steps < 0 || !(dt > 0.0)) {
        set_error("nep_md_step: bad arguments");
        return NEP_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    nep_model* m = md->m;
    const int n = md->n;
    NeighborList& nl = md->ws.nl;
    const int nb = site_blocks(n);
    double* part_e = md->ws.partials;
    double* part_a = md->ws.partials + ((nb + 7) / 8) * 8;
    double* part_h = part_a + 13 * (size_t)nb;  // HNEMD kick partials
    const bool drive = md->drive;
    const int kt = step_threads(n), nbk = blocks_for(n, kt);
    const double kef = 0.5 * md->mass * kAmuA2Fs2InEv;
    ForceArgs fa{m->d_z, m->hp.n_neu, (float)m->hp.rc_R, (float)m->hp.rc_A, md->box};
    fa.nr = m->hp.n_max_R + 1;
    fa.na = m->hp.n_max_A + 1;
    fa.typed = md_zatom(md) != nullptr;
    if (m->zatom && !fa.typed) {
        set_error("nep_md_step: species were set for %d atoms, not %d", m->zatom_n, n);
        return NEP_ERR_ARG;
    }
    const double rmax = m->hp.rc_R > m->hp.rc_A ? m->hp.rc_R : m->hp.rc_A;
    const double conv = kAmuA2Fs2InEv;
    int rc;
    if (md->tau > 0.0 && n < 2) {
        set_error("nep_md_step: the thermostat needs at least two atoms");
        return NEP_ERR_ARG;
    }

    // site energies and partial forces: the optimised pass, or the plain FP32
    // comparator (literal Eq. 13, unfused) when selected
    Workspace& wsp = md->ws;
    auto site_pass = [&](cudaStream_t q, int& b1, bool after) {
        if (md->plain)
            return launch_plain_site(fa, nl, n, wsp.plain, wsp.plain + (size_t)kNdes * n, nullptr, part_e, m->d_err, q,
                                     b1);
        return launch_site_partial_forces(fa, nl, n, nullptr, part_e, m->d_err, q, b1, after);
    };
    const bool init = md->need_init;
    if (init) {
        // forces of the starting configuration (list built unconditionally)
        if ((rc = build_neighbor_list(nl, md->box, n, pos, md_zatom(md), true, md->x_ref, md->r_list, m->d_err, nullptr, st)))
            return rc;
        int b1 = 0, b2 = 0, c2 = 0;
        if ((rc = site_pass(st, b1, true))) return rc;
        AssembleArgs aa{};
        aa.rc_max = (float)rmax;
        aa.box = md->box;
        aa.vel = nullptr;
        if ((rc = launch_assemble(aa, nl, n, md->ws.force, drive ? md->w_atom : nullptr, part_a, m->d_err, st, b2,
                                  c2)))
            return rc;
        if (drive) {
            // the starting forces include the driving force (no kick: hdt/m = 0)
            if ((rc = launch_sum(SumSet{part_a, b2, 1, c2, (size_t)b2, md->red + 1}, SumSet{}, st))) return rc;
            k_hnemd_kick<<<nbk, kt, 0, st>>>(n, md->ws.force, md->w_atom, vel, md->fe[0], md->fe[1], md->fe[2],
                                              md->red + 1, 1.0 / n, 0.0, kef, part_h, m->d_err);
        }
    }
    // where the control words hold this call's rows and numbers already, the step
    // counter alone starts anew: a memset, as the kernel costs 2 us more (one-step
    // calls of 4,096 atoms).  Under capture nothing runs yet, and a replay sets them
    // unseen: from the first captured call on every call sets them all
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((rc = cuda_fail(cudaStreamIsCapturing(st, &cap), "capture status"))) return rc;
    md->captured = md->captured || cap != cudaStreamCaptureStatusNone;
    const nep_md::CtlValues cv{thermo, heat, md->t0, md->tau};
    if (init || md->captured || !(cv == md->ctl_values)) {
        md->ctl_values = {};
        k_md_begin<<<1, 1, 0, st>>>(md->ctl, init ? 1 : 0, thermo, heat, md->t0, md->tau);
        if ((rc = cuda_fail(cudaGetLastError(), "md step kernels"))) return rc;
        md->ctl_values = cv;
        md->need_init = false;
    } else if ((rc = cuda_fail(cudaMemsetAsync(&md->ctl->step, 0, sizeof(unsigned), st), "cudaMemsetAsync"))) {
        return rc;
    }

    const double hdtm = 0.5 * dt / (md->mass * conv);
    const float thresh = 0.5f * md->skin;
    const double dof_kb = (3.0 * n - 3.0) * kBoltzmannEv;

    // one step in three parts: kick-drift and the rebuild decision, the list
    // rebuild, then forces, second half kick and the step's sums
    // (count: steps to count; follows: another step comes before it in the stream,
    // whose sums are `prev` if it has left them)
    StepSums prev;
    const double* lam = nullptr;  // the previous step left its Berendsen factor to the next kick
    // threads per sum: with a thermostat always sums of their own, else as in the
    // kick, so that a step's sums have the same bits wherever a graph ends
    const int ft = md->tau > 0.0 ? 512 : kt;
    auto head = [&](cudaStream_t q, bool use_cond, cudaGraphConditionalHandle cond, int count, bool follows) {
        Profiler::Slot* pk = m->prof.begin(NEP_PROFILE_STEP, q);
        auto kick = kt == 64 ? (lam ? k_kick_drift<64, true> : k_kick_drift<64, false>)
                             : (lam ? k_kick_drift<256, true> : k_kick_drift<256, false>);
        launch_after(follows, kick, nbk + prev.nsum, kt, 0, q, prev, lam, n, pos,
                     vel, md->ws.force, hdtm, dt, nl.xr, md->x_ref, md->ctl, thresh * thresh, count, md->rebuilds, cond,
                     use_cond ? 1 : 0);
        prev.nsum = 0;
        lam = nullptr;
        m->prof.end(pk, q);
    };
    auto rebuild = [&](cudaStream_t q, const unsigned* g) {
        Profiler::Slot* pk = m->prof.begin(NEP_PROFILE_NEIGHBOR, q);
        const int r = build_neighbor_list(nl, md->box, n, pos, md_zatom(md), true, md->x_ref, md->r_list, m->d_err, g, q);
        m->prof.end(pk, q);
        return r;
    };
    // row: the step's row from the step counter; follows: another step comes in the same graph,
    // whose kick takes the sums or the Berendsen factor along
    auto tail = [&](cudaStream_t q, int row, bool follows) {
        int b1 = 0, b2 = 0, c2 = 0, r;
        // spectral heat current: this step's W_i goes to the ring when sampled
        const bool sample = md->shc_lags > 0 && md->shc_step % md->shc_every == 0;
        const int slot = sample ? (int)(md->shc_samples % md->shc_lags) : 0;
        float* w_out = sample ? md->shc_ring + (size_t)slot * 9 * n : (drive ? md->w_atom : nullptr);
        Profiler::Slot* ps = m->prof.begin(NEP_PROFILE_SITE, q);
        if ((r = site_pass(q, b1, false))) return r;  // after the conditional node
        m->prof.end(ps, q);
        AssembleArgs aa{};
        aa.rc_max = (float)rmax;
        aa.box = md->box;
        aa.vel = drive ? nullptr : vel;  // with HNEMD the kick waits for the total virial
        aa.half_dt_over_m = hdtm;
        aa.ke_factor = kef;
        aa.heat = heat != nullptr;
        ps = m->prof.begin(NEP_PROFILE_ASSEMBLE, q);
        if ((r = launch_assemble(aa, nl, n, md->ws.force, w_out, part_a, m->d_err, q, b2, c2))) return r;
        m->prof.end(ps, q);
        Profiler::Slot* pk = m->prof.begin(NEP_PROFILE_STEP, q);
        if (drive) {
            // the kick needs the total virial first
            if ((r = launch_sum(SumSet{part_a, b2, 1, c2, (size_t)b2, md->red + 1}, SumSet{}, q, true))) return r;
            launch_after(true, k_hnemd_kick, nbk, kt, 0, q, n, md->ws.force, w_out, vel, md->fe[0], md->fe[1],
                         md->fe[2], md->red + 1, 1.0 / n, hdtm, kef, part_h, m->d_err);
        }
        StepSums S{drive ? 5 : 1 + c2, part_e, b1, drive ? part_h : part_a, drive ? nbk : b2, drive ? 4 : 1,
                   drive ? 1 : (size_t)b2, drive ? 10 : 1, md->red, md->ctl, row, md->tau > 0.0, dt,
                   dof_kb};
        if (follows && md->tau <= 0.0)
            prev = S;
        else
            launch_after(true, ft == 64 ? k_md_finish<64> : ft == 256 ? k_md_finish<256> : k_md_finish<512>, S.nsum, ft,
                         0, q, S);
        if (sample) {  // v is that of J: after the second half kick, before the thermostat
            const int avail = (int)(md->shc_samples + 1 < md->shc_lags ? md->shc_samples + 1 : md->shc_lags);
            const int chunks = (n + kShcChunk - 1) / kShcChunk;
            k_shc_corr<<<dim3((avail + kShcLagsPerBlock - 1) / kShcLagsPerBlock, chunks), 32 * kShcLagsPerBlock, 0,
                         q>>>(n, md->shc_lags, avail, slot, md->shc_ring, vel, md->shc_part);
            k_shc_reduce<<<(avail * 3 + 127) / 128, 128, 0, q>>>(md->shc_lags, avail, chunks, md->shc_part,
                                                                  md->shc_sum);
            ++md->shc_samples;
        }
        if (md->shc_lags > 0) ++md->shc_step;
        if (md->tau > 0.0 && n > 1) {
            if (follows)
                lam = md->red;
            else
                launch_after(!sample, k_scale_v, nbk, kt, 0, q, n, vel, md->red);
        }
        m->prof.end(pk, q);
        return cuda_fail(cudaGetLastError(), "md step kernels");
    };

    // Without phase timing and without the per-step host logic of the
    // spectral heat current, the steps run from CUDA graphs of one and, where it
    // pays, of kGraphSteps steps, captured when first needed: the list rebuild is the
    // body of a conditional node that the last block of k_kick_drift switches,
    // so a step without a rebuild launches none of the list kernels.
    if (!m->prof.on && md->shc_lags == 0) {
        auto drop = [&]() {
            for (auto& e : md->gexec) {
                if (e) cudaGraphExecDestroy(e);
                e = nullptr;
            }
        };
        // `steps` steps as one graph
        auto capture = [&](int steps, cudaGraphExec_t* exec) {
            cudaGraph_t g = nullptr;
            int r = cuda_fail(cudaGraphCreate(&g, 0), "graph create");
            if (!r) r = cuda_fail(cudaStreamBeginCaptureToGraph(md->gcap, g, nullptr, nullptr, 0,
                                                                cudaStreamCaptureModeRelaxed), "begin capture");
            if (r) {
                if (g) cudaGraphDestroy(g);
                return r;
            }
            for (int s = 0; s < steps && !r; ++s) {
                cudaGraphConditionalHandle cond;
                r = cuda_fail(cudaGraphConditionalHandleCreate(&cond, g, 0, cudaGraphCondAssignDefault), "handle");
                if (r) break;
                head(md->gcap, true, cond, s == 0 ? steps : 0, s > 0);
                cudaStreamCaptureStatus cs;
                const cudaGraphNode_t* deps = nullptr;
                size_t nd = 0;
                r = cuda_fail(cudaStreamGetCaptureInfo(md->gcap, &cs, nullptr, nullptr, &deps, nullptr, &nd),
                              "capture info");
                cudaGraphNodeParams cp = {};
                cp.type = cudaGraphNodeTypeConditional;
                cp.conditional.handle = cond;
                cp.conditional.type = cudaGraphCondTypeIf;
                cp.conditional.size = 1;
                cudaGraphNode_t cnode = nullptr;
                if (!r) r = cuda_fail(cudaGraphAddNode(&cnode, g, deps, nullptr, nd, &cp), "conditional node");
                if (!r)
                    r = cuda_fail(cudaStreamUpdateCaptureDependencies(md->gcap, &cnode, nullptr, 1,
                                                                      cudaStreamSetCaptureDependencies),
                                  "capture dependencies");
                if (!r) {
                    cudaGraph_t body = cp.conditional.phGraph_out[0];
                    r = cuda_fail(cudaStreamBeginCaptureToGraph(md->gcap2, body, nullptr, nullptr, 0,
                                                                cudaStreamCaptureModeRelaxed), "begin body capture");
                    if (!r) {
                        r = rebuild(md->gcap2, nullptr);
                        cudaGraph_t b2 = nullptr;
                        const cudaError_t e = cudaStreamEndCapture(md->gcap2, &b2);
                        if (!r && e != cudaSuccess) r = cuda_fail(e, "end body capture");
                    }
                }
                if (!r) r = tail(md->gcap, s - steps, s < steps - 1);
            }
            cudaGraph_t g2 = nullptr;
            const cudaError_t e = cudaStreamEndCapture(md->gcap, &g2);
            if (!r && e != cudaSuccess) r = cuda_fail(e, "end capture");
            if (!r) r = cuda_fail(cudaGraphInstantiate(exec, g, 0), "instantiate step graph");
            cudaGraphDestroy(g);
            return r;
        };
        nep_md::GraphKey key{pos, vel, dt, {md->fe[0], md->fe[1], md->fe[2]}, md->tau > 0.0, drive, md_zatom(md),
                             md->plain};
        if (!(key == md->gkey) || !(md->gexec[0] || md->gexec[1])) {
            drop();
            if (!md->gcap && (rc = cuda_fail(cudaStreamCreateWithFlags(&md->gcap, cudaStreamNonBlocking), "stream")))
                return rc;
            if (!md->gcap2 && (rc = cuda_fail(cudaStreamCreateWithFlags(&md->gcap2, cudaStreamNonBlocking), "stream")))
                return rc;
            md->gkey = key;
            md->gsteps = 0;
        }
        // behind the starting forces of a large box the capture costs nothing
        const bool hidden = init && n >= kHiddenCapture;
        const bool several =
            n_steps >= kGraphSteps && (md->gexec[1] || hidden || md->gsteps + (long long)n_steps >= graph_pays(n));
        if (md->gsteps < graph_pays(n)) md->gsteps += std::min(n_steps, graph_pays(n));
        auto ensure = [&](int u) {
            if (md->gexec[u]) return (int)NEP_OK;
            const int r = capture(u ? kGraphSteps : 1, &md->gexec[u]);
            if (r) md->gexec[u] = nullptr;
            return r;
        };
        // the first steps singly where the graph of several is missing: the host
        // captures it while the GPU works on them
        const int single = several && !md->gexec[1] && !hidden ? kGraphSteps : 0;
        for (int s = 0; s < n_steps;) {
            const int u = several && s >= single && n_steps - s >= kGraphSteps ? 1 : 0;
            if ((rc = ensure(u))) return rc;
            if ((rc = cuda_fail(cudaGraphLaunch(md->gexec[u], st), "launch step graph"))) return rc;
            s += u ? kGraphSteps : 1;
            if (s == single && (rc = ensure(1))) return rc;
        }
        return NEP_OK;
    }

    const unsigned* gate = &md->ctl->gate;
    for (int s = 0; s < n_steps; ++s) {
        head(st, false, cudaGraphConditionalHandle{}, 1, s > 0);
        if ((rc = rebuild(st, gate))) return rc;
        if ((rc = tail(st, -1, false))) return rc;
    }
    return NEP_OK;
}

}  // extern "C"
