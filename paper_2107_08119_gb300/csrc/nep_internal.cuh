// nep_internal.cuh -- shared definitions of the sm_103a NEP library.
//
// Data layout in device memory (n atoms, M = neighbour capacity per atom):
//   positions        FP64 [3][n] (caller) + FP32 hi/lo records xr [n][8]
//   neighbour list   int32 nbr[M][n] = j | image_code << 24, count[n]
//                    int32 rev[M][n] = slot of i in j's list (reverse pair)
//                    int32 vala[n][M]: direct list, the list values atom-major;
//                    cells path, the rank of each unsorted slot
//   partial forces   FP32 pf[M][n] float4 (x, y, z, unused) = dU_i/dr_ij
//                    (Eq. 23), slot-major: one 16-byte gather per reverse pair
//   forces           FP32 [3][n], per-atom virials FP32 [9][n]
// Slot-major layouts make the per-atom loops of a warp read consecutive
// addresses at every slot.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nep.h"

namespace nep {

__host__ __device__ __forceinline__ int imin(int a, int b) { return a < b ? a : b; }

// Packed FP32 pairs.  On the device these are the f32x2 instructions
// (__ffma2_rn / __fmul2_rn: two IEEE round-to-nearest operations per
// instruction, bitwise the same as two scalar fmaf / products); on the host
// the two scalar operations.  bcast2(x) = (x, x) is the broadcast operand.
__host__ __device__ __forceinline__ float2 bcast2(float x) { return make_float2(x, x); }

__host__ __device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c)
{
#ifdef __CUDA_ARCH__
    return __ffma2_rn(a, b, c);
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}

__host__ __device__ __forceinline__ float2 fadd2(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    return __fadd2_rn(a, b);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}

// ---------------------------------------------------------------- sizes
constexpr int kNR = 8;               // radial orders n = 0..7
constexpr int kNA = 6;               // angular radial orders n = 0..5
constexpr int kLmax = 4;             // Legendre orders l = 1..4
constexpr int kLM = 24;              // real harmonics with 1 <= l <= 4: 3+5+7+9
constexpr int kNdes = kNR + kNA * kLmax;  // 32
constexpr int kMaxNeu = 64;
constexpr int kMaxAtoms = (1 << 24) - 1;
constexpr int kImgCenter = 62;       // image code of the zero shift
// Largest cell grid of the list build (nc[0] nc[1] nc[2]).  A large, sparse
// box would otherwise need more cells than an int counts; the grid is then
// made coarser, which stays correct because every cell edge is still at
// least the list radius.
constexpr int kMaxCells = 1 << 22;

// device error word bits
enum : unsigned {
    kErrOverflow = 1u,
    kErrNonFinite = 2u,
    kErrReverse = 4u,
    kErrTimeout = 8u,
};

// Orthorhombic periodic box; lengths split into FP32 hi + lo parts so that a
// pair vector can be formed to FP32 rounding from hi/lo positions.
struct Box {
    double L[3];
    float Lh[3];
    float Ll[3];
    int nc[3];      // cells per direction (0 when the brute-force list is used)
    double cpl[3];  // cells per unit length nc / L (binning without a division)
    int img[3];     // largest |image shift| a pair can need per direction
};

// Image code of shift (sx, sy, sz), each in [-2, 2].
__host__ __device__ __forceinline__ int image_code(int sx, int sy, int sz)
{
    return (sx + 2) * 25 + (sy + 2) * 5 + (sz + 2);
}

__host__ __device__ __forceinline__ void image_shift(int code, int& sx, int& sy, int& sz)
{
    sx = code / 25 - 2;
    sy = (code / 5) % 5 - 2;
    sz = code % 5 - 2;
}

// r = (x_a + s L) - x_b from hi/lo parts.  The box length is combined first
// with whichever atom sits near the far face (b when s > 0, a when s < 0), so
// that subtraction is exact (Sterbenz) and only the final small difference
// rounds; adding L to the atom near the origin would round at ulp(L).
__host__ __device__ __forceinline__ float diff1(float ah, float al, float bh, float bl, float s, float Lh, float Ll)
{
    const float hi = (s > 0.f) ? ah - fmaf(-s, Lh, bh) : fmaf(s, Lh, ah) - bh;
    const float lo = fmaf(s, Ll, al - bl);
    return hi + lo;
}

// Pair vector r_ij = x_j + shift(code) - x_i.  Swapping the two atoms (and the
// sign of the shift) swaps the operands of every subtraction in diff1, so
// r_ji == -r_ij exactly whichever of the two evaluates it.  Most pairs cross
// no box face: their shift is zero and the general form reduces to three
// subtractions and sums (the same values), without the decoding of the image.
__host__ __device__ __forceinline__ void pair_vector(int code, const float (&hi)[3], const float (&li)[3],
                                                     const float (&hj)[3], const float (&lj)[3], const Box& b,
                                                     float& rx, float& ry, float& rz)
{
    if (code == kImgCenter) {
        rx = (hj[0] - hi[0]) + (lj[0] - li[0]);
        ry = (hj[1] - hi[1]) + (lj[1] - li[1]);
        rz = (hj[2] - hi[2]) + (lj[2] - li[2]);
        return;
    }
    int sx, sy, sz;
    image_shift(code, sx, sy, sz);
    rx = diff1(hj[0], lj[0], hi[0], li[0], (float)sx, b.Lh[0], b.Ll[0]);
    ry = diff1(hj[1], lj[1], hi[1], li[1], (float)sy, b.Lh[1], b.Ll[1]);
    rz = diff1(hj[2], lj[2], hi[2], li[2], (float)sz, b.Lh[2], b.Ll[2]);
}

// pair_vector that also returns the rounding residual of each component:
// r_exact = r + r_lo to within the tiny rounding of the lo parts (~1e-14 A).
// The hi-part difference is exact, so r = hi + lo rounds once and Fast2Sum
// recovers what that rounding dropped.
__host__ __device__ __forceinline__ float diff1_lo(float ah, float al, float bh, float bl, float s, float Lh, float Ll,
                                                   float& r_lo)
{
    const float hi = (s > 0.f) ? ah - fmaf(-s, Lh, bh) : fmaf(s, Lh, ah) - bh;
    const float lo = fmaf(s, Ll, al - bl);
    const float r = hi + lo;
    r_lo = lo - (r - hi);
    return r;
}

__host__ __device__ __forceinline__ void pair_vector_lo(int code, const float (&hi)[3], const float (&li)[3],
                                                        const float (&hj)[3], const float (&lj)[3], const Box& b,
                                                        float (&r)[3], float (&r_lo)[3])
{
    if (code == kImgCenter) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float h = hj[d] - hi[d], l = lj[d] - li[d];
            r[d] = h + l;
            r_lo[d] = l - (r[d] - h);
        }
        return;
    }
    int s[3];
    image_shift(code, s[0], s[1], s[2]);
#pragma unroll
    for (int d = 0; d < 3; ++d) r[d] = diff1_lo(hj[d], lj[d], hi[d], li[d], (float)s[d], b.Lh[d], b.Ll[d], r_lo[d]);
}

#pragma nv_diag_suppress 550  // the record's last word is loaded and not used
// FP32 hi/lo positions: one 32-byte record (x, y, z, species number; lo parts
// x, y, z, 0) per atom, so that a neighbour's coordinates are one sector and
// one 32-byte load (two 16-byte arrays before: two sectors; an MD step of the
// 125,000-atom crystal 315 -> 309 us together with the site pass loading its
// records a slot ahead).  An ordinary load in volatile assembly: it stays behind
// the wait of a dependent kernel (block_after), as the read-only path would not.
__host__ __device__ __forceinline__ void load_pos(const float* __restrict__ xr, int i, float (&h)[3], float (&l)[3],
                                                  float& zi)
{
#ifdef __CUDA_ARCH__
    float u, pad;
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(h[0]), "=f"(h[1]), "=f"(h[2]), "=f"(u), "=f"(l[0]), "=f"(l[1]), "=f"(l[2]), "=f"(pad)
        : "l"(xr + 8 * (size_t)i));
    zi = u;
    (void)pad;
#else
    const float* r = xr + 8 * (size_t)i;
    for (int d = 0; d < 3; ++d) {
        h[d] = r[d];
        l[d] = r[4 + d];
    }
    zi = r[3];
#endif
}

#pragma nv_diag_default 550
__host__ __device__ __forceinline__ void load_pos(const float* __restrict__ xr, int i, float (&h)[3], float (&l)[3])
{
    float zi;
    load_pos(xr, i, h, l, zi);
}

// the hi part of the record (x, y, z, species number)
__host__ __device__ __forceinline__ float4 load_hi(const float* __restrict__ xr, int i)
{
    return reinterpret_cast<const float4*>(xr)[2 * (size_t)i];
}

// Split an FP64 value into FP32 hi + lo.
__host__ __device__ __forceinline__ void split_hilo(double x, float& h, float& l)
{
    h = (float)x;
    l = (float)(x - (double)h);
}

// (float)x and its value as a double by integer operations (round to nearest
// even): conversions from and to FP64 run at the rate of the FP64 pipe, two
// lanes per clock and SM, and bounded the kernels that split positions
// (k_kick_drift at 921,600 atoms 51.9 -> 45.6 us, k_bin 35.1 -> 29.2).  In the
// assembly, which waits for gathers, the same changed nothing.
__device__ __forceinline__ float to_float(double x, double& back)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned e = (unsigned)(b >> 52) & 0x7FFu;
    if (e - 922u >= 200u) {  // zero, beyond 2^99 or below 2^-101, infinite or not a number
        const float f = (float)x;
        back = (double)f;
        return f;
    }
    const unsigned long long r = b + 0x0FFFFFFFull + ((b >> 29) & 1ull);
    back = __longlong_as_double((long long)(r & ~0x1FFFFFFFull));
    return __uint_as_float(((unsigned)(r >> 32) & 0x80000000u) | ((unsigned)(r >> 29) - (896u << 23)));
}

__device__ __forceinline__ double to_double(float f)
{
    const unsigned u = __float_as_uint(f), a = u & 0x7FFFFFFFu;
    if (a - 0x00800000u >= 0x7F000000u) return (double)f;  // zero, denormal, infinite or not a number
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
}

// The hi part's fourth word carries the atom's species number Z (1 for a
// single species): the multicomponent weighting f_c -> f_c sqrt(Z_i Z_j).
__host__ __device__ __forceinline__ void store_pos(float* __restrict__ xr, int i, const double (&x)[3], float zi = 1.f)
{
    float h[3], l[3];
#ifdef __CUDA_ARCH__
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double hd, ld;
        h[d] = to_float(x[d], hd);
        l[d] = to_float(x[d] - hd, ld);
    }
#else
    for (int d = 0; d < 3; ++d) split_hilo(x[d], h[d], l[d]);
#endif
    float4* r = reinterpret_cast<float4*>(xr) + 2 * (size_t)i;
    r[0] = make_float4(h[0], h[1], h[2], zi);
    r[1] = make_float4(l[0], l[1], l[2], 0.f);
}

__host__ __device__ __forceinline__ float load_z(const float* __restrict__ xr, int i)
{
    return reinterpret_cast<const float4*>(xr)[2 * (size_t)i].w;
}

// Warp sum of K <= 16 doubles held by every lane.  Each butterfly level keeps
// half of the remaining components (the lane sends the half its partner keeps),
// so a lane does 8 + 4 + 2 + 1 + 1 additions instead of 5 K.  On return
// lanes 2c and 2c + 1 hold the warp total of component warp_comp(lane) (the
// pattern is fixed, so the sums are deterministic).
__device__ __forceinline__ int warp_comp(int lane)
{
    return ((lane & 16) ? 8 : 0) + ((lane & 8) ? 4 : 0) + ((lane & 4) ? 2 : 0) + ((lane & 2) ? 1 : 0);
}

template <int K>
__device__ __forceinline__ double warp_sum_multi(const double (&v)[K])
{
    static_assert(K <= 16, "at most 16 components");
    const int lane = threadIdx.x & 31;
    double a[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) a[c] = c < K ? v[c] : 0.0;
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int c = 0; c < h; ++c) {
            const double send = upper ? a[c] : a[c + h];
            const double keep = upper ? a[c + h] : a[c];
            a[c] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return a[0] + __shfl_xor_sync(0xffffffffu, a[0], 1);
}

// Block-wide sum of K doubles; writes out[k * stride].  blockDim.x must be a
// multiple of 32 and at most 1024.
template <int K>
__device__ __forceinline__ void block_sum_store(double (&v)[K], double* __restrict__ out, size_t stride = 1)
{
    __shared__ double red[32][K];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    if constexpr (K >= 4) {
        const double s = warp_sum_multi<K>(v);
        const int c = warp_comp(lane);
        if ((lane & 1) == 0 && c < K) red[warp][c] = s;
        __syncthreads();
        if (warp == 0) {
            double w[K];
#pragma unroll
            for (int k = 0; k < K; ++k) w[k] = lane < nw ? red[lane][k] : 0.0;
            const double t = warp_sum_multi<K>(w);
            if ((lane & 1) == 0 && c < K) out[c * stride] = t;
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < K; ++k) red[warp][k] = v[k];
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                double s = lane < nw ? red[lane][k] : 0.0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) out[k * stride] = s;
            }
        }
    }
}

// Sum over b < nb of src[b stride] by the THREADS threads of a block, in a
// fixed order: each thread a fixed stride of the values (eight loads in flight
// ahead of the ordered adds), a shuffle tree, the warps in order.  Thread 0
// returns it.
template <int THREADS>
__device__ __forceinline__ double sum_partials(const double* __restrict__ src, int nb, int stride)
{
    __shared__ double wsum[THREADS / 32];
    double v = 0.0;
#pragma unroll 8
    for (int b = threadIdx.x; b < nb; b += THREADS) v += src[(size_t)b * stride];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < THREADS / 32; ++q) t += wsum[q];
    return t;
}

// Launches right behind another kernel.  A kernel that launch_after enqueues
// with after = true is set up while the last blocks of its predecessor in the
// stream run, so the gap between the two is that of a block, not of a grid.  It
// begins with block_after(), which waits until everything before it in the
// stream is done and visible; no kernel lets its successor start any earlier
// than that (an early trigger made a driven step of 13,824 atoms 9 % slower:
// waiting blocks took the running ones' places).  after is true only where the
// predecessor is a kernel of the same call on the same stream, not a wait for an
// event, a copy or a conditional node.  96 atoms 92 -> 81 us per call, 125,000
// atoms 430 -> 416, MD step of 4,096 atoms 45.0 -> 43.8 us.
// What orders the loads: the wait clobbers memory, so ordinary loads and stores
// stay behind it, but a load that the compiler may take for invariant does not
// have to.  So a kernel that calls block_after() has no __restrict__ parameter,
// uses no read-only load (__ldg, ld.global.nc), and reaches global memory in
// inline assembly only where that is volatile, or through a pointer that
// reread() has passed on behind the wait.
// Returns blockIdx.x (read in the assembly of the wait it was no longer known to
// be uniform: steps of 64,000 two-species atoms 2.5 % slower).
__device__ __forceinline__ int block_after()
{
    cudaGridDependencySynchronize();
    return (int)blockIdx.x;
}

// The same pointer, known only behind block_after()
template <class T>
__device__ __forceinline__ T* reread(T* p)
{
    asm volatile("" : "+l"(p)::"memory");
    return p;
}

template <class... Par, class... Arg>
cudaError_t launch_after(bool after, void (*kern)(Par...), dim3 grid, int block, size_t smem, cudaStream_t st,
                         Arg... arg)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = after ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, Par(arg)...);
}

// Dynamic shared memory that a kernel gets without asking: 48 KB hold its static
// part too, here taken as at most 1 KB (the site pass has 576 bytes).
constexpr size_t kDefaultShared = 47 * 1024;

// ---------------------------------------------------------------- workspace
struct NeighborList {
    int n_cap = 0;       // atoms the buffers hold
    int m_cap = 0;       // neighbour slots per atom
    int ncell_cap = 0;
    int* count = nullptr;
    int* nbr = nullptr;
    int* rev = nullptr;
    int* vala = nullptr;     // direct list: list values atom-major [n][m_cap]; cells path: ranks of the unsorted slots
    float* pf = nullptr;
    float* xr = nullptr;     // hi/lo position records [n][8]
    int* atom_cell = nullptr;
    int* cell_count = nullptr;
    int* cell_start = nullptr;
    float4* xs = nullptr;    // hi parts and indices in cell order [n]
    // [3][n] words: bit k of atom i set when slot k lies within the cutoff,
    // written by the site pass from its cutoff tests; `mask_set`
    // (host) says whether the last site pass launched wrote them, so that
    // the assembly skips the other slots' loads.
    unsigned* mask = nullptr;
    bool mask_set = false;
};

struct Workspace {
    NeighborList nl;
    double* partials = nullptr;  // per-block FP64 partial sums
    int partial_cap = 0;         // doubles
    float* force = nullptr;      // [3][n] FP32 (MD and internal use)
    int force_cap = 0;
    float* plain = nullptr;      // [2][32][n] q and G of the plain comparator (on demand)
    int plain_cap = 0;
};

// host-side helpers (nep_api.cu)
void set_error(const char* fmt, ...);
int cuda_fail(cudaError_t e, const char* what);
int ensure_workspace(Workspace& ws, int n, int m_cap, int ncell, int nblocks_partials);
void free_workspace(Workspace& ws);
int setup_box(const double* box9, double r_list, Box& b);

// neighbour list (nep_neighbor.cu)
// mode: build from positions `pos` (FP64 [3][n]); when wrap_in_place is true
// the wrapped positions are written back to pos and to x_ref (if non-null).
// zatom: species number of every atom (dev [n]) or NULL (all 1)
int build_neighbor_list(NeighborList& nl, const Box& b, int n, double* pos, const float* zatom, bool wrap_in_place,
                        double* x_ref,
                        float r_list, unsigned* d_err, const unsigned* d_gate, cudaStream_t st);

// whether the list of n atoms in a box with a cell grid is built by direct tests
bool list_is_direct(int n);

// force path (nep_force.cu)
struct ForceArgs {
    const float* z;          // parameters on the device
    int n_neu;
    float rcR, rcA;
    Box box;
    int typed = 0;           // species numbers in the position records are used (multicomponent)
    int nr = kNR;            // radial orders n_max^R + 1 (8, or 13 for the split model)
    int na = kNA;            // angular radial orders n_max^A + 1 (6, or 7)
};
// The descriptor sizes with force-path kernels: the 32-descriptor model
// (n_max^R = 7, n_max^A = 5) and the split 41-descriptor model (12, 6),
// both with l_max = 4.  Only the force path (energies, forces, virials, MD)
// has kernels for the second; training sets, the plain comparator and the
// allocation-free call need the first.
inline bool sizes_default(const nep_hyper& h) { return h.n_max_R == kNR - 1 && h.n_max_A == kNA - 1; }
inline bool sizes_split(const nep_hyper& h) { return h.n_max_R == 12 && h.n_max_A == 6; }
// Atoms per 128-thread block of the site pass and the assembly: 8 or 16 while
// one wave of blocks (152 SMs x 5) holds them all, else 32.  More threads per
// atom shorten a block's run, fewer waste less (harmonics evaluated by every
// lane of an atom, narrower rows).  Site pass with 8 / 16 / 32 atoms per block:
// 512 atoms 10.7 / 13.8 / 20.4 us, 5832 atoms 17.3 / 18.2 / 24.0, 8000 atoms
// 25.8 / 21.5 / 24.3, 13824 atoms 37.9 / 33.5 / 28.9, 32768 atoms 79 / 62 / 57.
constexpr int kSiteWave = 152 * 5;
constexpr int site_atoms_per_block(int n) { return n <= 8 * kSiteWave ? 8 : n <= 16 * kSiteWave ? 16 : 32; }
// blocks of the site pass (its per-block energy partials), which also bounds
// the block counts of the assembly and of the plain comparator
constexpr int site_blocks(int n) { return (n + site_atoms_per_block(n) - 1) / site_atoms_per_block(n); }
// after: the predecessor in the stream is a kernel that lets this one be set up
int launch_site_partial_forces(const ForceArgs& a, NeighborList& nl, int n, double* e_atom, double* e_partials,
                               unsigned* d_err, cudaStream_t st, int& nblocks, bool after = false);
struct AssembleArgs {
    float rc_max;
    Box box;
    // MD extras (used when vel != nullptr)
    double* vel;
    double half_dt_over_m;   // dt/2 / (m * unit)
    double ke_factor;        // 0.5 m * unit
    bool heat;
};
int launch_assemble(const AssembleArgs& a, NeighborList& nl, int n, float* force, float* virial_atom,
                    double* partials, unsigned* d_err, cudaStream_t st, int& nblocks, int& ncomp);
// ncomp totals: out[w] = the sum over b < nb of src[w cstride + b bstride]
// (out NULL: none)
struct SumSet {
    const double* src = nullptr;
    int nb = 0, bstride = 1, ncomp = 0;
    size_t cstride = 0;
    double* out = nullptr;
};
int launch_sum(const SumSet& a, const SumSet& b, cudaStream_t st, bool after = false);
// the plain FP32 comparator (nep_plain.cu): descriptors, network and partial
// forces by the literal formulas, q and G [32][n] scratch
int launch_plain_site(const ForceArgs& a, NeighborList& nl, int n, float* q, float* G, double* e_atom,
                      double* e_partials, unsigned* d_err, cudaStream_t st, int& nblocks);

}  // namespace nep

namespace nep {
// CUDA-event pairs around kernel launches (enabled on demand).
struct Profiler {
    bool on = false;
    struct Slot {
        cudaEvent_t a = nullptr, b = nullptr;
        int kind = 0;
    };
    Slot* slots = nullptr;
    int cap = 0, used = 0;
    // returns the slot to bracket a launch of `kind`, or nullptr when off/full
    Slot* begin(int kind, cudaStream_t st);
    void end(Slot* s, cudaStream_t st);
    int read(double* ms, long long* cnt);  // ms[NEP_PROFILE_KINDS], cnt[...]; synchronises
    void release();
};
// tensor-core population network (nep_pop_tc.cu)
size_t pop_tc_packed_bytes(int P);
// kernel attributes of the tensor-core path; call outside any stream capture
int prepare_pop_tc();
// G [N][32][Pst] FP32, U [N][P] FP64 (launches only: capturable)
// the descriptors packed as split-BF16 GEMM-1 A tiles, once per training set
size_t pop_tc_qpack_bytes(int N);
int launch_pack_q_tc(int N, const float* q, unsigned char* qpack, cudaStream_t st);
// Layout of G written by the population network:
//   kGRowsF32  [N][32][Pst] FP32;   kGRowsF16  [N][32][Pst] FP16;
//   kGTilesF16 per atom the tensor-core B tile of the owner pass: members
//              as rows of a K-major [8 ceil(Pst / 8)] x 32 FP16 tile
//              (owner_tc_g_bytes(Pst) bytes per atom, nep_tc.cuh layout).
enum GLayout { kGRowsF32 = 0, kGRowsF16 = 1, kGTilesF16 = 2 };
// z: the population [P][n_par] (packed into the group records by the launch),
// or NULL when `packed` already holds it (launch_pack_tc_draw)
// pipelined: the persistent warp-specialised kernel (same bits), else one CTA
// per (member group, 128-atom tile)
int launch_pop_tc(int N, int P, int Pst, int n_neu, const unsigned char* qpack, const float* z, unsigned char* packed,
                  void* G, int g_layout, double* U, unsigned* err, bool pipelined, cudaStream_t st);
// An SNES generation's draws and population packed in one launch: r [P][n_par]
// the standard normals of generation *d_gen (the stream of nep_philox.cuh),
// z = m + s (.) r, and the group records of z, with the same bits as the draw
// kernel followed by the packing of launch_pop_tc.
int launch_pack_tc_draw(int P, int n_neu, unsigned long long seed, const unsigned* d_gen, const float* m,
                        const float* s, float* r, float* z, unsigned char* packed, cudaStream_t st);

// The first contraction pass on the tensor cores (BF16 precision mode).  A
// tile is up to 128 rows of one owner atom j: three per pair (the Jacobian
// rows d p / d G of components x, y, z), and in the owner's first tile three
// rows of its own term (B_j) and six of its virial contribution
// (-sum_pairs r^a J^b, components xx yy zz xy yz zx).
struct OwnerTile {
    int j;           // owner atom
    int nt;          // pairs in this tile
    int extra;       // 1: the own-term and virial rows follow the pair rows
    int groups;      // 8-row groups stored
    long long q0;    // first pair (owner order)
    long long row0;  // first row of the tile in the packed operand (multiple of 8)
};
constexpr int kOwnerTcPairs = 39;  // pairs of a first tile (3 x 39 + 9 <= 128 rows)
constexpr int kOwnerTcMorePairs = 42;  // pairs of each further tile
// bytes of one atom's G tile in the kGTilesF16 layout
__host__ __device__ inline size_t owner_tc_g_bytes(int Pst) { return (size_t)((Pst + 7) / 8) * 512; }
struct PairRec;
// packs the Jacobian rows of every tile as FP16 (each row scaled by a power
// of two, kept in rowscale, so that its largest entry lies in [2^13, 2^14));
// once per training set
int launch_pack_owner_tc(int n_tiles, const OwnerTile* tiles, const PairRec* rec, const long long* aidx,
                         const float* ang, const float* B, const long long* pstart, unsigned char* apack,
                         float* rowscale, cudaStream_t st);
int prepare_owner_tc();
// tiles [t0, t1): partial forces p_kji (FP16, at the receiver's slot rev[q]),
// own terms and virial terms (FP32), as the CUDA-core owner pass writes them
int launch_owner_tc(int t0, int t1, const OwnerTile* tiles, const unsigned char* apack, const float* rowscale,
                    const void* G, int Pst, const long long* rev, void* pbuf, float* fown, float* w6, unsigned* err,
                    cudaStream_t st);

}  // namespace nep

struct nep_model {
    nep_hyper hp;
    nep::Profiler prof;
    int n_des = 0;
    int n_par = 0;
    float* d_z = nullptr;
    unsigned* d_err = nullptr;   // latched device error bits
    nep::Workspace ws;
    float* zatom = nullptr;      // species numbers of the atoms (nep_set_species), or NULL
    int zatom_n = 0;
};

namespace nep {
// status from latched device error bits
int status_from_bits(unsigned bits);
}
