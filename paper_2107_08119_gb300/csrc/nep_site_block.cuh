// nep_site_block.cuh -- the site pass of the force path as a cooperation of
// four warps on 32 (or 16 or 8) atoms.
//
// What bounds it: instruction issue and dependency latency, not memory (the
// list, positions and partial forces of a 125k-atom box are about 150 MB per
// pass).  One thread per atom needs 255 registers for the 144 harmonic sums,
// leaves two warps per scheduler and, below 39k atoms, one thread's serial
// run of ~30k instructions as the time of the whole pass.  Here lane l of
// every warp works on atom i0 + l and the warps split the rest:
//   pair geometry    warp w takes the slots k = w mod 4: pair vector, cutoff
//                    tests, unit vector and radial functions, into a shared
//                    tile of 16 slots (lane-minor: no bank conflicts);
//   descriptor sums  from the tile, slots in descending order: warps 0-2
//                    eight of the 24 harmonics each, warp 3 the radial sums
//                    (each sum in one thread);
//   network          warp w takes the neurons mu = w mod 4, then a quarter of
//                    the input gradient G;
//   partial forces   warp w takes its slots again, each angular pair against
//                    the coefficients A in shared memory.
// Measured on a GB300, one thread per atom -> this form: 248 -> 186 us for the
// 125,000-atom crystal (7.6 -> 18.6 warps per SM), 104 -> 71 us for the whole MD
// step of 4,096 atoms.  Warp instructions per atom there, on the list without a
// skin: 1190 one thread per atom, 1122 this form at first, 1215 with each record
// loaded a slot ahead (the moves between the two records; no change of time
// here, and MD steps 2 % shorter), 1219 with the block sizes below.  On a list
// with 1 A of skin 1291: 46 instead of 28 slots per atom are tested.
#pragma once

#include "nep_site.cuh"

namespace nep {

constexpr int kSiteWarps = 4;
constexpr int kSiteThreads = 32 * kSiteWarps;
constexpr int kSiteChunk = 16;  // slots per shared tile

// A block takes AT = 32, 16 or 8 atoms: lane l works on atom l mod AT, and the
// 32 / AT lanes of an atom in a warp ("subs") split what the warps split once
// more (slots, neurons, quarters of G; within a harmonic or radial role the
// radial orders).
template <int AT>
struct SiteSplit {
    static constexpr int SUB = 32 / AT;
    static constexpr int WAYS = kSiteWarps * SUB;  // threads per atom
    static_assert(kSiteChunk % WAYS == 0, "every thread takes the same number of slots of a tile");
};

// Marks a tile entry outside the cutoff: both a Chebyshev argument and a
// component of a unit vector lie in [-1, 1].
constexpr float kNoPair = 2.f;

// float4 words per atom of the region that holds first the pair tile, then
// the harmonic sums S and the coefficients A
template <class D>
__host__ __device__ constexpr int site_block_quads()
{
    return ((D::NA * kLM > (3 + D::NA) * kSiteChunk ? D::NA * kLM : (3 + D::NA) * kSiteChunk) + 3) / 4;
}

// Place of S_nlm (and A_nlm) in a lane's column: harmonics in pairs (2j, 2j + 1)
// side by side, so that one 8-byte operand of a packed FMA holds both, the
// radial orders of a pair next to each other; 16-byte words are atom-minor
// ([word][AT atoms]).
template <class D, int AT>
__host__ __device__ constexpr int site_block_at(int n, int lm)
{
    const int f = 2 * ((lm >> 1) * D::NA + n) + (lm & 1);
    return (f >> 2) * 4 * AT + (f & 3);
}

// shared memory: weights | tile / S / A | q / G | radial tile / neuron states and slopes | mask words
template <class D, int AT>
__host__ __device__ constexpr size_t site_block_smem(int n_par, int n_neu)
{
    const size_t x_rows = 2 * (n_neu > kSiteChunk ? n_neu : kSiteChunk);
    return sizeof(float) * (((size_t)n_par + 31) / 32 * 32 +
                            (size_t)AT * (4 * site_block_quads<D>() + D::Ndes + x_rows + 3));
}

// Whether component a of the gradient of harmonic lm is zero for every
// direction: the 0.f entries of NEP_SH_TABLE (bit a: component a).
__host__ __device__ constexpr bool sh_zero(int lm, int a)
{
    constexpr unsigned char z[kLM] = {6, 5, 3, 4, 1, 2, 3, 4, 4, 0, 1, 3, 2, 0, 4, 4, 0, 0, 1, 3, 2, 0, 0, 4};
    return (z[lm] >> a) & 1;
}

// The values NEP_SH_TABLE refers to, for one unit vector (partial forces).
struct ShFast {
    float x, y, z, x2, y2, z2, xy, yz, xz, x2my2, a5, a7, b7, c21, e19;
    __device__ __forceinline__ void set(float ux, float uy, float uz)
    {
        x = ux;
        y = uy;
        z = uz;
        NEP_SH_LOCALS_FAST(ux, uy, uz)
        this->x2 = x2;
        this->y2 = y2;
        this->z2 = z2;
        this->xy = xy;
        this->yz = yz;
        this->xz = xz;
        this->x2my2 = x2my2;
        this->a5 = a5;
        this->a7 = a7;
        this->b7 = b7;
        this->c21 = c21;
        this->e19 = e19;
    }
};

// B += cd Y, V += cg grad Y for harmonic LM (its unprojected gradient).
template <int LM>
__device__ __forceinline__ void sh_add(const ShFast& s, float cg, float cd, float& B, float (&V)[3])
{
    const float x = s.x, y = s.y, z = s.z, x2 = s.x2, y2 = s.y2, z2 = s.z2, xy = s.xy, yz = s.yz, xz = s.xz;
    const float x2my2 = s.x2my2, z2l = 0.f, a5 = s.a5, a7 = s.a7, b7 = s.b7, c21 = s.c21, e19 = s.e19;
    (void)x; (void)y; (void)z; (void)x2; (void)y2; (void)z2; (void)xy; (void)yz; (void)xz;
    (void)x2my2; (void)z2l; (void)a5; (void)a7; (void)b7; (void)c21; (void)e19;
#define NEP_T(lm, Yv, gx, gy, gz)                                                       \
    if constexpr (LM == lm) {                                                           \
        B = fmaf(cd, Yv, B);                                                            \
        const float d[3] = {gx, gy, gz};                                                \
        _Pragma("unroll") for (int a = 0; a < 3; ++a) if (!sh_zero(lm, a)) V[a] = fmaf(cg, d[a], V[a]); \
    }
    NEP_SH_TABLE(NEP_T)
#undef NEP_T
}

// Harmonic sums of lm in [LO, LO + 8) over the tile's slots, last slot first:
// S[j][o] = (S_n,LO+2j, S_n,LO+2j+1) for the orders n = sub + SUB o (an order
// past the last repeats it and is not stored).  slots: those with a pair in
// any lane.
template <class D, int AT, int LO, int NO>
__device__ __forceinline__ void site_block_harmonics(const float* tile, int sub, unsigned slots, float2 (&S)[4][NO])
{
    constexpr int row = kSiteChunk * AT;
#pragma unroll 1
    while (slots) {
        const int s = 31 - __clz((int)slots);
        slots ^= 1u << s;
        const float* t = tile + s * AT;
        const float x = t[0];
        if (x > 1.5f) continue;  // kNoPair
        const float y = t[row], z = t[2 * row];
        float2 g[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            const int n = sub + SiteSplit<AT>::SUB * o;
            g[o] = bcast2(t[(3 + (n < D::NA ? n : D::NA - 1)) * row]);
        }
        float Y[8];
        NEP_SH_LOCALS(x, y, z)
#define NEP_T(lm, Yv, gx, gy, gz) \
    if constexpr (lm >= LO && lm < LO + 8) Y[lm - LO] = Yv;
        NEP_SH_TABLE(NEP_T)
#undef NEP_T
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int o = 0; o < NO; ++o) S[j][o] = ffma2(make_float2(Y[2 * j], Y[2 * j + 1]), g[o], S[j][o]);
    }
}

// The descriptors q_nl of order n from the harmonic sums in the atom's column
// (compensated over m): q_nl = sum_m c_lm S_nlm^2
template <class D, int AT>
__device__ __forceinline__ void site_block_descriptors(int n, const float* s_S, float* s_q)
{
    float q[kLmax] = {0.f, 0.f, 0.f, 0.f}, qc[kLmax] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int m = 0; m < kLM; ++m) {
        const int l = sh_l(m);
        const float h = s_S[site_block_at<D, AT>(n, m)];
        const float y = fmaf(sh_c(m) * h, h, -qc[l]);
        const float t = q[l] + y;
        qc[l] = (t - q[l]) - y;
        q[l] = t;
    }
#pragma unroll
    for (int l = 0; l < kLmax; ++l) s_q[(D::NR + n * kLmax + l) * AT] = q[l] - qc[l];
}

// A_nlm = 2 c_lm G_nl S_nlm in place, order n of the atom's column
template <class D, int AT>
__device__ __forceinline__ void site_block_coefficients(int n, float* s_A, const float* s_G)
{
    float g[kLmax];
#pragma unroll
    for (int l = 0; l < kLmax; ++l) g[l] = s_G[(D::NR + n * kLmax + l) * AT];
#pragma unroll
    for (int m = 0; m < kLM; ++m) {
        float* a = s_A + site_block_at<D, AT>(n, m);
        *a = *a * (2.f * sh_c(m) * g[sh_l(m)]);
    }
}

// What a pair's partial force needs of its geometry: the distance and its
// square, the unit vector u and 1/|r|, and for the energy correction what
// rounding left out of d (dd) and of u (du); w the pair's weight.
struct PairGeom {
    float u[3], d, d2, inv, dd, du[3], w;
};

// a neighbour's list value and position record
struct NbRecord {
    int v;
    float h[3], l[3], z;
};

__device__ __forceinline__ void site_pair_geometry(const NbRecord& nb, const Box& box, const SiteParams& P,
                                                   const float (&hi)[3], const float (&li)[3], float zi, PairGeom& g)
{
    float r[3], r_lo[3], u_res[3], dres;
    pair_vector_lo(nb.v >> 24, hi, li, nb.h, nb.l, box, r, r_lo);
    g.d2 = fmaf(r[0], r[0], fmaf(r[1], r[1], r[2] * r[2]));
    g.d = sqrtf(g.d2);
    unit_vector_res(r[0], r[1], r[2], g.d, g.u[0], g.u[1], g.u[2], u_res, dres, g.inv);
    const float ur = fmaf(g.u[0], r_lo[0], fmaf(g.u[1], r_lo[1], g.u[2] * r_lo[2]));
    g.dd = dres + ur;
#pragma unroll
    for (int a = 0; a < 3; ++a) g.du[a] = fmaf(fmaf(-g.u[a], ur, r_lo[a]), g.inv, u_res[a]);
    g.w = pair_weight(P, zi, nb.z);
}

// radial part of dU/dd (0 beyond the radial cutoff); s_G: the atom's column of G
template <class D, int AT>
__device__ __forceinline__ float site_pair_radial(const PairGeom& g, const SiteParams& P, const float* s_G)
{
    float radial = 0.f;
    if (g.d2 < P.rcR2) {
        float2 gd[D::NR];
        radial_gd<D::NR>(g.d, P.rcR, P.inv_rcR, gd, g.w);
#pragma unroll
        for (int a = 0; a < D::NR; ++a) radial = fmaf(s_G[a * AT], gd[a].y, radial);
    }
    return radial;
}

// Angular terms of one pair against the atom's coefficients:
// (cg, cd) = sum_n A_nlm (g_n, g_n'), B += cd Y, V += cg grad_u Y,
// two harmonics per packed FMA.  Gradient components that are zero for every
// direction (a third of them) are left out.  gg, gp: (g_n, g_n), (g_n', g_n').
template <class D, int AT, int J>
__device__ __forceinline__ void site_angular_terms(const float* s_A, const ShFast& sh, const float2 (&gg)[D::NA],
                                                   const float2 (&gp)[D::NA], float& B, float (&V)[3])
{
    if constexpr (J < kLM / 2) {
        float2 cg = make_float2(0.f, 0.f), cd = make_float2(0.f, 0.f);
#pragma unroll
        for (int n = 0; n < D::NA; ++n) {
            const float2 A = *reinterpret_cast<const float2*>(s_A + site_block_at<D, AT>(n, 2 * J));
            cg = ffma2(A, gg[n], cg);
            cd = ffma2(A, gp[n], cd);
        }
        sh_add<2 * J>(sh, cg.x, cd.x, B, V);
        sh_add<2 * J + 1>(sh, cg.y, cd.y, B, V);
        site_angular_terms<D, AT, J + 1>(s_A, sh, gg, gp, B, V);
    }
}

// One lane's atom and its pairs: the MD list (slot-major nbr[k][n], partial
// forces pf[k][n] float4), or a training set's CSR pairs (pj[p0 + k], partial
// forces of three floats each).
struct SlotMajorPairs {
    const int* nbr;
    float4* pf;
    size_t n;
    int ia;
    __device__ __forceinline__ int value(int k) const { return nbr[(size_t)k * n + ia]; }
    __device__ __forceinline__ void store(int k, float x, float y, float z) const
    {
        pf[(size_t)k * n + ia] = make_float4(x, y, z, 0.f);
    }
};

struct CsrPairs {
    const int* pj;  // of the atom's first pair
    float* pf;
    __device__ __forceinline__ int value(int k) const { return pj[k]; }
    __device__ __forceinline__ void store(int k, float x, float y, float z) const
    {
        pf[3 * (size_t)k] = x;
        pf[3 * (size_t)k + 1] = y;
        pf[3 * (size_t)k + 2] = z;
    }
};

// Shared memory of a block of AT atoms.
template <class D, int AT>
struct SiteShared {
    float* w;        // parameters
    float* A;        // [quads][AT] float4: pair tile, then S, then A
    float* q;        // [ND][AT]: q, then G
    float* x;        // radial tile; then x_mu, w2 (1 - x_mu^2): [n_neu][AT][2]
    unsigned* mask;  // [3][AT]
    __device__ __forceinline__ SiteShared(float* base, int n_par, int n_neu)
    {
        w = base;
        A = w + (n_par + 31) / 32 * 32;
        q = A + 4 * AT * site_block_quads<D>();
        x = q + AT * D::Ndes;
        mask = reinterpret_cast<unsigned*>(x + 2 * AT * (n_neu > kSiteChunk ? n_neu : kSiteChunk));
    }
};

// Descriptor sums of the block's atoms: q in sh.q, the harmonic sums S in
// sh.A, and the own-slot bits of the thread (slot k = WAYS b + way is bit
// b mod 32 of word b / 32): kept (within either cutoff) and ang (within the
// angular one).  Also zeroes sh.mask and loads the parameters z.  Ends with a
// barrier.
template <class D, int AT, int WORDS, class Pairs>
__device__ __forceinline__ void site_block_sums(const Pairs& pairs, int cnt, const float* __restrict__ xr,
                                                const Box& box, const float* __restrict__ z, int n_par,
                                                const SiteParams& P, const SiteShared<D, AT>& sh,
                                                const float (&hi)[3], const float (&li)[3], float zi,
                                                unsigned (&kept)[WORDS], unsigned (&ang)[WORDS])
{
    constexpr int NR = D::NR, NA = D::NA;
    constexpr int SUB = SiteSplit<AT>::SUB, WAYS = SiteSplit<AT>::WAYS;
    constexpr int OWN = kSiteChunk / WAYS;  // slots of a tile per thread
    __shared__ unsigned s_any[kSiteChunk];  // per tile slot: 1 an angular pair in some lane, 2 a radial one
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int at = lane % AT, sub = lane / AT;
    const int way = SUB * warp + sub;  // this thread's share of the atom's work
    float *s_A = sh.A, *s_q = sh.q, *s_x = sh.x;
    for (int t = threadIdx.x; t < n_par; t += kSiteThreads) sh.w[t] = z[t];
    if (threadIdx.x < 3 * AT) sh.mask[threadIdx.x] = 0u;
    if (threadIdx.x < kSiteChunk) s_any[threadIdx.x] = 0u;
    const int kmax = __reduce_max_sync(0xffffffffu, cnt);  // the same in every warp
    const int chunks = (kmax + kSiteChunk - 1) / kSiteChunk;
    const float rc2max = P.rcR2 > P.rcA2 ? P.rcR2 : P.rcA2;
#pragma unroll
    for (int w = 0; w < WORDS; ++w) kept[w] = ang[w] = 0u;

    // ---- descriptor sums, 16 slots at a time, the farthest first
    {
        // this warp's sums: harmonics 8 warp .. 8 warp + 7 (warps 0-2), or the
        // radial orders in pairs with their negated compensations (warp 3)
        constexpr int NO = (NA + SUB - 1) / SUB;             // angular orders per thread
        constexpr int NP = ((NR + 1) / 2 + SUB - 1) / SUB;   // pairs of radial orders per thread
        static_assert(2 * NP <= 4 * NO, "the radial sums fit the harmonic sums' registers");
        float2 S[4][NO];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int o = 0; o < NO; ++o) S[j][o] = make_float2(0.f, 0.f);
        float* tile = s_A + at;
        float2* tileR = reinterpret_cast<float2*>(s_x) + at;
        // the thread's slots in turn: k_of(0) is its first of the last tile;
        // a record is loaded one slot ahead and its list value two ahead
        auto k_of = [&](int q) { return (chunks - 1 - q / OWN) * kSiteChunk + WAYS * (q % OWN) + way; };
        auto load_v = [&](int q) {
            const int k = k_of(q);
            return q < OWN * chunks && k < cnt ? pairs.value(k) : -1;
        };
        auto load_record = [&](int v, NbRecord& r) {
            r.v = v;
            if (v >= 0) load_pos(xr, v & 0xFFFFFF, r.h, r.l, r.z);
        };
        NbRecord nx;
        load_record(load_v(0), nx);
        int v_nx = load_v(1);
        __syncthreads();  // s_any and s_mask are zero, the weights loaded
#pragma unroll 1
        for (int c = chunks - 1, q = 0; c >= 0; --c) {
#pragma unroll 1
            for (int t = 0; t < OWN; ++t, ++q) {
                const int s = WAYS * t + way;
                const NbRecord cur = nx;
                load_record(v_nx, nx);
                v_nx = load_v(q + 2);
                float x = kNoPair, fc = 0.f, ux = kNoPair;
                if (cur.v >= 0) {
                    float rx, ry, rz;
                    pair_vector(cur.v >> 24, hi, li, cur.h, cur.l, box, rx, ry, rz);
                    const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
                    if (d2 < rc2max) {
                        const int b = OWN * c + t;
                        const float w = pair_weight(P, zi, cur.z);
                        const float d = sqrtf(d2);
#pragma unroll
                        for (int w32 = 0; w32 < WORDS; ++w32)
                            if (WORDS == 1 || (b >> 5) == w32) kept[w32] |= 1u << (b & 31);
                        if (d2 < P.rcR2) radial_x(d, P.rcR, P.inv_rcR, w, x, fc);
                        if (d2 < P.rcA2) {
#pragma unroll
                            for (int w32 = 0; w32 < WORDS; ++w32)
                                if (WORDS == 1 || (b >> 5) == w32) ang[w32] |= 1u << (b & 31);
                            float g[NA], uy, uz;
                            radial_g<NA>(d, P.rcA, P.inv_rcA, g, w);
                            unit_vector(rx, ry, rz, ux, uy, uz);
                            tile[(kSiteChunk + s) * AT] = uy;
                            tile[(2 * kSiteChunk + s) * AT] = uz;
#pragma unroll
                            for (int a = 0; a < NA; ++a) tile[((3 + a) * kSiteChunk + s) * AT] = g[a];
                        }
                    }
                }
                tile[s * AT] = ux;
                tileR[s * AT] = make_float2(x, fc);
                // a slot's lanes lie in one warp: its first lane keeps the flags
                const unsigned any_a = __ballot_sync(0xffffffffu, ux < 1.5f);
                const unsigned any_r = __ballot_sync(0xffffffffu, x < 1.5f);
                if (at == 0) {
                    const unsigned m = AT == 32 ? 0xffffffffu : (1u << (AT & 31)) - 1u;
                    s_any[s] = ((any_a >> (sub * AT % 32)) & m ? 1u : 0u) | ((any_r >> (sub * AT % 32)) & m ? 2u : 0u);
                }
            }
            __syncthreads();
            unsigned slots = __ballot_sync(0xffffffffu, lane < kSiteChunk && (s_any[lane & (kSiteChunk - 1)] &
                                                                              (warp < 3 ? 1u : 2u)) != 0u);
            if (warp == 0) {
                site_block_harmonics<D, AT, 0>(tile, sub, slots, S);
            } else if (warp == 1) {
                site_block_harmonics<D, AT, 8>(tile, sub, slots, S);
            } else if (warp == 2) {
                site_block_harmonics<D, AT, 16>(tile, sub, slots, S);
            } else {
                const float2 minus = make_float2(-1.f, -1.f);
#pragma unroll 1
                while (slots) {
                    const int s = 31 - __clz((int)slots);
                    slots ^= 1u << s;
                    const float2 xf = tileR[s * AT];
                    if (xf.x > 1.5f) continue;  // kNoPair
                    float g[NR + 1];
                    float(&gn)[NR] = reinterpret_cast<float(&)[NR]>(g);
                    cheb_g<NR>(xf.x, xf.y, gn);
                    g[NR] = 0.f;
                    // Kahan: y = g - c, t = R + y, c = (t - R) - y with -c kept
#pragma unroll
                    for (int o = 0; o < NP; ++o) {
                        float2 gp = make_float2(g[2 * o * SUB], g[2 * o * SUB + 1]);
#pragma unroll
                        for (int u = 1; u < SUB; ++u)
                            if (2 * (o * SUB + u) < NR && sub == u)
                                gp = make_float2(g[2 * (o * SUB + u)], g[2 * (o * SUB + u) + 1]);
                        float2& R = S[(2 * o) / NO][(2 * o) % NO];
                        float2& nc = S[(2 * o + 1) / NO][(2 * o + 1) % NO];
                        const float2 y = fadd2(gp, nc);
                        const float2 t = fadd2(R, y);
                        nc = fadd2(y, ffma2(t, minus, R));
                        R = t;
                    }
                }
            }
            __syncthreads();
        }
        if (warp < 3) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    const int a = sub + SUB * o;
                    const int f = 2 * ((4 * warp + j) * NA + a);  // site_block_at(a, 8 warp + 2 j)
                    if (a < NA)
                        *reinterpret_cast<float2*>(s_A + (f >> 2) * 4 * AT + 4 * at + (f & 3)) = S[j][o];
                }
        } else {
#pragma unroll
            for (int o = 0; o < NP; ++o) {
                const int a = 2 * (o * SUB + sub);
                const float2 R = S[(2 * o) / NO][(2 * o) % NO], nc = S[(2 * o + 1) / NO][(2 * o + 1) % NO];
                if (a < NR) s_q[a * AT + at] = R.x + nc.x;
                if (a + 1 < NR) s_q[(a + 1) * AT + at] = R.y + nc.y;
            }
        }
    }
    __syncthreads();
    for (int a = way; a < NA; a += WAYS) site_block_descriptors<D, AT>(a, s_A + 4 * at, s_q + at);
    __syncthreads();
}

// The site pass of the block's atoms.  z: the parameters; mask: in-cutoff
// bits [3][n] of the first 96 slots, or NULL (i, n: the lane's atom and the
// number of atoms).  WORDS: 32-bit words of own-slot bits per thread.  The
// first AT lanes of warp 0 return the site energies (hi + lo).
template <class D, int AT, int WORDS, class Pairs>
__device__ __forceinline__ void site_block(const Pairs& pairs, int i, bool active, int n, int cnt,
                                           const float* __restrict__ xr, const Box& box,
                                           const float* __restrict__ z, int n_par, SiteParams P,
                                           unsigned* __restrict__ mask, float& U_hi, float& U_lo)
{
    constexpr int NA = D::NA, ND = D::Ndes;
    constexpr int SUB = SiteSplit<AT>::SUB, WAYS = SiteSplit<AT>::WAYS;
    extern __shared__ __align__(16) float s_site[];
    __shared__ float s_dU[WAYS][AT];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int at = lane % AT, sub = lane / AT;
    const int way = SUB * warp + sub;  // this thread's share of the atom's work
    const SiteShared<D, AT> sh(s_site, n_par, P.n_neu);
    float *s_w = sh.w, *s_A = sh.A, *s_q = sh.q, *s_x = sh.x;
    unsigned* s_mask = sh.mask;
    P.w = s_w;
    const int ia = active ? i : 0;
    float hi[3], li[3], zi;
    load_pos(xr, ia, hi, li, zi);
    unsigned kept[WORDS], ang[WORDS];
    site_block_sums<D, AT, WORDS>(pairs, cnt, xr, box, z, n_par, P, sh, hi, li, zi, kept, ang);
    if (mask) {
        // slot k = WAYS b + way is bit k mod 32 of word k / 32
        if constexpr (WAYS == 4) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {  // own bits 8 j .. 8 j + 7, spread to every fourth
                unsigned e = (kept[0] >> (8 * j)) & 0xFFu;
                e = (e | (e << 12)) & 0x000F000Fu;
                e = (e | (e << 6)) & 0x03030303u;
                e = (e | (e << 3)) & 0x11111111u;
                if (e) atomicOr(s_mask + j * AT + at, e << way);
            }
        } else {
            for (unsigned m = kept[0]; m; m &= m - 1) {
                const int k = WAYS * (__ffs((int)m) - 1) + way;
                atomicOr(s_mask + (k >> 5) * AT + at, 1u << (k & 31));
            }
        }
    }

    // ---- network: neurons mu = way mod WAYS
    const float* b1 = s_w + P.n_neu * ND;
    const float* w2 = b1 + P.n_neu;
    float2* s_xd = reinterpret_cast<float2*>(s_x) + at;
    {
        float q[ND];
#pragma unroll
        for (int a = 0; a < ND; ++a) q[a] = s_q[a * AT + at];
#pragma unroll 1
        for (int mu = way; mu < P.n_neu; mu += WAYS) {
            const float x = neuron_state<ND>(s_w + mu * ND, b1[mu], q);
            s_xd[mu * AT] = make_float2(x, w2[mu] * fmaf(-x, x, 1.f));
        }
    }
    __syncthreads();
    if (mask && warp < 3 && lane < AT && active) mask[(size_t)warp * n + i] = s_mask[warp * AT + lane];
    {
        // G_v of this thread's share of the descriptors, in s_q
        constexpr int VB = (ND + WAYS - 1) / WAYS;
        const int v0 = way * VB;
        if constexpr (ND % (4 * WAYS) == 0) {  // 16-byte aligned shares
            float2 G[VB / 2];
#pragma unroll
            for (int v = 0; v < VB / 2; ++v) G[v] = make_float2(0.f, 0.f);
#pragma unroll 2
            for (int mu = 0; mu < P.n_neu; ++mu) {
                const float2 d = bcast2(s_xd[mu * AT].y);
                const float4* row = reinterpret_cast<const float4*>(s_w + mu * ND + v0);
#pragma unroll
                for (int v = 0; v < VB / 4; ++v) {
                    const float4 t = row[v];
                    G[2 * v] = ffma2(d, make_float2(t.x, t.y), G[2 * v]);
                    G[2 * v + 1] = ffma2(d, make_float2(t.z, t.w), G[2 * v + 1]);
                }
            }
#pragma unroll
            for (int v = 0; v < VB / 2; ++v) {
                s_q[(v0 + 2 * v) * AT + at] = G[v].x;
                s_q[(v0 + 2 * v + 1) * AT + at] = G[v].y;
            }
        } else {
            float G[VB];
#pragma unroll
            for (int v = 0; v < VB; ++v) G[v] = 0.f;
#pragma unroll 2
            for (int mu = 0; mu < P.n_neu; ++mu) {
                const float d = s_xd[mu * AT].y;
                const float* row = s_w + mu * ND + v0;
#pragma unroll
                for (int v = 0; v < VB; ++v)
                    if (v0 + v < ND) G[v] = fmaf(d, row[v], G[v]);
            }
#pragma unroll
            for (int v = 0; v < VB; ++v)
                if (v0 + v < ND) s_q[(v0 + v) * AT + at] = G[v];
        }
    }
    __syncthreads();

    // ---- coefficients A (warps 1-3) and the compensated output sum (warp 0)
    if (warp == 0) {
        float s = 0.f, c = 0.f;
        for (int mu = 0; mu < P.n_neu; ++mu) neuron_energy(w2[mu], s_xd[mu * AT].x, s, c);
        float t, e;
        two_sum(s, -w2[P.n_neu], t, e);
        U_hi = t;
        U_lo = c + e;
    } else {
        for (int a = way - SUB; a < NA; a += WAYS - SUB)
            site_block_coefficients<D, AT>(a, s_A + 4 * at, s_q + at);
    }
    __syncthreads();

    // ---- partial forces dU_i/dr_ij of the own slots (Eqs. 23-25): radial
    // G_n g_n' rhat, angular sum_nlm A_nlm grad(g_n Z_lm); and the first-order
    // correction of the site energy for the roundings of the pair's geometry
    // in the descriptor sums.  There the descriptors were evaluated at the FP32
    // distance d and unit vector u (each rounded), from the pair vector r
    // rounded from the exact r + r_lo; with dU/dd (the radial coefficient) and
    // dU/du (the unprojected harmonic gradient V, Z_lm being polynomials in u)
    //   dE = dU/dd (|r + r_lo| - d) + dU/du . ((r + r_lo)/|r + r_lo| - u)
    // removes those roundings from U_i to second order (~1e-14 relative; the
    // terms are ~1e-7 eV, summed in FP32).
    float dU = 0.f;
    const float* sA = s_A + 4 * at;
    const float* sG = s_q + at;
    // the next own slot, the angular pairs of a word before the others: k, or
    // -1; its list value is loaded two pairs ahead, the record one ahead
    auto next_slot = [&](bool& angular) {
#pragma unroll
        for (int w = 0; w < WORDS; ++w)
            if (kept[w]) {
                angular = ang[w] != 0u;
                const int b = __ffs((int)(angular ? ang[w] : kept[w])) - 1;
                ang[w] &= ~(1u << b);
                kept[w] &= ~(1u << b);
                return WAYS * (32 * w + b) + way;
            }
        return -1;
    };
    {
        bool angular = false, angular_nx = false;
        NbRecord nb, nb_nx;
        int k = next_slot(angular);
        if (k >= 0) {
            nb.v = pairs.value(k);
            load_pos(xr, nb.v & 0xFFFFFF, nb.h, nb.l, nb.z);
        }
        int k_nx = next_slot(angular_nx);
        if (k_nx >= 0) nb_nx.v = pairs.value(k_nx);
#pragma unroll 1
        while (k >= 0) {
            bool angular_n2 = false;
            const int k_n2 = next_slot(angular_n2);
            int v_n2 = 0;
            if (k_nx >= 0) load_pos(xr, nb_nx.v & 0xFFFFFF, nb_nx.h, nb_nx.l, nb_nx.z);
            if (k_n2 >= 0) v_n2 = pairs.value(k_n2);
            PairGeom g;
            site_pair_geometry(nb, box, P, hi, li, zi, g);
            float radial = site_pair_radial<D, AT>(g, P, sG);
            float V[3] = {0.f, 0.f, 0.f};
            float eu = 0.f;
            if (angular) {
                float2 gg[NA], gp[NA];
                {
                    float2 gd[NA];
                    radial_gd<NA>(g.d, P.rcA, P.inv_rcA, gd, g.w);
#pragma unroll
                    for (int a = 0; a < NA; ++a) {
                        gg[a] = bcast2(gd[a].x);
                        gp[a] = bcast2(gd[a].y);
                    }
                }
                ShFast sh;
                sh.set(g.u[0], g.u[1], g.u[2]);
                site_angular_terms<D, AT, 0>(sA, sh, gg, gp, radial, V);
                eu = fmaf(V[0], g.du[0], fmaf(V[1], g.du[1], V[2] * g.du[2]));
                // tangential projection of V, divided by r
                const float uv = fmaf(g.u[0], V[0], fmaf(g.u[1], V[1], g.u[2] * V[2]));
#pragma unroll
                for (int a = 0; a < 3; ++a) V[a] = (V[a] - uv * g.u[a]) * g.inv;
            }
            dU += fmaf(radial, g.dd, eu);
            pairs.store(k, fmaf(radial, g.u[0], V[0]), fmaf(radial, g.u[1], V[1]), fmaf(radial, g.u[2], V[2]));
            k = k_nx;
            angular = angular_nx;
            nb = nb_nx;
            k_nx = k_n2;
            angular_nx = angular_n2;
            nb_nx.v = v_n2;
        }
    }
    s_dU[way][at] = dU;
    __syncthreads();
    if (warp == 0) {
        float t[WAYS];
#pragma unroll
        for (int w = 0; w < WAYS; ++w) t[w] = s_dU[w][at];
#pragma unroll
        for (int h = WAYS / 2; h >= 1; h >>= 1)
#pragma unroll
            for (int w = 0; w < h; ++w) t[w] += t[w + h];
        U_lo += t[0];
    }
}

}  // namespace nep
