// nep_neighbor.cu -- cell binning and Verlet neighbour list on the device.
//
// The paper keeps neighbour lists of atoms within the cutoffs (Sec. III.C,
// "memory consumption") without describing their construction.  Here:
//   1. wrap positions into the orthorhombic box, split them into FP32 hi/lo,
//      bin atoms into cells of edge >= the list radius;
//   2. exclusive scan of the cell counts and scatter (the order of atoms
//      within a cell is whatever the atomics give: the list order below
//      depends only on the sort keys, so it stays deterministic);
//   3. every pair within the list radius is tested once, by the atom whose
//      half shell of cells holds the other, and goes into both atoms' rows
//      (full list, both directions), unsorted; each row is then ordered by
//      increasing distance, and the reverse-pair index (for slot k of atom
//      i, the slot of i in j's list) follows from the partners' ranks
//      (k_half_cells, k_sort_tile, k_rev_tile below);
// Boxes with fewer than 3 cells in a direction (small training cells) and
// small atom counts test every pair instead (k_list_direct: the sorted keys
// atom-major in the partial-force buffer, the values in vala), with the
// reverse index by binary search over j's keys (k_reverse).
// Every kernel takes an optional device gate word: when it is zero the kernel
// returns at once, which lets the MD step skip the rebuild without a host
// round trip.
#include <algorithm>
#include <cstdio>

#include "nep_internal.cuh"

namespace nep {

namespace {

__device__ __forceinline__ bool gated_off(const unsigned* gate)
{
    return gate != nullptr && *((volatile const unsigned*)gate) == 0u;
}

// A non-finite coordinate latches kErrNonFinite: such an atom would
// otherwise be binned into a clamped cell and simply see no neighbours.
__global__ void k_bin(int n, double* __restrict__ pos, const float* __restrict__ zatom, int wrap_in_place,
                      double* __restrict__ x_ref, float* __restrict__ xr,
                      int* __restrict__ atom_cell, int* __restrict__ cell_count, int* __restrict__ count, Box b,
                      const unsigned* gate, unsigned* __restrict__ err)
{
    if (gated_off(gate)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    count[i] = 0;  // the half-shell search counts each row's entries with atomics
    int c[3];
    double wx[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double L = b.L[d];
        const double x = pos[(size_t)d * n + i];
        // FP64 operations are slow here (comparisons and division among them):
        // 0 <= x < L, nearly every atom, is one integer comparison of the bits
        // (a negative or non-finite x compares above), and atoms within one box
        // length of the box wrap without a division: exactly from above, with one
        // rounding from below (a tiny negative x gives L, then 0)
        double w = x;
        if ((unsigned long long)__double_as_longlong(x) >= (unsigned long long)__double_as_longlong(L)) {
            if (!isfinite(x)) atomicOr(err, kErrNonFinite);
            if (x >= L && x < 2.0 * L)
                w = x - L;
            else if (x < 0.0 && x >= -L)
                w = x + L;
            else if (!(x == 0.0))
                w = x - L * floor(x / L);
            if (w >= L) w -= L;
            if (w < 0.0) w = 0.0;
        }
        if (wrap_in_place) {
            pos[(size_t)d * n + i] = w;
            if (x_ref) x_ref[(size_t)d * n + i] = w;
        }
        wx[d] = w;
        if (b.nc[0] > 0) {
            // any cell within rounding of the true one is valid (cells are at
            // least the list radius wide); the list order depends only on keys
            int ci = (int)(w * b.cpl[d]);
            c[d] = ci < 0 ? 0 : (ci >= b.nc[d] ? b.nc[d] - 1 : ci);
        }
    }
    store_pos(xr, i, wx, zatom ? zatom[i] : 1.f);
    if (b.nc[0] > 0) {
        const int cid = (c[0] * b.nc[1] + c[1]) * b.nc[2] + c[2];
        atom_cell[i] = cid;
        atomicAdd(cell_count + cid, 1);
    }
}

// Exclusive scan cell_start[c] = sum_{c' < c} count[c'] by blocks that do not
// wait on one another: each adds up all counts before its slice (they are in L2),
// then scans the slice in rounds of blockDim * kScanPer cells through shared
// memory (coalesced global reads and writes; padded so that a thread's run of
// kScanPer consecutive cells is conflict-free); warp shuffles and the warp totals
// give the prefix.  A round is a chain of four barriers, so one block for all
// cells took 12.8 us at 19,683 and 51 at 93,312 cells (now 3.8 and 6.2; the call
// of 125,000 atoms 410 -> 403 us).  Slices of one round up to 152 of
// them: the reads before the slices are at most 76 times the counts.
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 8;  // 32 cells per thread and a third of the rounds took the same time
constexpr int kScanRound = kScanThreads * kScanPer;

__device__ __forceinline__ int scan_pad(int x) { return x + (x >> 5); }

__global__ void __launch_bounds__(kScanThreads) k_scan(int ncell, int slice, const int* count,
                                                       int* start, const unsigned* gate)
{
    const int c0 = block_after() * slice, c1 = min(ncell, c0 + slice);
    if (gated_off(gate)) return;
    __shared__ int sc[kScanRound + kScanRound / 32];
    __shared__ int wsum[kScanThreads / 32];
    __shared__ int carry;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int before = 0;
    const int4* c4 = reinterpret_cast<const int4*>(count);  // c0 is a multiple of 4, the counts are 256-byte aligned
#pragma unroll 4
    for (int x = t; x < c0 / 4; x += kScanThreads) {
        const int4 q = c4[x];
        before += (q.x + q.y) + (q.z + q.w);
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) wsum[warp] = before;
    __syncthreads();
    if (warp == 0) {
        const int all = __reduce_add_sync(0xffffffffu, wsum[lane]);
        if (lane == 0) carry = all;
    }
    __syncthreads();
    for (int base = c0; base < c1; base += kScanRound) {
#pragma unroll
        for (int e = 0; e < kScanPer; ++e) {
            const int x = e * kScanThreads + t;
            sc[scan_pad(x)] = base + x < c1 ? count[base + x] : 0;
        }
        __syncthreads();
        int v[kScanPer];
        int s = 0;
#pragma unroll
        for (int e = 0; e < kScanPer; ++e) {
            v[e] = sc[scan_pad(t * kScanPer + e)];
            s += v[e];
        }
        int incl = s;  // inclusive scan of the thread sums within the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            int w = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            wsum[lane] = w;  // inclusive over warps
        }
        __syncthreads();
        int run = carry + (warp > 0 ? wsum[warp - 1] : 0) + incl - s;
#pragma unroll
        for (int e = 0; e < kScanPer; ++e) {
            sc[scan_pad(t * kScanPer + e)] = run;
            run += v[e];
        }
        __syncthreads();  // every thread has read carry and wsum, and sc holds the prefixes
        if (t == kScanThreads - 1) carry = run;
#pragma unroll
        for (int e = 0; e < kScanPer; ++e) {
            const int x = e * kScanThreads + t;
            if (base + x < c1) start[base + x] = sc[scan_pad(x)];
        }
        __syncthreads();
    }
    if (t == 0 && c1 == ncell) start[ncell] = carry;
}

// Atoms in cell order: their hi parts with the index in the fourth word, so
// that a cell's candidates are contiguous 16-byte reads.  Counts down the cells'
// counters, which are zero again after it.
__global__ void k_scatter(int n, const int* atom_cell, const int* cell_start,
                          int* cell_count, const float* xr, float4* xs,
                          const unsigned* gate)
{
    const int block = block_after();
    if (gated_off(gate)) return;
    const int i = block * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = atom_cell[i];
    const int slot = atomicSub(cell_count + c, 1) - 1;
    const float4 h = load_hi(xr, i);
    xs[cell_start[c] + slot] = make_float4(h.x, h.y, h.z, __int_as_float(i));
}

// Warps per block of the warp-per-atom list kernels.
constexpr int kVerletWarps = 4;

// (squared distance, packed index) as one unsigned 64-bit sort key: d2 >= 0,
// so its IEEE bits order like its value, and the packed index is below 2^31.
__device__ __forceinline__ unsigned long long sort_key(float d2, int v)
{
    return ((unsigned long long)__float_as_uint(d2) << 32) | (unsigned)v;
}

// The list in three steps, each pair's distance tested once (the cells path):
//   k_half_cells  one block per cell gathers the 14 cells of its half shell
//                 (cell offsets after (0, 0, 0) in x-slowest order, and the
//                 cell itself for j > i) into shared memory, and a warp per
//                 atom i of the cell tests them, so that every pair within the
//                 list radius is met by exactly one of its two atoms: a quick
//                 hi-part test, the exact hi/lo test on the survivors, and
//                 each accepted pair goes into both rows unsorted at slots
//                 taken with atomics: (value, distance word, the partner
//                 entry's slot).  The rows live in the partial-force buffer,
//                 four words per slot.
//   k_sort_tile   one warp per atom ranks its row by (squared distance,
//                 value), which is unique, and writes the sorted values
//                 (slot-major nbr, through a shared tile of 32 atoms so that
//                 the stores are whole rows), the rank of every unsorted
//                 slot (vala), and into the fourth word of each partner
//                 entry the rank it got here: the partner's reverse index
//                 (k_sort_rows, a warp per atom storing nbr directly, above
//                 185 slots).
//   k_rev_tile    rev[rank of slot s][i] = the fourth word of i's slot s,
//                 within each row, 32 atoms per block transposed through
//                 shared memory into whole-row stores (k_rev_perm, a warp
//                 per atom, above 352 slots).
// The pair vector is computed once per pair in the canonical orientation, so
// the rows and the reverse index are the same as those of the full-shell
// search (the order of the unsorted slots, which the atomics decide, does
// not reach the results).  The counts are cleared by k_bin.
// What bounds the search: issue.  A warp per atom that looked up its own cells,
// prefix sums and candidate indices spent most of its instructions on those;
// per cell they are done once for ~6 to 16 atoms, and the candidates are
// contiguous reads: 105 -> 75 us for 125,000 atoms at 5 A, 92 -> 70 us for
// 64,000 of the split model at 8 A.  WARPS warps share a cell's atoms: eight
// while the cells are few (343 cells of 17 atoms: 17 us, with four 26), two for
// small cells (6.4 atoms: 75 us, with four 86, with eight 131), else four (16
// atoms: 70 us, with two 78, with eight 79).
constexpr int kHalfQuick = 96;  // survivors of the quick test waiting for the exact one, per warp
constexpr int kHalfRanges = 10;

template <int WARPS>
__device__ __forceinline__ void half_cell(int cell, int m_cap, float rv2, int cap, const float* __restrict__ xr,
                                          const float4* __restrict__ xs, const int* __restrict__ cell_start,
                                          int* __restrict__ count, int* __restrict__ rows, const Box& b)
{
    extern __shared__ __align__(16) float4 s_cand[];  // [cap]: x, y, z from the cell's corner, packed value
    __shared__ int s_sq[WARPS][kHalfQuick];
    __shared__ int s_r0[kHalfRanges], s_at[kHalfRanges + 1], s_code[kHalfRanges];
    __shared__ float s_shift[kHalfRanges][3];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = cell_start[cell], c1 = cell_start[cell + 1];
    if (c0 == c1) return;
    const int cz = cell % b.nc[2];
    const int cy = (cell / b.nc[2]) % b.nc[1];
    const int cx = cell / (b.nc[2] * b.nc[1]);
    const float ox = (float)cx * (b.Lh[0] / (float)b.nc[0]), oy = (float)cy * (b.Lh[1] / (float)b.nc[1]),
                oz = (float)cz * (b.Lh[2] / (float)b.nc[2]);
    if (warp == 0) {
        // lane r < 10: range r of candidates.  0: the cell itself; 1: the next
        // along z; 2 + 2 c + part: column c of (dx, dy) = (0, 1), (1, -1),
        // (1, 0), (1, 1), contiguous in z, part 1 what wraps across a z face
        int r0 = 0, rn = 0, sx = 0, sy = 0, sz = 0;
        if (lane < kHalfRanges) {
            int x2 = cx, y2 = cy, z0 = cz, z1 = cz;
            if (lane == 1) {
                z0 = z1 = cz + 1;
                if (z0 == b.nc[2]) {
                    z0 = z1 = 0;
                    sz = 1;
                }
            } else if (lane >= 2) {
                const int col = (lane - 2) >> 1;
                x2 += col == 0 ? 0 : 1;
                y2 += col == 0 ? 1 : col - 2;
                if (x2 >= b.nc[0]) { x2 -= b.nc[0]; sx = 1; }
                if (y2 < 0) { y2 += b.nc[1]; sy = -1; } else if (y2 >= b.nc[1]) { y2 -= b.nc[1]; sy = 1; }
                z0 = max(cz - 1, 0);
                z1 = min(cz + 1, b.nc[2] - 1);
                if (lane & 1) {
                    z1 = z0 - 1;  // nothing
                    if (cz == 0) {
                        z0 = z1 = b.nc[2] - 1;
                        sz = -1;
                    } else if (cz == b.nc[2] - 1) {
                        z0 = z1 = 0;
                        sz = 1;
                    }
                }
            }
            if (z0 <= z1) {
                const int base = (x2 * b.nc[1] + y2) * b.nc[2];
                r0 = cell_start[base + z0];
                rn = cell_start[base + z1 + 1] - r0;
            }
        }
        int incl = rn;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane < kHalfRanges) {
            s_r0[lane] = r0 - (incl - rn);  // candidate e of the concatenation is xs[e + s_r0] in its range
            s_at[lane + 1] = incl;
            s_code[lane] = image_code(sx, sy, sz) << 24;
            s_shift[lane][0] = (float)sx * b.Lh[0];  // exact: s in {-1, 0, 1}
            s_shift[lane][1] = (float)sy * b.Lh[1];
            s_shift[lane][2] = (float)sz * b.Lh[2];
        }
        if (lane == 0) s_at[0] = 0;
    }
    __syncthreads();
    const int own = s_at[1], total = s_at[kHalfRanges];
    // the hi parts alone are within half an ulp of the edge of the positions:
    // the margin never drops a pair that the exact test keeps
    const float rq = sqrtf(rv2) + 1e-3f + 1e-6f * fmaxf(b.Lh[0], fmaxf(b.Lh[1], b.Lh[2])), rq2 = rq * rq;
    int* sq = s_sq[warp];
    // a dense spot in a coarse grid can hold more candidates than the buffer
    for (int f0 = 0; f0 < total; f0 += cap) {
        if (f0) __syncthreads();  // the previous piece is read
        const int m = min(cap, total - f0);
        for (int e = threadIdx.x; e < m; e += 32 * WARPS) {
            int r = 0;
            while (s_at[r + 1] <= f0 + e) ++r;
            const float4 h = xs[s_r0[r] + f0 + e];
            s_cand[e] = make_float4((h.x - ox) + s_shift[r][0], (h.y - oy) + s_shift[r][1], (h.z - oz) + s_shift[r][2],
                                    __int_as_float(__float_as_int(h.w) | s_code[r]));
        }
        __syncthreads();
        for (int c = c0 + warp; c < c1; c += WARPS) {
            const float4 me = xs[c];
            const int i = __float_as_int(me.w);
            const float hx = me.x - ox, hy = me.y - oy, hz = me.z - oz;
            float hi[3], li[3];
            load_pos(xr, i, hi, li);
            int nq = 0;
            // the exact test of the waiting survivors; an accepted pair takes a
            // slot in i's row (one atomic per warp round) and one in j's row
            auto flush = [&]() {
                __syncwarp();
                for (int e0 = 0; e0 < nq; e0 += 32) {
                    const int e = e0 + lane;
                    bool accept = false;
                    int v = 0, j = 0;
                    float d2 = 0.f;
                    if (e < nq) {
                        v = sq[e];
                        j = v & 0xFFFFFF;
                        float hj[3], lj[3], rx, ry, rz;
                        load_pos(xr, j, hj, lj);
                        pair_vector(v >> 24, hi, li, hj, lj, b, rx, ry, rz);
                        d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
                        accept = d2 < rv2;
                    }
                    const unsigned mask = __ballot_sync(0xffffffffu, accept);
                    int si0 = 0;
                    if (lane == 0 && mask) si0 = atomicAdd(count + i, __popc(mask));
                    si0 = __shfl_sync(0xffffffffu, si0, 0);
                    if (accept) {
                        const int si = si0 + __popc(mask & ((1u << lane) - 1u));
                        const int sj = atomicAdd(count + j, 1);
                        const int vj = i | ((124 - (v >> 24)) << 24);  // the reverse image
                        // the fourth word is written by the partner's sort
                        if (si < m_cap) {
                            int* ri = rows + ((size_t)i * m_cap + si) * 4;
                            *reinterpret_cast<int2*>(ri) = make_int2(v, (int)__float_as_uint(d2));
                            ri[2] = sj;
                        }
                        if (sj < m_cap) {
                            int* rj = rows + ((size_t)j * m_cap + sj) * 4;
                            *reinterpret_cast<int2*>(rj) = make_int2(vj, (int)__float_as_uint(d2));
                            rj[2] = si;
                        }
                    }
                }
                nq = 0;
                __syncwarp();
            };
#pragma unroll 2
            for (int e0 = 0; e0 < m; e0 += 32) {
                const int e = e0 + lane;
                bool pass = false;
                int v = 0;
                if (e < m) {
                    const float4 q = s_cand[e];
                    const float qx = q.x - hx, qy = q.y - hy, qz = q.z - hz;
                    v = __float_as_int(q.w);
                    // the cell itself: the pairs with j > i only
                    pass = fmaf(qx, qx, fmaf(qy, qy, qz * qz)) < rq2 && (f0 + e >= own || (v & 0xFFFFFF) > i);
                }
                const unsigned mask = __ballot_sync(0xffffffffu, pass);
                const int pos = nq + __popc(mask & ((1u << lane) - 1u));
                if (pass) sq[pos] = v;
                nq += __popc(mask);
                if (nq > kHalfQuick - 32) flush();
            }
            flush();
        }
    }
}

// A block per cell, or with a gate a few blocks per SM that walk the cells: a
// launch whose gate is off then retires in 5 us instead of 13 (125,000 atoms).
// (One form for both spilled registers.)
// ATOMS: a block (or a turn of the walk) per atom in cell order, of which the
// first of a cell takes the cell: for sparse grids, where nearly every block of the
// other form found an empty cell.  50,000 atoms, whole call, by cells -> by atoms:
// 1.5 atoms per cell 159 -> 169 us, 0.91 157 -> 162, 0.59 159 -> 158, 0.23 204 ->
// 153, 0.03 995 -> 175; 1,000,000 atoms, 0.75 per cell 2467 -> 2503.  The line lies
// at half an atom per cell.
template <int WARPS, bool GATED, bool ATOMS>
__global__ void __launch_bounds__(32 * WARPS) k_half_cells(int items, int m_cap, float rv2, int cap,
                                                          const float* xr,
                                                          const float4* xs, const int* atom_cell,
                                                          const int* cell_start,
                                                          int* count, int* rows, Box b,
                                                          const unsigned* gate)
{
    const int block = block_after();
    auto take = [&](int t) {
        int cell = t;
        if constexpr (ATOMS) {
            cell = atom_cell[__float_as_int(xs[t].w)];
            if (cell_start[cell] != t) return;
        }
        half_cell<WARPS>(cell, m_cap, rv2, cap, xr, xs, cell_start, count, rows, b);
    };
    if constexpr (!GATED) {
        take(block);
    } else {
        if (gated_off(gate)) return;
        for (int t = block; t < items; t += gridDim.x) {
            if (t != block) __syncthreads();  // the previous cell's tables are read
            take(t);
        }
    }
}

// Ranks a warp's row entries c0 + lane + 32 t against all ns (keys in sk)
// and writes each at its rank: the value to out[rank * out_stride] (the
// atom's column of the slot-major nbr, or of a shared-memory tile), the rank
// to inv[i][unsorted slot] and to the fourth word of the partner entry (the
// partner's reverse index; j's slot sp[e] of the atom in the value).
template <int EPL>
__device__ __forceinline__ void rank_rows_write(int c0, int ns, int lane, const unsigned long long* sk,
                                                const int* sp, int i, int out_stride, int m_cap, int* out,
                                                int* __restrict__ rows, int* __restrict__ inv)
{
    unsigned long long ke[EPL];
    int rk[EPL];
#pragma unroll
    for (int t = 0; t < EPL; ++t) {
        const int e = c0 + lane + 32 * t;
        ke[t] = e < ns ? sk[e] : ~0ull;
        rk[t] = 0;
    }
    // by the distance words alone; equal distances (the ranks then miss some
    // value, and their sum is short) are ranked again by the whole keys
    const unsigned* hi = reinterpret_cast<const unsigned*>(sk) + 1;
    int sum = 0;
#pragma unroll 4
    for (int f = 0; f < ns; ++f) {
        const unsigned kf = hi[2 * f];
#pragma unroll
        for (int t = 0; t < EPL; ++t) rk[t] += (unsigned)(ke[t] >> 32) > kf ? 1 : 0;
    }
#pragma unroll
    for (int t = 0; t < EPL; ++t) sum += c0 + lane + 32 * t < ns ? rk[t] : 0;
    if (ns > 32 * EPL || __reduce_add_sync(0xffffffffu, sum) != ns * (ns - 1) / 2) {
#pragma unroll
        for (int t = 0; t < EPL; ++t) rk[t] = 0;
        for (int f = 0; f < ns; ++f) {
            const unsigned long long kf = sk[f];
#pragma unroll
            for (int t = 0; t < EPL; ++t) rk[t] += ke[t] > kf ? 1 : 0;
        }
    }
#pragma unroll
    for (int t = 0; t < EPL; ++t) {
        const int e = c0 + lane + 32 * t;
        if (e < ns) {
            const int v = (int)(unsigned)ke[t];
            inv[(size_t)i * m_cap + e] = rk[t];
            out[(size_t)rk[t] * out_stride] = v;
            const int ps = sp[e];
            if (ps < m_cap) rows[((size_t)(v & 0xFFFFFF) * m_cap + ps) * 4 + 3] = rk[t];
        }
    }
}

__global__ void __launch_bounds__(32 * kVerletWarps) k_sort_rows(int n, int m_cap, int lcap, int* rows,
                                                                const int* count, int* nbr,
                                                                int* inv, unsigned* err,
                                                                const unsigned* gate)
{
    const int block = block_after();
    if (gated_off(gate)) return;
    extern __shared__ unsigned long long s_sort[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long* sk = s_sort + (size_t)warp * lcap * 3 / 2;  // lcap keys, then lcap partner slots
    int* sp = reinterpret_cast<int*>(sk + lcap);
    // a lane's entries of the next atom's row (e = lane + 32 t), loaded while
    // the current row is sorted
    constexpr int kPre = 4;  // 128 entries per row at most
    int4 pre[kPre];
    int pre_cnt = 0;
    const int stride = gridDim.x * kVerletWarps;
    auto fetch = [&](int a) {
        pre_cnt = a < n ? count[a] : 0;
        const int ns_a = min(min(pre_cnt, m_cap), lcap);
#pragma unroll
        for (int t = 0; t < kPre; ++t) {
            const int e = lane + 32 * t;
            if (e < ns_a) pre[t] = *reinterpret_cast<const int4*>(rows + ((size_t)a * m_cap + e) * 4);
        }
    };
    fetch(block * kVerletWarps + warp);
    for (int i = block * kVerletWarps + warp; i < n; i += stride) {
        const int cnt = pre_cnt;
        if (cnt > m_cap && lane == 0) atomicOr(err, kErrOverflow);
        const int m = cnt < m_cap ? cnt : m_cap;
        const int ns = m < lcap ? m : lcap;
#pragma unroll
        for (int t = 0; t < kPre; ++t) {
            const int e = lane + 32 * t;
            if (e < ns) {
                sk[e] = sort_key(__int_as_float(pre[t].y), pre[t].x);
                sp[e] = pre[t].z;
            }
        }
        for (int e = 32 * kPre + lane; e < ns; e += 32) {  // rows longer than the prefetch (m_cap > 128)
            const int4 r = *reinterpret_cast<const int4*>(rows + ((size_t)i * m_cap + e) * 4);
            sk[e] = sort_key(__int_as_float(r.y), r.x);
            sp[e] = r.z;
        }
        __syncwarp();
        fetch(i + stride);
        if (ns <= 32)
            rank_rows_write<1>(0, ns, lane, sk, sp, i, n, m_cap, nbr + i, rows, inv);
        else if (ns <= 64)
            rank_rows_write<2>(0, ns, lane, sk, sp, i, n, m_cap, nbr + i, rows, inv);
        else
            for (int c0 = 0; c0 < ns; c0 += 128)
                rank_rows_write<4>(c0, ns, lane, sk, sp, i, n, m_cap, nbr + i, rows, inv);
        __syncwarp();
    }
}

// The same sort with the slot-major nbr stores made whole: a block of
// kSortWarps warps takes tiles of 32 consecutive atoms in turn, warp w the
// atoms w, w + 8, w + 16, w + 24 of each (the next one's row loaded into
// registers while the current one sorts); the sorted values go to a shared
// tile (atom a's column), stored after the block barrier as rows of 32
// consecutive atoms (one 128-byte store each).  inv and the partner words are
// written as in k_sort_rows, which takes longer rows.  Shared memory: the warps' key buffers (lcap x
// 12 bytes each), then the m_cap x 33-int tile.
constexpr int kSortWarps = 8;
constexpr int kSortAtoms = 32;
constexpr int kSortGridCap = 152 * 8;
// the default 48 KB hold the kernel's counts too: up to 185 slots per atom
constexpr size_t kSortTileMaxSmem = 48 * 1024 - sizeof(int) * kSortAtoms;

__global__ void __launch_bounds__(32 * kSortWarps) k_sort_tile(int n, int m_cap, int lcap, int* rows,
                                                              const int* count, int* nbr,
                                                              int* inv, unsigned* err,
                                                              const unsigned* gate)
{
    const int block = block_after();
    if (gated_off(gate)) return;
    extern __shared__ unsigned long long s_sort[];
    __shared__ int s_cnt[kSortAtoms];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long* sk = s_sort + (size_t)warp * lcap * 3 / 2;  // lcap keys, then lcap partner slots
    int* sp = reinterpret_cast<int*>(sk + lcap);
    int* s_tile = reinterpret_cast<int*>(s_sort + (size_t)kSortWarps * lcap * 3 / 2);  // [m_cap][33]
    constexpr int kPer = kSortAtoms / kSortWarps;  // atoms per warp and tile
    const int tiles = (n + kSortAtoms - 1) / kSortAtoms;
    // this warp's k-th atom: tile block + (k / kPer) gridDim.x, column warp + kSortWarps (k % kPer)
    auto atom_of = [&](int k, int& tile, int& a) {
        tile = block + (k / kPer) * gridDim.x;
        a = warp + kSortWarps * (k % kPer);
        return tile * kSortAtoms + a;
    };
    constexpr int kPre = 4;  // 128 entries per row at most
    int4 pre[kPre];
    int pre_cnt = 0;
    auto fetch = [&](int k) {
        int tile, a;
        const int at = atom_of(k, tile, a);
        pre_cnt = tile < tiles && at < n ? count[at] : 0;
        const int ns_a = min(min(pre_cnt, m_cap), lcap);
#pragma unroll
        for (int t = 0; t < kPre; ++t) {
            const int e = lane + 32 * t;
            if (e < ns_a) pre[t] = *reinterpret_cast<const int4*>(rows + ((size_t)at * m_cap + e) * 4);
        }
    };
    fetch(0);
    for (int k = 0;; ++k) {
        int tile, a;
        const int i = atom_of(k, tile, a);
        if (tile >= tiles) break;
        const int cnt = pre_cnt;  // 0 past the last atom
        if (cnt > m_cap && lane == 0) atomicOr(err, kErrOverflow);
        const int m = cnt < m_cap ? cnt : m_cap;
        const int ns = m < lcap ? m : lcap;
        if (lane == 0) s_cnt[a] = ns;
#pragma unroll
        for (int t = 0; t < kPre; ++t) {
            const int e = lane + 32 * t;
            if (e < ns) {
                sk[e] = sort_key(__int_as_float(pre[t].y), pre[t].x);
                sp[e] = pre[t].z;
            }
        }
        for (int e = 32 * kPre + lane; e < ns; e += 32) {  // rows longer than the prefetch (m_cap > 128)
            const int4 r = *reinterpret_cast<const int4*>(rows + ((size_t)i * m_cap + e) * 4);
            sk[e] = sort_key(__int_as_float(r.y), r.x);
            sp[e] = r.z;
        }
        __syncwarp();
        fetch(k + 1);
        int* col = s_tile + a;
        if (ns == 0) {
        } else if (ns <= 32)
            rank_rows_write<1>(0, ns, lane, sk, sp, i, kSortAtoms + 1, m_cap, col, rows, inv);
        else if (ns <= 64)
            rank_rows_write<2>(0, ns, lane, sk, sp, i, kSortAtoms + 1, m_cap, col, rows, inv);
        else
            for (int c0 = 0; c0 < ns; c0 += 128)
                rank_rows_write<4>(c0, ns, lane, sk, sp, i, kSortAtoms + 1, m_cap, col, rows, inv);
        __syncwarp();
        if (k % kPer == kPer - 1) {
            // the tile is complete: its rows to nbr, 32 consecutive atoms each
            __syncthreads();
            const int i0 = tile * kSortAtoms;
            const int ca = s_cnt[lane];
            for (int r = warp; r < m_cap; r += kSortWarps)
                if (r < ca) nbr[(size_t)r * n + i0 + lane] = s_tile[r * (kSortAtoms + 1) + lane];
            __syncthreads();  // the tile and the counts are read before the next tile writes them
        }
    }
}

// rev[inv[i][s]][i] = the reverse index left in the fourth word of i's
// unsorted slot s by the partner's sort; one warp per atom.  A value outside
// the partner's kept entries (only after an overflow, already latched) is
// latched again and replaced by the slot's own rank.
__global__ void k_rev_perm(int n, int m_cap, const int* count, const int* rows,
                           const int* inv, int* rev, unsigned* err, const unsigned* gate)
{
    const int block = block_after();
    if (gated_off(gate)) return;
    const int lane = threadIdx.x & 31;
    const int warps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int i = (int)(((size_t)block * blockDim.x + threadIdx.x) >> 5); i < n; i += warps) {
        const int ci = min(count[i], m_cap);
        for (int s = lane; s < ci; s += 32) {
            const int r = inv[(size_t)i * m_cap + s];
            int v = rows[((size_t)i * m_cap + s) * 4 + 3];
            if (v < 0 || v >= m_cap) {
                atomicOr(err, kErrReverse);
                v = r;
            }
            rev[(size_t)r * n + i] = v;
        }
    }
}

// The same reverse index with the slot-major stores made whole: a block of
// eight warps takes tiles of 32 consecutive atoms in turn; each warp fills the shared tile
// columns of its atoms (rev value of sorted slot r of atom a at tile[r][a],
// reading the rows as k_rev_perm does), then each warp stores tile rows, 32
// consecutive atoms per 128-byte store.  Slots at or past an atom's count are
// not stored.  Shared memory: m_cap x 33 ints.
constexpr int kRevAtoms = 32;
constexpr int kRevThreads = 256;
constexpr int kRevTileMaxSlots = 352;  // 352 x 33 x 4 bytes stay under 48 KB
constexpr int kRevGridCap = 152 * 8;   // blocks walk the 32-atom tiles; a gated-off launch retires fast

__global__ void __launch_bounds__(kRevThreads) k_rev_tile(int n, int m_cap, const int* count,
                                                          const int* rows, const int* inv,
                                                          int* rev, unsigned* err, const unsigned* gate)
{
    const int block = block_after();
    if (gated_off(gate)) return;
    extern __shared__ int s_tile[];  // [m_cap][kRevAtoms + 1]
    __shared__ int s_cnt[kRevAtoms];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles = (n + kRevAtoms - 1) / kRevAtoms;
    for (int tile = block; tile < tiles; tile += gridDim.x) {
        const int i0 = tile * kRevAtoms;
        if (threadIdx.x < kRevAtoms) {
            const int i = i0 + threadIdx.x;
            s_cnt[threadIdx.x] = i < n ? min(count[i], m_cap) : 0;
        }
        __syncthreads();
        for (int a = warp; a < kRevAtoms; a += kRevThreads / 32) {
            const int i = i0 + a, ci = s_cnt[a];
            for (int s = lane; s < ci; s += 32) {
                const int r = inv[(size_t)i * m_cap + s];
                int v = rows[((size_t)i * m_cap + s) * 4 + 3];
                if (v < 0 || v >= m_cap) {
                    atomicOr(err, kErrReverse);
                    v = r;
                }
                if (r >= 0 && r < ci)
                    s_tile[r * (kRevAtoms + 1) + a] = v;
                else
                    atomicOr(err, kErrReverse);
            }
        }
        __syncthreads();
        const int ca = s_cnt[lane];
        for (int r = warp; r < m_cap; r += kRevThreads / 32)
            if (r < ca) rev[(size_t)r * n + i0 + lane] = s_tile[r * (kRevAtoms + 1) + lane];
        __syncthreads();  // the tile and the counts are read before the next tile writes them
    }
}

// The list by testing every atom, for boxes too small for a cell grid (all
// images) and for small atom counts (the nearest image): one launch instead of
// the cells path's scan, scatter, search and sort, each a few microseconds of
// latency.  A block takes two consecutive atoms; its threads walk all atoms j,
// test the hi parts against both (with a margin, as k_half_cells), test survivors exactly and
// append (squared distance, tie-break) keys to the atoms' shared rows.  The
// rows are then rank-sorted, 64 threads per row.
// IMAGES: every shift up to b.img, ties ordered by (j, image); else the
// nearest image (unique: the edges are at least three list radii), ties
// ordered by the packed value, as the cells path orders them.
// A cell of 96 atoms: 400 -> 8 us against one thread per atom with an insertion
// sort in global memory.  Eight atoms per block instead of two: 18 us there,
// 14.8 against 7.6 us for 1728 atoms.
constexpr int kDirectThreads = 128;
constexpr int kDirectAtoms = 2;

template <bool IMAGES>
__global__ void __launch_bounds__(kDirectThreads) k_list_direct(int n, int m_cap, float rv2,
                                                               const float* xr, int* count,
                                                               int* nbr, float* key,
                                                               int* vala, unsigned* err, Box b,
                                                               const unsigned* gate)
{
    const int block = block_after();
    if (gated_off(gate)) return;
    constexpr int AT = kDirectAtoms;
    extern __shared__ unsigned long long s_rows[];  // [AT][m_cap]
    __shared__ int s_cnt[AT];
    constexpr int PER = kDirectThreads / AT;  // threads that sort one row
    const int i0 = block * AT;
    if (threadIdx.x < AT) s_cnt[threadIdx.x] = 0;
    float hi[AT][3];
#pragma unroll
    for (int a = 0; a < AT; ++a) {
        const float4 h = load_hi(xr, min(i0 + a, n - 1));
        hi[a][0] = h.x;
        hi[a][1] = h.y;
        hi[a][2] = h.z;
    }
    __syncthreads();
    const float rq = sqrtf(rv2) + 1e-3f + 1e-6f * fmaxf(b.Lh[0], fmaxf(b.Lh[1], b.Lh[2])), rq2 = rq * rq;
    // the exact test of a survivor, and its key
    auto exact = [&](int a, int j, int code) {
        float h0[3], l0[3], hj[3], lj[3], rx, ry, rz;
        load_pos(xr, i0 + a, h0, l0);
        load_pos(xr, j, hj, lj);
        pair_vector(code, h0, l0, hj, lj, b, rx, ry, rz);
        const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
        if (!(d2 < rv2)) return;
        const int at = atomicAdd(s_cnt + a, 1);
        if (at < m_cap) s_rows[a * m_cap + at] = sort_key(d2, IMAGES ? (j << 7) | code : j | (code << 24));
    };
    if (IMAGES) {
        for (int sx = -b.img[0]; sx <= b.img[0]; ++sx)
            for (int sy = -b.img[1]; sy <= b.img[1]; ++sy)
                for (int sz = -b.img[2]; sz <= b.img[2]; ++sz) {
                    const int code = image_code(sx, sy, sz);
                    const float tx = (float)sx * b.Lh[0], ty = (float)sy * b.Lh[1], tz = (float)sz * b.Lh[2];
                    for (int j = threadIdx.x; j < n; j += kDirectThreads) {
                        const float4 h = load_hi(xr, j);
#pragma unroll
                        for (int a = 0; a < AT; ++a) {
                            const float qx = (h.x - hi[a][0]) + tx, qy = (h.y - hi[a][1]) + ty,
                                        qz = (h.z - hi[a][2]) + tz;
                            if (fmaf(qx, qx, fmaf(qy, qy, qz * qz)) < rq2 && i0 + a < n &&
                                !(j == i0 + a && code == kImgCenter))
                                exact(a, j, code);
                        }
                    }
                }
    } else {
        const float hx = 0.5f * b.Lh[0], hy = 0.5f * b.Lh[1], hz = 0.5f * b.Lh[2];
        // shift of the nearest image of a difference d (0 but across a face)
        auto nearest = [](float d, float half, float L, float& s) {
            s = d > half ? -1.f : d < -half ? 1.f : 0.f;
            return fmaf(s, L, d);
        };
        for (int j = threadIdx.x; j < n; j += kDirectThreads) {
            const float4 h = load_hi(xr, j);
#pragma unroll
            for (int a = 0; a < AT; ++a) {
                float sx, sy, sz;
                const float qx = nearest(h.x - hi[a][0], hx, b.Lh[0], sx);
                const float qy = nearest(h.y - hi[a][1], hy, b.Lh[1], sy);
                const float qz = nearest(h.z - hi[a][2], hz, b.Lh[2], sz);
                if (fmaf(qx, qx, fmaf(qy, qy, qz * qz)) < rq2 && i0 + a < n && j != i0 + a)
                    exact(a, j, image_code((int)sx, (int)sy, (int)sz));
            }
        }
    }
    __syncthreads();
    const int a = threadIdx.x / PER, t0 = threadIdx.x % PER, i = i0 + a;
    if (i >= n) return;
    const int cnt = s_cnt[a];
    if (t0 == 0) {
        count[i] = cnt;
        if (cnt > m_cap) atomicOr(err, kErrOverflow);
    }
    const int ns = min(cnt, m_cap);
    const unsigned long long* row = s_rows + a * m_cap;
    for (int e = t0; e < ns; e += PER) {
        const unsigned long long k = row[e];
        int rank = 0;
#pragma unroll 4
        for (int f = 0; f < ns; ++f) rank += k > row[f] ? 1 : 0;
        const unsigned low = (unsigned)k;
        const int v = IMAGES ? (int)((low >> 7) | ((low & 127u) << 24)) : (int)low;
        nbr[(size_t)rank * n + i] = v;
        vala[(size_t)i * m_cap + rank] = v;
        key[(size_t)i * m_cap + rank] = __uint_as_float((unsigned)(k >> 32));
    }
}

// rev[k][i] = slot of (i, -image) in j's list.  The pair vectors are exactly
// antisymmetric, so both directions carry the same squared distance and j's
// list (sorted by it) is binary-searched; a miss (only possible after an
// overflow) is latched as an error.  One warp per atom, a lane per slot; the
// keys and values are read from their atom-major copies, so every search
// stays inside one atom's contiguous row.
__global__ void k_reverse(int n, int m_cap, const int* count, const float* key,
                          const int* vala, int* rev, unsigned* err, const unsigned* gate)
{
    const int block = block_after();
    if (gated_off(gate)) return;
    const int lane = threadIdx.x & 31;
    const int warps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int i = (int)(((size_t)block * blockDim.x + threadIdx.x) >> 5); i < n; i += warps) {
        const int ci = min(count[i], m_cap);
        for (int k = lane; k < ci; k += 32) {
            const int v = vala[(size_t)i * m_cap + k];
            const int j = v & 0xFFFFFF;
            const int target = i | ((124 - (v >> 24)) << 24);
            const float kd = key[(size_t)i * m_cap + k];
            const int cj = min(count[j], m_cap);
            const float* kj = key + (size_t)j * m_cap;  // j's keys, contiguous
            int lo = 0, hi = cj;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (kj[mid] < kd)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            int found = -1;
            for (int t = lo; t < cj && kj[t] == kd; ++t)
                if (vala[(size_t)j * m_cap + t] == target) {
                    found = t;
                    break;
                }
            if (found < 0) {
                atomicOr(err, kErrReverse);
                found = k;  // keeps later reads in bounds
            }
            rev[(size_t)k * n + i] = found;
        }
    }
}

inline int blocks_for(int n, int t) { return (n + t - 1) / t; }

// grid of the warp-per-atom list kernels: 152 SMs x 16 blocks of 4 warps
// keep every SM full, and a launch whose gate is off retires in microseconds
constexpr int kListGridCap = 152 * 16;

}  // namespace

// Largest atom count of the direct list in a box with a cell grid.  The whole
// list build, cells path -> direct: 512 atoms 24.0 -> 12.0 us, 1728 25.2 ->
// 15.6, 4096 26.5 -> 35.8; split model 1728 43 -> 24, 5832 50 -> 71 (and three
// launches instead of six).
constexpr int kDirectMax = 2500;

bool list_is_direct(int n) { return n <= kDirectMax; }

int build_neighbor_list(NeighborList& nl, const Box& b, int n, double* pos, const float* zatom, bool wrap_in_place,
                        double* x_ref,
                        float r_list, unsigned* d_err, const unsigned* d_gate, cudaStream_t st)
{
    const int T = 256;
    const float rv2 = r_list * r_list;
    const bool grid_box = b.nc[0] > 0;
    const bool cells = grid_box && n > kDirectMax;
    const int ncell = cells ? b.nc[0] * b.nc[1] * b.nc[2] : 0;
    Box bb = b;
    if (!cells) bb.nc[0] = 0;  // no cell counts
    k_bin<<<blocks_for(n, T), T, 0, st>>>(n, pos, zatom, wrap_in_place ? 1 : 0, x_ref, nl.xr, nl.atom_cell,
                                          nl.cell_count, nl.count, bb, d_gate, d_err);
    if (cells) {
        const int rounds = blocks_for(blocks_for(ncell, kScanRound), 152), slice = rounds * kScanRound;
        launch_after(true, k_scan, blocks_for(ncell, slice), kScanThreads, 0, st, ncell, slice, nl.cell_count,
                     nl.cell_start, d_gate);
        launch_after(true, k_scatter, blocks_for(n, T), T, 0, st, n, nl.atom_cell, nl.cell_start, nl.cell_count, nl.xr,
                     nl.xs, d_gate);
        // per-warp buffers of the row sort: a power of two >= m_cap entries
        int lcap = 32;
        while (lcap < nl.m_cap) lcap <<= 1;
        const int grid = std::min(blocks_for(n, kVerletWarps), kListGridCap);
        int* rows = reinterpret_cast<int*>(nl.pf);  // four words per slot, free until the site pass
        // candidates per cell: 14 mean cells and half as many again
        const int cap = std::min(std::max(128, (int)(1.5 * 14.0 * n / ncell) / 32 * 32), 1024);
        const int warps = ncell <= 608 ? 8 : n < 8 * (long long)ncell ? 2 : 4;
        const bool sparse = 2LL * n < ncell;
        const int items = sparse ? n : ncell;
        auto half = sparse       ? (d_gate ? k_half_cells<2, true, true> : k_half_cells<2, false, true>)
                    : warps == 8 ? (d_gate ? k_half_cells<8, true, false> : k_half_cells<8, false, false>)
                    : warps == 2 ? (d_gate ? k_half_cells<2, true, false> : k_half_cells<2, false, false>)
                                 : (d_gate ? k_half_cells<4, true, false> : k_half_cells<4, false, false>);
        launch_after(true, half, d_gate ? std::min(items, kListGridCap) : items, 32 * warps,
                     (size_t)cap * sizeof(float4), st, items, nl.m_cap, rv2, cap, nl.xr, nl.xs, nl.atom_cell,
                     nl.cell_start, nl.count, rows, b, d_gate);
        const size_t sort_smem = (size_t)kSortWarps * lcap * 12 + (size_t)nl.m_cap * (kSortAtoms + 1) * sizeof(int);
        if (sort_smem <= kSortTileMaxSmem)
            launch_after(true, k_sort_tile, std::min(blocks_for(n, kSortAtoms), kSortGridCap), 32 * kSortWarps,
                         sort_smem, st, n, nl.m_cap, lcap, rows, nl.count, nl.nbr, nl.vala, d_err, d_gate);
        else
            launch_after(true, k_sort_rows, grid, 32 * kVerletWarps, (size_t)kVerletWarps * lcap * 12, st, n, nl.m_cap,
                         lcap, rows, nl.count, nl.nbr, nl.vala, d_err, d_gate);
        if (nl.m_cap <= kRevTileMaxSlots)
            launch_after(true, k_rev_tile, std::min(blocks_for(n, kRevAtoms), kRevGridCap), kRevThreads,
                         (size_t)nl.m_cap * (kRevAtoms + 1) * sizeof(int), st, n, nl.m_cap, nl.count, rows, nl.vala,
                         nl.rev, d_err, d_gate);
        else
            launch_after(true, k_rev_perm, std::min(blocks_for(n, 4), kListGridCap), 128, 0, st, n, nl.m_cap, nl.count,
                         rows, nl.vala, nl.rev, d_err, d_gate);
        return cuda_fail(cudaGetLastError(), "neighbour-list kernels");
    }
    const size_t rows_bytes = (size_t)kDirectAtoms * nl.m_cap * sizeof(unsigned long long);
    launch_after(true, grid_box ? k_list_direct<false> : k_list_direct<true>, blocks_for(n, kDirectAtoms),
                 kDirectThreads, rows_bytes, st, n, nl.m_cap, rv2, nl.xr, nl.count, nl.nbr, nl.pf, nl.vala, d_err, b,
                 d_gate);
    launch_after(true, k_reverse, std::min(blocks_for(n, 4), kListGridCap), 128, 0, st, n, nl.m_cap, nl.count, nl.pf,
                 nl.vala, nl.rev, d_err, d_gate);
    return cuda_fail(cudaGetLastError(), "neighbour-list kernels");
}

}  // namespace nep
