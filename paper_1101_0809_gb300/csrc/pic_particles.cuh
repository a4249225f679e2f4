// pic_particles.cuh -- per-particle kernels of the charge-conserving PIC step
// (Sokolov, arXiv:1101.0809, Appendix step 2): alternating-order gather, push,
// move and virtual-path deposit, run over tile-sorted particles.
//
// One thread block takes one work item: a contiguous range of particles that
// the last sort put in one tile.  The block stages E and B of the tile plus a
// halo of (halo + 1) cells in shared memory, and a current tile with a halo of
// (halo + 2) cells.  Each thread streams particles (coalesced SoA loads),
// gathers from shared memory, pushes, renormalizes offset and cell, writes the
// particle back and scatters its face currents into the shared current tile
// with shared-memory atomics: 54 (3D) or 21 (2D) for a particle that kept its
// cell, at once; up to 144 or 40 for one that changed cell, through its warp's
// queue, drained 32 particles at a time.  A particle that has drifted
// more than `halo` cells outside the tile since the last sort takes the same
// arithmetic on the global arrays instead (periodic indices, global atomics);
// an item that had such particles stages the tile where its particles are now
// (item_shift).
// At the end the block adds its current tile to the global J with atomics.
#pragma once

#include <cooperative_groups.h>

#include <algorithm>

#include "pic_internal.h"

namespace cg = cooperative_groups;

namespace pic {

template <typename R>
struct PartArgs {
    WorkItem *items;   // (`drifted` is written by the fused step)
    const int *n_items;
    const RunDev *runs;
    const GroupDev *groups;
    Pool<R> P;
    // MODE 0 right after a sort: the particles are read from S, particle p of
    // the new order at S[perm[p]], and written to P; otherwise S = P, perm null
    Pool<R> S;
    const unsigned *perm;
    Fields<R> F;
    int *old_cell;
    R *old_off[3];
    int qcap;             // entries of a warp's deposit queue in 3D FP64 (else kQueueCap)
    unsigned *far_list;   // pool-sized scratch: particles past their item's staged tile (process_item)
    int halo;
    int *err;   // err[0]: error word; err[1]: particles that ran past their tile's halo (counted by MODES 0, 1)
};

extern __shared__ __align__(16) unsigned char g_smem[];

// Per-warp deposit queue of particles that changed cell: capacity (a warp adds
// at most 32 entries to fewer than 32) and the values kept per entry (old and
// new offsets, u_z in 2D) besides one packed int (tile base << 8 | shifts + 1).
constexpr int kQueueCap = 64;
constexpr int kQueueVals = 7;
// 3D FP64: room for both kinds of particles that moved, fewer than 32 of each and 32 new
constexpr int kQueueCap3 = 96;

// Blocks per SM the kernels are compiled for: two (128 registers); three of the 2D
// FP32 fused step (80); four of the 2D FP32 split calls (64), whose 512 items of
// 256x256 cells and 16 + 16 particles then run at once (the push 40 us, 47 at three;
// the deposit 55 us, 64 at three and 61 at five).  Where the shared tiles leave room
// for one block only, the launches take the variant compiled for one.  In FP32 that
// has 512 threads, to have as many warps as two blocks would (61x47x53 cells in
// 8x8x8 tiles, 12 + 12 particles each, 20 steps: 6.3 ms, 7.7 with 256 threads).  In
// FP64 it has 256 threads and registers for everything; at 128 the l_a = 2 1/2
// deposit spills 148 bytes per thread, the l_a = 1 1/2 step 4.
template <int DIM, typename R, int MODE>
constexpr int min_blocks()
{
    return DIM == 2 && sizeof(R) == 4 ? (MODE == 0 ? 3 : 4) : 2;
}
// ... of the persistent step: the compiled geometries as the fused step (24 runs, 30
// steps: 18.1 ms, 19.5 at two), tiles read at run time at two (384x384 cells of 16 + 16
// particles, 10 steps: 12x12 tiles 1.75 ms, 1.79 at three; 24x24 1.83, 2.11 at three).
template <int DIM, typename R, bool DYN>
constexpr int min_blocks_persistent()
{
    return DYN ? 2 : min_blocks<DIM, R, 0>();
}
template <typename R, bool ONE>
constexpr int block_threads()
{
    return ONE && sizeof(R) == 4 ? 512 : kThreads;
}
// The shared memory of an SM, and what the system keeps of it per block.
inline bool one_block_per_sm(size_t smem) { return 2 * (smem + 1024) > 228 * 1024; }
inline int blocks_per_sm(size_t smem) { return (int)(228 * 1024 / (smem + 1024)); }
// The shared memory of a block of nt threads, given that of kThreads: more warps'
// deposit queues and counts.
template <typename R>
constexpr size_t queue_bytes(int nt)
{
    return (size_t)(nt / 32) * (kQueueCap * (kQueueVals * sizeof(R) + sizeof(int)) + sizeof(int));
}
template <typename R, int MODE>
constexpr size_t smem_of(size_t smem, int nt)
{
    return MODE == 1 ? smem : smem + queue_bytes<R>(nt) - queue_bytes<R>(kThreads);
}
// What the larger queues of 3D FP64 take more; the launches take them where they
// neither cost a block per SM nor pass the limit.
template <typename R>
constexpr size_t queue3_bytes(int nt)
{
    return (size_t)(nt / 32) * ((kQueueCap3 - kQueueCap) * (kQueueVals * sizeof(R) + sizeof(int)) + sizeof(int));
}
constexpr size_t kSmemMax = 227 * 1024 - 16;   // less MODE 1's static word

// Tile geometry of the particle kernels: extents T0 x T1 x T2, halo G and the
// shared tiles' x and y pitches P0, P1.  GeoDyn reads them from the run and the
// launch; a GeoFix kernel has them as constants, so that every shared-memory
// offset of the gather and the deposit is an immediate.  The host launches a
// GeoFix kernel only when the grid's geometry equals it (pic_particles_fixed.cu).
struct GeoDyn {
    static constexpr bool dyn = true;
    static constexpr int T0 = 0, T1 = 0, T2 = 0, G = 0, P0 = 0, P1 = 0;
};
template <int t0, int t1, int t2, int g, int p0, int p1>
struct GeoFix {
    static constexpr bool dyn = false;
    static constexpr int T0 = t0, T1 = t1, T2 = t2, G = g, P0 = p0, P1 = p1;
};

__device__ __forceinline__ bool finite3(float a, float b, float c) { return isfinite(a) && isfinite(b) && isfinite(c); }
__device__ __forceinline__ bool finite3(double a, double b, double c) { return isfinite(a) && isfinite(b) && isfinite(c); }

// Tile-local coordinate of global index i for a tile starting at o with extent T:
// the periodic image in [-G, T+G) if there is one (the grid is wider than the
// staged region, so at most one image lies there), else a value outside it.
__device__ __forceinline__ int local_coord(int i, int o, int T, int G, int n)
{
    int l = i - o;
    if (l >= T + G) l -= n;
    if (l < -G) l += n;
    return l;
}

// Where the particles of a drifted item are now: the mean displacement of
// (up to) NT (threads) of them, evenly spaced over the item, from the centre of its
// tile, in whole cells.  The item then stages the tile moved by that much.  Any
// shift gives the same step; it only decides which particles find their stencil
// in shared memory.  A plasma that streams or is pushed by a laser carries a
// tile's particles along together.  One cell per thread is read, and only by items
// that had one in 256 of their particles (summed over the steps since the sort) on
// the global-memory path: ten steps of a slab behind a wave of a0 = 5, in 4x4x4 tiles
// of halo 2 and unsorted, take 14.7 ms, 16.7 with one in 8 and 22.4 with the tile
// staged where it was sorted; a thermal plasma's few (8x8x8 tiles, sort every 10
// steps) cost the same with each.
template <int DIM, typename R, bool OLD, int NT>
__device__ __forceinline__ void item_shift(const PartArgs<R> &a, const WorkItem &it, const RunDev &rn, const int T[3],
                                           int o[3])
{
    int *const sum = reinterpret_cast<int *>(g_smem);   // four words, before the tiles are staged
    if (threadIdx.x < 4) sum[threadIdx.x] = 0;
    __syncthreads();
    const long long len = it.end - it.begin;
    int d[4] = {0, 0, 0, 0};
    if (threadIdx.x < len) {
        const long long p = it.begin + (len <= NT ? threadIdx.x : len * threadIdx.x / NT);
        const int cell = OLD ? a.old_cell[p] : a.P.cell[p];
        const int at = OLD && cell < 0 ? 0 : cell;   // < 0: none was saved
        const int rest = divu31(at, rn.div_nx);
        const int k = DIM == 3 ? divu31(rest, rn.div_ny) : 0;
        const int c[3] = {at - rest * rn.n[0], rest - k * rn.n[1], k};
#pragma unroll
        for (int x = 0; x < DIM; ++x) {
            if (OLD && cell < 0) break;
            d[x] = 2 * (c[x] - o[x]) - (T[x] - 1);   // twice the distance from the tile's centre, nearest image
            if (d[x] > rn.n[x]) d[x] -= 2 * rn.n[x];
            if (d[x] < -rn.n[x]) d[x] += 2 * rn.n[x];
        }
        d[3] = OLD && cell < 0 ? 0 : 1;
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int v = __reduce_add_sync(0xffffffffu, d[x]);
        if ((threadIdx.x & 31) == 0) atomicAdd(&sum[x], v);
    }
    __syncthreads();
    const float w = 0.5f / (float)max(sum[3], 1);
#pragma unroll
    for (int x = 0; x < DIM; ++x) o[x] = wrapi(o[x] + (int)rintf((float)sum[x] * w), rn.n[x]);
    __syncthreads();   // the words are free for the tiles
}

// A particle past the staged tile: the same arithmetic on the periodic global
// arrays, for particle p of the item's group, read from a.S at sp with RP.  Out of
// line, so that it does not raise the register count of the tiled path, and
// called for all of an item's such particles together (see process_item).  On the global
// arrays the fourth cell and third face along an axis that the particle did
// not cross carry nothing and are skipped, as on the tiled path (`full`).
template <int DIM, typename R, int MODE, int ORD, bool RP>
__device__ __noinline__ void far_particle(const PartArgs<R> &a, int group, long long p, long long sp)
{
    constexpr bool F32 = sizeof(R) == 4;
    const GroupDev &gr = a.groups[group];
    const RunDev &rn = a.runs[gr.run];
    const int nx = rn.n[0], ny = rn.n[1], nz = rn.n[2];
    const long long cb = rn.cell_base;
    R c2, cl, hq;
    if constexpr (F32) { cl = rn.cf; hq = gr.hqf; } else { cl = rn.c; hq = gr.hq; }
    c2 = cl * cl;
    const Pool<R> &src = RP ? a.S : a.P;
    const int cell0 = MODE == 2 ? a.old_cell[p] : src.cell[sp];
    const R o0 = MODE == 2 ? a.old_off[0][p] : src.off[0][sp];
    const R o1 = MODE == 2 ? a.old_off[1][p] : src.off[1][sp];
    const R o2 = DIM == 3 ? (MODE == 2 ? a.old_off[2][p] : src.off[2][sp]) : R(0);
    R w[3] = {R(0), R(0), R(0)};
    if (MODE != 2 || DIM == 2) {
        w[0] = src.w[0][sp];
        w[1] = src.w[1][sp];
        w[2] = src.w[2][sp];
    }
    const int rest = divu31(cell0, rn.div_nx);
    const int i = cell0 - rest * nx;
    const int k = DIM == 3 ? divu31(rest, rn.div_ny) : 0, j = DIM == 3 ? rest - k * ny : rest;
    // l_a = 2 1/2: the base index is the cell or the next one
    R a0 = o0, a1 = o1, a2 = o2;
    int u0 = 0, u1 = 0, u2 = 0;
    if constexpr (ORD == 5) {
        a2 = R(0.5);
        u0 = split5(o0, a0);
        u1 = split5(o1, a1);
        if (DIM == 3) u2 = split5(o2, a2);
    }
    int s0 = 0, s1 = 0, s2 = 0;
    R n0 = o0, n1 = o1, n2 = o2, uz = R(0);
    if (MODE != 2) {
        R Ep[3], Bp[3];
        if constexpr (ORD == 3) {
            GlobalReader<R> rd;
            for (int c = 0; c < 3; ++c) { rd.E[c] = a.F.E[c]; rd.B[c] = a.F.B[c]; }
            for (int q = 0; q < 4; ++q) {
                rd.xi[q] = cb + wrapi(i - 1 + q, nx);
                rd.yj[q] = (long long)nx * wrapi(j - 1 + q, ny);
                rd.zk[q] = DIM == 3 ? (long long)nx * ny * wrapi(k - 1 + q, nz) : 0;
            }
            R fx[2], Sx[3], fy[2], Sy[3], fz[2] = {R(1), R(0)}, Sz[3] = {R(0), R(1), R(0)};
            form_factor(o0, fx, Sx);
            form_factor(o1, fy, Sy);
            if (DIM == 3) form_factor(o2, fz, Sz);
            gather<DIM>(rd, fx, Sx, fy, Sy, fz, Sz, Ep, Bp);
        } else {
            GlobalReader5<R> rd;   // offsets -2..2 from the base index (l_a = 2 1/2) or the cell (Eq. wrong1)
            for (int c = 0; c < 3; ++c) { rd.E[c] = a.F.E[c]; rd.B[c] = a.F.B[c]; }
            for (int q = 0; q < 5; ++q) {
                rd.xi[q] = cb + wrapi(i + u0 - 2 + q, nx);
                rd.yj[q] = (long long)nx * wrapi(j + u1 - 2 + q, ny);
                rd.zk[q] = DIM == 3 ? (long long)nx * ny * wrapi(k + u2 - 2 + q, nz) : 0;
            }
            if constexpr (ORD == 5) {
                R f[21];   // f (3) and S (4) along x, y, z
                form_factor5(a0, f, f + 3);
                form_factor5(a1, f + 7, f + 10);
                form_factor5(a2, f + 14, f + 17);
                gather5<DIM>(rd, f, f + 3, f + 7, f + 10, f + 14, f + 17, Ep, Bp);
            } else {
                R f[2], S[9] = {R(0), R(1), R(0), R(0), R(1), R(0), R(0), R(1), R(0)};
                form_factor(o0, f, S);
                form_factor(o1, f, S + 3);
                if (DIM == 3) form_factor(o2, f, S + 6);
                gather_w1<DIM>(rd, S, S + 3, S + 6, Ep, Bp);
            }
        }
        boris(w, Ep, Bp, hq, c2);
        const bool live = finite3(w[0], w[1], w[2]);
        int cell1 = cell0;
        if (live) {
            R cN0, cN1, cN2;
            if constexpr (F32) { cN0 = rn.cNf[0]; cN1 = rn.cNf[1]; cN2 = rn.cNf[2]; }
            else { cN0 = rn.cN[0]; cN1 = rn.cN[1]; cN2 = rn.cN[2]; }
            const R ig = rsqrt_r(w[0] * w[0] + w[1] * w[1] + w[2] * w[2] + c2);
            s0 = renormalize(o0, w[0] * ig * cN0, n0);
            s1 = renormalize(o1, w[1] * ig * cN1, n1);
            if (DIM == 3) s2 = renormalize(o2, w[2] * ig * cN2, n2);
            uz = cl * w[2] * ig;
            cell1 = wrapi(i + s0, nx) + nx * (wrapi(j + s1, ny) + ny * (DIM == 3 ? wrapi(k + s2, nz) : 0));
            if (MODE == 1) {
                a.old_cell[p] = cell0;
                a.old_off[0][p] = o0;
                a.old_off[1][p] = o1;
                if (DIM == 3) a.old_off[2][p] = o2;
            }
        } else {
            atomicOr(a.err, ERR_NONFINITE);   // as in process_item: it keeps x^n and contributes no current
            if (MODE == 1) a.old_cell[p] = -1;
        }
        if (live || RP) {
            if (RP) a.P.id[p] = a.S.id[sp];
            a.P.cell[p] = cell1;
            a.P.off[0][p] = n0;
            a.P.off[1][p] = n1;
            if (DIM == 3) a.P.off[2][p] = n2;
            for (int c = 0; c < 3; ++c) a.P.w[c][p] = w[c];
        }
        if (MODE == 1 || !live) return;
    } else {
        const int cell1 = a.P.cell[p];
        n0 = a.P.off[0][p];
        n1 = a.P.off[1][p];
        if (DIM == 3) n2 = a.P.off[2][p];
        const int r1 = divu31(cell1, rn.div_nx);
        const int k1 = DIM == 3 ? divu31(r1, rn.div_ny) : 0;
        s0 = cell1 - r1 * nx - i; if (s0 > 1) s0 -= nx; if (s0 < -1) s0 += nx;
        s1 = r1 - k1 * ny - j; if (s1 > 1) s1 -= ny; if (s1 < -1) s1 += ny;
        if (DIM == 3) { s2 = k1 - k; if (s2 > 1) s2 -= nz; if (s2 < -1) s2 += nz; }
        if (DIM == 2) uz = cl * w[2] * rsqrt_r(w[0] * w[0] + w[1] * w[1] + w[2] * w[2] + c2);
    }
    R kf[3];
    for (int c = 0; c < 3; ++c) { if constexpr (F32) kf[c] = gr.kff[c]; else kf[c] = gr.kf[c]; }
    if constexpr (ORD == 5) {
        R b0, b1, b2 = R(0.5);
        const int q0 = s0 + split5(n0, b0) - u0, q1 = s1 + split5(n1, b1) - u1;
        const int q2 = DIM == 3 ? s2 + split5(n2, b2) - u2 : 0;
        AxisWin5<R> X, Y, Z;
        axis_window5(a0, b0, q0, X);
        axis_window5(a1, b1, q1, Y);
        if (DIM == 3) axis_window5(a2, b2, q2, Z); else Z = X;
        GlobalAcc<R, 5> acc;
        for (int c = 0; c < 3; ++c) acc.J[c] = a.F.J[c];
        acc.set(cb, i + u0, j + u1, k + u2, nx, ny, nz, X.lo, Y.lo, Z.lo, DIM == 3);
        deposit5<DIM>(acc, X, Y, Z, kf, uz, (q0 != 0 ? 1 : 0) | (q1 != 0 ? 2 : 0) | (q2 != 0 ? 4 : 0));
    } else {
        AxisWin<R> X, Y, Z;
        axis_window(o0, n0, s0, X);
        axis_window(o1, n1, s1, Y);
        if (DIM == 3) axis_window(o2, n2, s2, Z); else Z = X;
        GlobalAcc<R, 4> acc;
        for (int c = 0; c < 3; ++c) acc.J[c] = a.F.J[c];
        acc.set(cb, i, j, k, nx, ny, nz, X.lo, Y.lo, Z.lo, DIM == 3);
        deposit<DIM>(acc, X, Y, Z, kf, uz, (s0 != 0 ? 1 : 0) | (s1 != 0 ? 2 : 0) | (s2 != 0 ? 4 : 0));
    }
}

// MODE 0: fused gather + push + move + deposit (pic_step).
// MODE 1: gather + push + move, keeping x^n (pic_gather_push).
// MODE 2: deposit from the kept x^n and the current x^{n+1} (pic_deposit_current).
// Shared memory: E and B tiles (6 * nf values of R) for MODES 0, 1; the current
// tile for MODES 0, 2: in FP32 two int32 fixed-point words per value, in FP64
// one double -- 24 * nj bytes either way.
// ORD = 3 is l_a = 1 1/2, ORD = 5 is l_a = 2 1/2 (Sec. 4.5): its stencil
// reaches one cell further, so the field tile has a halo of (halo + 2) cells
// and the current tile one of (halo + 3), and every particle deposits through
// the bias-removing accumulator (the per-cell counts serve the l_a = 1 1/2
// stencil only).  ORD = 4 is the comparison scheme of Eq. wrong1: its gather
// reaches the integer points -1..2 (field tile halo (halo + 2)); its charge and
// current are those of l_a = 1 1/2.
template <int DIM, typename R, int MODE, class GEO, int ORD = 3, bool PERM = false, int NT = kThreads>
__device__ __forceinline__ void process_item(const PartArgs<R> &a, int item)
{
    // MODE 0 right after a sort whose arrays have not moved: the state comes
    // from a.S through a.perm, and the stepped particle goes to its new slot
    constexpr bool RP = PERM && MODE == 0;
    constexpr bool FIX = sizeof(R) == 4;
    const WorkItem it = a.items[item];
    const GroupDev gr = a.groups[it.group];
    const RunDev rn = a.runs[gr.run];
    const int G = GEO::dyn ? a.halo : GEO::G;
    const int nx = rn.n[0], ny = rn.n[1], nz = rn.n[2];
    const int T0 = GEO::dyn ? rn.tile[0] : GEO::T0, T1 = GEO::dyn ? rn.tile[1] : GEO::T1;
    const int T2 = DIM == 3 ? (GEO::dyn ? rn.tile[2] : GEO::T2) : 1;
    const int tx = it.tile % rn.ntile[0];
    const int ty = (it.tile / rn.ntile[0]) % rn.ntile[1];
    const int tz = DIM == 3 ? it.tile / (rn.ntile[0] * rn.ntile[1]) : 0;
    int org[3] = {tx * T0, ty * T1, tz * T2};
    if (!RP && 256LL * it.drifted > it.end - it.begin) {   // uniform over the block; none right after a sort
        const int T[3] = {T0, T1, T2};
        item_shift<DIM, R, MODE == 2, NT>(a, it, rn, T, org);
    }
    const int ox = org[0], oy = org[1], oz = org[2];
    constexpr int FH = ORD == 3 ? 1 : 2, JH = ORD == 5 ? 3 : 2;   // field and current halo beyond G
    const int fe0 = T0 + 2 * (G + FH), fe1 = T1 + 2 * (G + FH), fe2 = DIM == 3 ? T2 + 2 * (G + FH) : 1;
    const int je0 = T0 + 2 * (G + JH), je1 = T1 + 2 * (G + JH), je2 = DIM == 3 ? T2 + 2 * (G + JH) : 1;
    // the field tile is stored with the current tile's x and y pitches, so that
    // a particle's field and current bases differ by a constant and one bank
    // order of the particles (set by the tile sort) serves both
    const int P0 = GEO::dyn ? rn.pitch[0] : GEO::P0;   // >= je0 (see the tile layout choice)
    const int P1 = GEO::dyn ? rn.pitch[1] : GEO::P1;   // >= je1
    const int nf = P0 * P1 * fe2, nj = P0 * P1 * je2;
    // l_a = 2 1/2, FP32: particles whose base index stayed add raw words and the
    // bias comes off at the flush, which sums 64 counts per word of the current
    // tile.  That pays when the item has at least about 2/3 of a particle per
    // word (each such particle saves two integer subtractions on each of its
    // 144 contributions); sparser items take the bias off per contribution.
    // The choice is uniform over the block.
    const bool fix5 = FIX && ORD == 5 && (it.end - it.begin) * 3 >= 2LL * nj;
    constexpr bool NEED_F = MODE != 2;
    constexpr bool NEED_J = MODE != 1;
    const long long cb = rn.cell_base;

    R *sE[3], *sB[3];
    R *sJ[3];          // FP64 current tile
    int *sJh[3], *sJl[3];   // FP32 fixed-point current tile
    int *scnt = nullptr;    // FP32: particles that stayed in their cell, per base cell
    {
        unsigned char *sp = g_smem;
        if (NEED_F) {
            R *f = reinterpret_cast<R *>(sp);
            for (int c = 0; c < 3; ++c) { sE[c] = f + c * nf; sB[c] = f + (3 + c) * nf; }
            sp += 6 * (size_t)nf * sizeof(R);
        }
        if (NEED_J) {
            for (int c = 0; c < 3; ++c) {
                sJ[c] = reinterpret_cast<R *>(sp) + c * nj;
                sJh[c] = reinterpret_cast<int *>(sp) + c * nj;
                sJl[c] = reinterpret_cast<int *>(sp) + (3 + c) * nj;
            }
            if (FIX) scnt = reinterpret_cast<int *>(sp) + 6 * nj;
        }
    }

    // Deposit queue of this warp (MODES 0, 2).  A particle that stayed in its
    // cell along every axis deposits at once with three-cell windows (54
    // contributions in 3D, 21 in 2D), where its lane's bank is the one the tile
    // sort gave it.  A particle that changed cell needs four-cell windows along
    // the axes it crossed; it is queued and deposited later together with 31
    // other such particles, so that the wider windows are paid only by warps
    // of moved particles.  The integer current sums do not depend on the order.
    // The warps' queues lie one after another (values, then codes), followed by
    // one count per warp for the merged drain at the end of the item.
    const int warp = threadIdx.x >> 5;
    // In 3D FP64, where the queue has room for it (kQueueCap3), the particles that
    // crossed one axis only, most of those that moved, are queued apart, from the
    // queue's start, and drained with the windows they need (deposit_one_axis); the
    // others from its end.  48^3 cells of 16 + 16 particles, 4 steps: 17.4 ms, 18.0 with
    // one queue.  In FP32 the second drain costs the loop registers (128^3: 3 percent).
    constexpr bool SPLIT = DIM == 3 && !FIX && ORD != 5 && NEED_J;
    const int QC = SPLIT ? a.qcap : kQueueCap;
    const bool split = SPLIT && QC == kQueueCap3;
    R *qv0 = nullptr, *qv = nullptr;
    int *qs0 = nullptr, *qs = nullptr, *qcnt = nullptr, *qcnt1 = nullptr;
    if (NEED_J) {
        unsigned char *qb = g_smem + (NEED_F ? 6 * (size_t)nf * sizeof(R) : 0) + (FIX ? 28 : 24) * (size_t)nj;
        qv0 = reinterpret_cast<R *>(qb);
        qs0 = reinterpret_cast<int *>(qb + (size_t)(NT / 32) * QC * kQueueVals * sizeof(R));
        qcnt = qs0 + (NT / 32) * QC;
        qcnt1 = qcnt + NT / 32;   // with split
        qv = qv0 + (size_t)warp * QC * kQueueVals;
        qs = qs0 + warp * QC;
    }

    // Particles past the staged tile: their indices in the item go to the item's
    // part of far_list, and far_particle steps them together after the others.  A
    // warp with one such lane would otherwise run the global-memory path for it
    // alone, and a call from inside
    // the loop would spill what the loop keeps in registers.
    // Their number stands in a value of the queue that this dimension does not
    // use, so that the kernels take no more shared memory for it.
    int *nfar;
    if constexpr (NEED_J) {
        nfar = reinterpret_cast<int *>(qv0 + (DIM == 3 ? 6 : 2) * QC);
    } else {
        __shared__ int count;
        nfar = &count;
    }
    if (threadIdx.x == 0) *nfar = 0;

    if (NEED_F) {
        // Asynchronous copies, so that all of a thread's are in flight at once, of two
        // values each where the rows allow it: the box starts on an even cell of an
        // even row length, so a pair lies in one row on both sides of the wrap.  With
        // the present kernels the pairs change little: the 3D push and the persistent
        // steps gain 0.3 to 2 percent, the slab and l_a = 2 1/2 lose 0.7.
        if (((P0 | fe0 | nx | (ox - G - FH)) & 1) == 0 && (cb & 1) == 0) {
            const int h0 = fe0 >> 1;
            for (int q = threadIdx.x; q < h0 * fe1 * fe2; q += blockDim.x) {
                const int lx = 2 * (q % h0), r = q / h0, ly = r % fe1, lz = r / fe1;
                const int gx = wrapi(ox - G - FH + lx, nx);
                const int gy = wrapi(oy - G - FH + ly, ny);
                const int gz = DIM == 3 ? wrapi(oz - G - FH + lz, nz) : 0;
                const long long gi = cb + gx + (long long)nx * (gy + (long long)ny * gz);
                const int l = lx + P0 * (ly + P1 * lz);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    copy_async<2 * sizeof(R)>(sE[c] + l, a.F.E[c] + gi);
                    copy_async<2 * sizeof(R)>(sB[c] + l, a.F.B[c] + gi);
                }
            }
        } else {
            for (int q = threadIdx.x; q < fe0 * fe1 * fe2; q += blockDim.x) {
                const int lx = q % fe0, r = q / fe0, ly = r % fe1, lz = r / fe1;
                const int gx = wrapi(ox - G - FH + lx, nx);
                const int gy = wrapi(oy - G - FH + ly, ny);
                const int gz = DIM == 3 ? wrapi(oz - G - FH + lz, nz) : 0;
                const long long gi = cb + gx + (long long)nx * (gy + (long long)ny * gz);
                const int l = lx + P0 * (ly + P1 * lz);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    copy_async<sizeof(R)>(sE[c] + l, a.F.E[c] + gi);
                    copy_async<sizeof(R)>(sB[c] + l, a.F.B[c] + gi);
                }
            }
        }
    }
    if (NEED_J) {
        int *z = sJh[0];   // 24 * nj bytes = 6 * nj words in both precisions, + nj counts in FP32
        const int nw = (FIX ? 7 : 6) * nj;
        int l0 = 0;
        if ((nf & 1) == 0 || !NEED_F) {   // 16-byte aligned: 6 * nf * sizeof(R) bytes from the start
            for (int l = threadIdx.x; l < nw >> 2; l += blockDim.x) reinterpret_cast<int4 *>(z)[l] = make_int4(0, 0, 0, 0);
            l0 = nw & ~3;
        }
        for (int l = l0 + threadIdx.x; l < nw; l += blockDim.x) z[l] = 0;
    }
    if (NEED_F) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // constants of the group and run, prepared on the host (no FP64 arithmetic
    // runs in the FP32 kernels)
    R hq, cl, cN0, cN1, cN2;
    R kf[3], kfs[3];   // kfs: prefactors with the fixed-point scale of the FP32 current tile folded in
    if constexpr (FIX) {
        hq = gr.hqf;
        cl = rn.cf;
        cN0 = rn.cNf[0]; cN1 = rn.cNf[1]; cN2 = rn.cNf[2];
        for (int c = 0; c < 3; ++c) { kf[c] = gr.kff[c]; kfs[c] = gr.kfsf[c]; }
    } else {
        hq = gr.hq;
        cl = rn.c;
        cN0 = rn.cN[0]; cN1 = rn.cN[1]; cN2 = rn.cN[2];
        for (int c = 0; c < 3; ++c) { kf[c] = gr.kf[c]; kfs[c] = gr.kf[c]; }
    }
    const R c2 = cl * cl;

    const int lane = threadIdx.x & 31;
    int qn = 0;   // entries in this warp's queue (warp-uniform): at its start, or with split at its end
    int q1 = 0;   // with split: entries at its start


    auto deposit_local = [&](int base, const AxisWin<R> &X, const AxisWin<R> &Y, const AxisWin<R> &Z, R uz,
                             int full, int only) {
        if constexpr (FIX) {
            FixedAcc acc;   // bias taken off per contribution (variable stencil)
            for (int c = 0; c < 3; ++c) { acc.hi[c] = sJh[c]; acc.lo[c] = sJl[c]; }
            acc.base = base;
            acc.s1 = P0;
            acc.s2 = P0 * P1;
            deposit<DIM>(acc, X, Y, Z, kfs, uz, full, only);
        } else {
            SmemAcc<R> acc;
            for (int c = 0; c < 3; ++c) acc.J[c] = sJ[c];
            acc.base = base;
            acc.s1 = P0;
            acc.s2 = P0 * P1;
            deposit<DIM>(acc, X, Y, Z, kf, uz, full, only);
        }
    };
    auto deposit_local5 = [&](int base, const AxisWin5<R> &X, const AxisWin5<R> &Y, const AxisWin5<R> &Z, R uz,
                              int full, int only) {
        if constexpr (FIX) {
            FixedAcc acc;
            for (int c = 0; c < 3; ++c) { acc.hi[c] = sJh[c]; acc.lo[c] = sJl[c]; }
            acc.base = base;
            acc.s1 = P0;
            acc.s2 = P0 * P1;
            deposit5<DIM>(acc, X, Y, Z, kfs, uz, full, only);
        } else {
            SmemAcc<R> acc;
            for (int c = 0; c < 3; ++c) acc.J[c] = sJ[c];
            acc.base = base;
            acc.s1 = P0;
            acc.s2 = P0 * P1;
            deposit5<DIM>(acc, X, Y, Z, kf, uz, full, only);
        }
    };
    // deposits, on each lane with `on`, entry `slot` of the queue whose values
    // and codes start at sv and ss (a whole warp calls it): all of its current, or
    // the component `only` (warp-uniform)
    auto drain = [&](const R *sv, const int *ss, int slot, bool on, int only) {
        R d0 = R(0), d1 = R(0), d2 = R(0), e0 = R(0), e1 = R(0), e2 = R(0), u = R(0);
        int code = 1 | (1 << 2) | (1 << 4);
        if (on) {
            d0 = sv[0 * QC + slot];
            d1 = sv[1 * QC + slot];
            e0 = sv[3 * QC + slot];
            e1 = sv[4 * QC + slot];
            if (DIM == 3) {
                d2 = sv[2 * QC + slot];
                e2 = sv[5 * QC + slot];
            } else {
                u = sv[6 * QC + slot];
            }
            code = ss[slot];
        }
        const int q0 = (code & 3) - 1, q1 = ((code >> 2) & 3) - 1, q2 = ((code >> 4) & 3) - 1;
        const int full = (__any_sync(0xffffffffu, q0 != 0) ? 1 : 0) | (__any_sync(0xffffffffu, q1 != 0) ? 2 : 0) |
                         (DIM == 3 && __any_sync(0xffffffffu, q2 != 0) ? 4 : 0);
        if (on) {
            if constexpr (ORD == 5) {   // the entries hold the l_a = 2 1/2 d values
                AxisWin5<R> X, Y, Z;
                axis_window5(d0, e0, q0, X);
                axis_window5(d1, e1, q1, Y);
                if (DIM == 3) axis_window5(d2, e2, q2, Z); else Z = X;
                deposit_local5(code >> 8, X, Y, Z, u, full, only);
            } else {
                AxisWin<R> X, Y, Z;
                axis_window(d0, e0, q0, X);
                axis_window(d1, e1, q1, Y);
                if (DIM == 3) axis_window(d2, e2, q2, Z); else Z = X;
                deposit_local(code >> 8, X, Y, Z, u, full, only);
            }
        }
    };
    // the same for entries that crossed one axis
    auto drain_one = [&](const R *sv, const int *ss, int slot, bool on, int only) {
        if constexpr (SPLIT) {
            if (!on) return;
            const int code = ss[slot];
            const int A = (code & 3) != 1 ? 0 : ((code >> 2) & 3) != 1 ? 1 : 2;
            const int B = A == 2 ? 0 : A + 1, Cx = A == 0 ? 2 : A - 1;
            auto of = [](int ax, auto v0, auto v1, auto v2) { return ax == 0 ? v0 : ax == 1 ? v1 : v2; };
            const int s[3] = {of(A, 1, P0, P0 * P1), of(B, 1, P0, P0 * P1), of(Cx, 1, P0, P0 * P1)};
            const R k[3] = {of(A, kfs[0], kfs[1], kfs[2]), of(B, kfs[0], kfs[1], kfs[2]),
                            of(Cx, kfs[0], kfs[1], kfs[2])};
            R *const J[3] = {sJ[0] + A * nj, sJ[0] + B * nj, sJ[0] + Cx * nj};
            AxisWin<R> X, Y, Z;
            axis_window(sv[A * QC + slot], sv[(3 + A) * QC + slot], ((code >> (2 * A)) & 3) - 1, X);
            axis_window_still(sv[B * QC + slot], sv[(3 + B) * QC + slot], Y);
            axis_window_still(sv[Cx * QC + slot], sv[(3 + Cx) * QC + slot], Z);
            deposit_one_axis<R>(J, X, Y, Z, k, (code >> 8) + X.lo * s[0] - s[1] - s[2], s, only);
        }
    };

    // warps run whole rounds of 32 consecutive particles (the last one partial)
    // RP: the permutation index of the lane's next particle is read one round ahead
    unsigned sp_next = 0;
    if (RP && it.begin + threadIdx.x < it.end) sp_next = a.perm[it.begin + threadIdx.x];
    // PRE: a round's state is read while the round before is worked on.  256x256
    // cells of 16 particles, 40 steps: 2.34 ms, 2.37 without; the 24 batched runs, 30
    // steps: 18.1 and 19.6; 128^3 cells of 32 + 32, 12 steps: 100.8 and 102.1.  Not in
    // FP64, where it changes nothing, nor for halos of two, whose particles are often
    // not in the tile (the slab 14.9 ms with it, 14.7 without).  Nor in 3D with tiles
    // read at run time or through a sort's permutation, where it lost a little when
    // it came in (with the present kernels it would gain 0.6 and 1.2 percent).
    constexpr bool PRE = FIX && MODE == 0 && (DIM == 2 || (!RP && !GEO::dyn && GEO::G < 2));
    int pre_c = 0, pre_id = 0;
    unsigned sp_after = 0;   // RP with PRE: the permutation index of the round after next
    if (PRE && RP && it.begin + NT + threadIdx.x < it.end) sp_after = a.perm[it.begin + NT + threadIdx.x];
    R pre_o0 = 0, pre_o1 = 0, pre_o2 = 0, pre_w0 = 0, pre_w1 = 0, pre_w2 = 0;
    auto fetch = [&](long long q) {
        if (q < it.end) {
            const Pool<R> &src = RP ? a.S : a.P;
            const long long sq = RP ? (long long)sp_next : q;
            pre_c = src.cell[sq];
            pre_o0 = src.off[0][sq];
            pre_o1 = src.off[1][sq];
            if (DIM == 3) pre_o2 = src.off[2][sq];
            pre_w0 = src.w[0][sq];
            pre_w1 = src.w[1][sq];
            pre_w2 = src.w[2][sq];
            if (RP) pre_id = src.id[sq];
        }
    };
    if (PRE) fetch(it.begin + threadIdx.x);
    for (long long pw = it.begin + (threadIdx.x & ~31); pw < it.end; pw += NT) {
        const long long p = pw + lane;
        const bool valid = p < it.end;
        const long long pn = pw + NT;   // the warp's next round
        unsigned sp_cur = 0;
        if (RP) {
            sp_cur = sp_next;
            if (PRE) {
                sp_next = sp_after;
                if (pn + NT + lane < it.end) sp_after = a.perm[pn + NT + lane];
            } else if (pn + lane < it.end) {
                sp_next = a.perm[pn + lane];
            }
        }
        bool live = false;   // the particle moves and deposits this step
        bool far = false;    // it lies past the staged tile: far_particle steps it later
        int i = 0, j = 0, k = 0, li = 0, lj = 0, lk = 0;
        R o0 = R(0), o1 = R(0), o2 = R(0), n0 = R(0), n1 = R(0), n2 = R(0), uz = R(0);
        int s0 = 0, s1 = 0, s2 = 0, id = 0;
        if (valid) {
            // ---- the particle's state at x^n (old) -------------------------------
            const long long sp = RP ? (long long)sp_cur : p;   // where the state is read
            const Pool<R> &src = RP ? a.S : a.P;
            const int cell0 = PRE ? pre_c : MODE == 2 ? a.old_cell[p] : src.cell[sp];
            o0 = PRE ? pre_o0 : MODE == 2 ? a.old_off[0][p] : src.off[0][sp];
            o1 = PRE ? pre_o1 : MODE == 2 ? a.old_off[1][p] : src.off[1][sp];
            o2 = DIM == 3 ? (PRE ? pre_o2 : MODE == 2 ? a.old_off[2][p] : src.off[2][sp]) : R(0);
            R w[3] = {R(0), R(0), R(0)};
            if (PRE) {
                w[0] = pre_w0;
                w[1] = pre_w1;
                w[2] = pre_w2;
                id = pre_id;
                fetch(pn + lane);
            } else if (MODE != 2 || DIM == 2) {
                w[0] = src.w[0][sp];
                w[1] = src.w[1][sp];
                w[2] = src.w[2][sp];
            }

            const int rest = divu31(cell0, rn.div_nx);
            i = cell0 - rest * nx;
            if (DIM == 3) {
                k = divu31(rest, rn.div_ny);
                j = rest - k * ny;
            } else {
                j = rest;
            }
            li = local_coord(i, ox, T0, G, nx);
            lj = local_coord(j, oy, T1, G, ny);
            lk = DIM == 3 ? local_coord(k, oz, T2, G, nz) : 0;
            const bool inr =
                li >= -G && li < T0 + G && lj >= -G && lj < T1 + G && (DIM == 2 || (lk >= -G && lk < T2 + G));
            const bool saved = MODE != 2 || cell0 >= 0;   // < 0: its momentum became non-finite in the push
            far = !inr && saved;

            n0 = o0; n1 = o1; n2 = o2;
            live = inr && saved;
            if (far) {
                // stepped after the others, a block's width of them at a time
            } else if (MODE != 2) {
                R Ep[3], Bp[3];
                if constexpr (ORD == 5) {
                    R e0, e1, e2 = R(0.5);
                    const int u0 = split5(o0, e0), u1 = split5(o1, e1), u2 = DIM == 3 ? split5(o2, e2) : 0;
                    R w[21];   // f (3) and S (4) along x, y, z
                    form_factor5(e0, w, w + 3);
                    form_factor5(e1, w + 7, w + 10);
                    form_factor5(e2, w + 14, w + 17);
                    SmemReader<R> rd;
                    for (int c = 0; c < 3; ++c) { rd.E[c] = sE[c]; rd.B[c] = sB[c]; }
                    rd.base = (li + u0 + G + FH) +
                              P0 * ((lj + u1 + G + FH) + (DIM == 3 ? P1 * (lk + u2 + G + FH) : 0));
                    rd.s1 = P0;
                    rd.s2 = P0 * P1;
                    gather5<DIM>(rd, w, w + 3, w + 7, w + 10, w + 14, w + 17, Ep, Bp);
                } else if constexpr (ORD == 4) {
                    R f[2], S[9] = {R(0), R(1), R(0), R(0), R(1), R(0), R(0), R(1), R(0)};   // S along x, y, z
                    form_factor(o0, f, S);
                    form_factor(o1, f, S + 3);
                    if (DIM == 3) form_factor(o2, f, S + 6);
                    SmemReader<R> rd;
                    for (int c = 0; c < 3; ++c) { rd.E[c] = sE[c]; rd.B[c] = sB[c]; }
                    rd.base = (li + G + FH) + P0 * ((lj + G + FH) + (DIM == 3 ? P1 * (lk + G + FH) : 0));
                    rd.s1 = P0;
                    rd.s2 = P0 * P1;
                    gather_w1<DIM>(rd, S, S + 3, S + 6, Ep, Bp);
                } else {
                    R fx[2], Sx[3], fy[2], Sy[3], fz[2], Sz[3];
                    form_factor(o0, fx, Sx);
                    form_factor(o1, fy, Sy);
                    if (DIM == 3) {
                        form_factor(o2, fz, Sz);
                    } else {
                        fz[0] = R(1); fz[1] = R(0);
                        Sz[0] = R(0); Sz[1] = R(1); Sz[2] = R(0);
                    }
                    SmemReader<R> rd;
                    for (int c = 0; c < 3; ++c) { rd.E[c] = sE[c]; rd.B[c] = sB[c]; }
                    rd.base = (li + G + 1) + P0 * ((lj + G + 1) + (DIM == 3 ? P1 * (lk + G + 1) : 0));
                    rd.s1 = P0;
                    rd.s2 = P0 * P1;
                    gather<DIM>(rd, fx, Sx, fy, Sy, fz, Sz, Ep, Bp);
                }
                boris(w, Ep, Bp, hq, c2);
                if (!finite3(w[0], w[1], w[2])) {
                    atomicOr(a.err, ERR_NONFINITE);
                    live = false;   // the particle keeps x^n and contributes no current
                    if (MODE == 1) a.old_cell[p] = -1;   // (which tells the deposit)
                    if (RP) {   // ... in its slot of the new order, with the momentum it reached
                        a.P.id[p] = PRE ? id : a.S.id[sp];
                        a.P.cell[p] = cell0;
                        a.P.off[0][p] = o0;
                        a.P.off[1][p] = o1;
                        if (DIM == 3) a.P.off[2][p] = o2;
                        for (int c = 0; c < 3; ++c) a.P.w[c][p] = w[c];
                    }
                } else {
                    const R ig = rsqrt_r(w[0] * w[0] + w[1] * w[1] + w[2] * w[2] + c2);
                    s0 = renormalize(o0, w[0] * ig * cN0, n0);
                    s1 = renormalize(o1, w[1] * ig * cN1, n1);
                    if (DIM == 3) s2 = renormalize(o2, w[2] * ig * cN2, n2);
                    uz = cl * w[2] * ig;
                    const int i1 = wrapi(i + s0, nx), j1 = wrapi(j + s1, ny), k1 = DIM == 3 ? wrapi(k + s2, nz) : 0;
                    const int cell1 = i1 + nx * (j1 + ny * k1);
                    if (MODE == 1) {
                        a.old_cell[p] = cell0;
                        a.old_off[0][p] = o0;
                        a.old_off[1][p] = o1;
                        if (DIM == 3) a.old_off[2][p] = o2;
                    }
                    if (RP) a.P.id[p] = PRE ? id : a.S.id[sp];   // the id moves with the particle
                    a.P.cell[p] = cell1;
                    a.P.off[0][p] = n0;
                    a.P.off[1][p] = n1;
                    if (DIM == 3) a.P.off[2][p] = n2;
                    a.P.w[0][p] = w[0];
                    a.P.w[1][p] = w[1];
                    a.P.w[2][p] = w[2];
                }
            } else {
                // deposit-only: x^{n+1} is the stored state, the shift follows from the cells
                const int cell1 = a.P.cell[p];
                n0 = a.P.off[0][p];
                n1 = a.P.off[1][p];
                if (DIM == 3) n2 = a.P.off[2][p];
                const int r1 = divu31(cell1, rn.div_nx);
                const int i1 = cell1 - r1 * nx;
                const int k1 = DIM == 3 ? divu31(r1, rn.div_ny) : 0;
                const int j1 = r1 - k1 * ny;
                s0 = i1 - i; if (s0 > 1) s0 -= nx; if (s0 < -1) s0 += nx;
                s1 = j1 - j; if (s1 > 1) s1 -= ny; if (s1 < -1) s1 += ny;
                if (DIM == 3) { s2 = k1 - k; if (s2 > 1) s2 -= nz; if (s2 < -1) s2 += nz; }
                if (DIM == 2) {
                    const R ig = rsqrt_r(w[0] * w[0] + w[1] * w[1] + w[2] * w[2] + c2);
                    uz = cl * w[2] * ig;
                }
            }
        }
        const unsigned fm = __ballot_sync(0xffffffffu, far);
        if (fm != 0u) {   // warp-uniform
            int at = 0;
            if (lane == 0) at = atomicAdd(nfar, __popc(fm));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(fm & ((1u << lane) - 1u));
            if (far) a.far_list[it.begin + at] = (unsigned)(p - it.begin);
        }
        if (MODE == 1) continue;

        // ---- virtual-path current (Eq. current) -------------------------------
        // The windows take the d values and shifts of the base index: for
        // l_a = 1 1/2 the offsets and cell shifts themselves; for l_a = 2 1/2 the
        // base index is cell + (offset >= 1/2), so it moves with the cell shift
        // and the half-offset flags.
        int q0 = s0, qy = s1, q2 = s2;
        R a0 = o0, a1 = o1, a2 = o2, b0 = n0, b1 = n1, b2 = n2;
        int ub0 = 0, ub1 = 0, ub2 = 0;   // old base index - old cell
        if constexpr (ORD == 5) {
            ub0 = split5(o0, a0);
            ub1 = split5(o1, a1);
            const int v0 = split5(n0, b0), v1 = split5(n1, b1);
            q0 = s0 + v0 - ub0;
            qy = s1 + v1 - ub1;
            if (DIM == 3) {
                ub2 = split5(o2, a2);
                q2 = s2 + split5(n2, b2) - ub2;
            }
        }
        const bool moved = (q0 | qy | q2) != 0;
        const int base = (li + ub0 + G + JH) +
                         P0 * ((lj + ub1 + G + JH) + (DIM == 3 ? P1 * (lk + ub2 + G + JH) : 0));
        if (live && !moved) {
            if constexpr (ORD == 5) {
                AxisWin5<R> X, Y, Z;
                axis_window5(a0, b0, 0, X);
                axis_window5(a1, b1, 0, Y);
                if (DIM == 3) axis_window5(a2, b2, 0, Z); else Z = X;
                if (fix5) {
                    // fixed stencil: the bias comes off once per word at the flush
                    FixedAccT<false> acc;
                    for (int c = 0; c < 3; ++c) { acc.hi[c] = sJh[c]; acc.lo[c] = sJl[c]; }
                    acc.base = base;
                    acc.s1 = P0;
                    acc.s2 = P0 * P1;
                    deposit5<DIM>(acc, X, Y, Z, kfs, uz, 0);
                    atomicAdd(&scnt[base], 1);
                } else {
                    deposit_local5(base, X, Y, Z, uz, 0, -1);
                }
            } else {
                AxisWin<R> X, Y, Z;
                axis_window_still(o0, n0, X);
                axis_window_still(o1, n1, Y);
                if (DIM == 3) axis_window_still(o2, n2, Z); else Z = X;
                if constexpr (FIX) {
                    // fixed stencil: the bias comes off once per word at the flush
                    FixedAccT<false> acc;
                    for (int c = 0; c < 3; ++c) { acc.hi[c] = sJh[c]; acc.lo[c] = sJl[c]; }
                    acc.base = base;
                    acc.s1 = P0;
                    acc.s2 = P0 * P1;
                    deposit<DIM>(acc, X, Y, Z, kfs, uz, 0);
                    atomicAdd(&scnt[base], 1);
                } else {
                    deposit_local(base, X, Y, Z, uz, 0, -1);
                }
            }
        }
        const bool enq = live && moved;
        const unsigned qm = __ballot_sync(0xffffffffu, enq);
        const bool one = split && enq && (q0 != 0) + (qy != 0) + (q2 != 0) == 1;
        const unsigned om = split ? __ballot_sync(0xffffffffu, one) : 0u;
        const unsigned mm = qm & ~om;
        if (enq) {
            const unsigned below = (1u << lane) - 1u;
            const int slot = one ? q1 + __popc(om & below)
                                 : split ? QC - 1 - (qn + __popc(mm & below)) : qn + __popc(mm & below);
            qv[0 * QC + slot] = a0;
            qv[1 * QC + slot] = a1;
            qv[3 * QC + slot] = b0;
            qv[4 * QC + slot] = b1;
            if (DIM == 3) {
                qv[2 * QC + slot] = a2;
                qv[5 * QC + slot] = b2;
            } else {
                qv[6 * QC + slot] = uz;
            }
            qs[slot] = (base << 8) | (q0 + 1) | ((qy + 1) << 2) | ((q2 + 1) << 4);
        }
        qn += __popc(mm);
        q1 += __popc(om);
        if (qn >= 32) {   // warp-uniform
            __syncwarp();
            qn -= 32;
            drain(qv, qs, split ? QC - 1 - (qn + lane) : qn + lane, true, -1);
            __syncwarp();   // the drained slots are free again
        }
        if (q1 >= 32) {   // warp-uniform
            __syncwarp();
            q1 -= 32;
            drain_one(qv, qs, q1 + lane, true, -1);
            __syncwarp();
        }
    }
    if (NEED_J && lane == 0) {
        qcnt[warp] = qn;
        if (split) qcnt1[warp] = q1;
    }
    __syncthreads();
    const int nf_all = *nfar;
    if (nf_all > 0) {
        for (int m = threadIdx.x; m < nf_all; m += blockDim.x) {
            const long long pf = it.begin + a.far_list[it.begin + m];
            far_particle<DIM, R, MODE, ORD, RP>(a, it.group, pf, RP ? (long long)a.perm[pf] : pf);
        }
        if (MODE != 2 && threadIdx.x == 0) {   // the sort policy's measure of drift, and item_shift's
            atomicAdd(reinterpret_cast<unsigned *>(a.err) + 1, (unsigned)nf_all);
            a.items[item].drifted = add_drifted(it.drifted, nf_all);
        }
    }
    if (NEED_J) {
        // The entries left in the warps' queues (fewer than 32 each) are drained
        // together: merged entry m is slot m - (entries of the warps before) of
        // its warp's queue, 32 of them per drain.  While they are few, each drain is
        // three, one per component of the current, on three warps: the block waits
        // for the longest, and a drain of all three components is as long as
        // a round of particles.  Few is one in FP32 (64^3 cells of 2 + 2 particles, 20
        // steps, 3.82 ms, 3.92 undivided; with up to five drains in thirds the slab lost 4.6
        // percent to forming the windows three times) and, in FP64, as many as give
        // a warp two thirds (32x32 cells, 50 steps, 2.21 and 2.31 ms; 48^3 of 16 + 16, 4
        // steps, 17.4 and 17.5).
        int tot = 0, tot1 = 0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) {
            tot += qcnt[w];
            if (split) tot1 += qcnt1[w];
        }
        const int nd1 = (tot1 + 31) >> 5, nd = nd1 + ((tot + 31) >> 5);
        const bool thirds = FIX ? nd <= 1 : 3 * nd <= 2 * (NT / 32);
        for (int d = warp; d < (thirds ? 3 * nd : nd); d += NT / 32) {   // uniform over the warp
            const int which = thirds ? d / 3 : d, only = thirds ? d % 3 : -1;
            const bool one = which < nd1;
            const int *cnt = one ? qcnt1 : qcnt;
            const int m = 32 * (one ? which : which - nd1) + lane;
            const bool on = m < (one ? tot1 : tot);
            int src = 0, slot = m;
#pragma unroll
            for (int w = 0; w < NT / 32 - 1; ++w) {
                const int c = cnt[src];
                if (slot >= c) {
                    slot -= c;
                    ++src;
                }
            }
            if (!on) src = slot = 0;
            const R *sv = qv0 + (size_t)src * QC * kQueueVals;
            const int *ss = qs0 + src * QC;
            if (one)
                drain_one(sv, ss, slot, on, only);
            else
                drain(sv, ss, split ? QC - 1 - slot : slot, on, only);
        }
        __syncthreads();
        const float jinv = gr.jinv;
        if constexpr (FIX && ORD != 5 && DIM == 3) {
            // A thread takes a column of words along z and keeps the counts of three
            // planes (all nine neighbours of the plane, and its +1 column and row): the
            // stencil of a particle that stayed in its cell, with base b, covers
            // b + (dx, dy, dz) with dx in {0, 1} and dy, dz in {-1, 0, 1} for J^x, likewise
            // for J^y and J^z, so word l received the counts of the 27 bases around l
            // less the +1 plane of the component's axis.  Bases lie two words or
            // more inside the tile, so the planes before the first and after the last
            // hold none.  Nine reads of counts per word instead of 27: 64^3 cells with 2 + 2
            // particles each, 20 steps, 3.82 ms against 3.92, 128^3 with 32 + 32, 12 steps,
            // 100.8 against 101.3.
            for (int q = threadIdx.x; q < je0 * je1; q += blockDim.x) {
                const int lx = q % je0, ly = q / je0;
                const int gx = wrapi(ox - G - JH + lx, nx), gy = wrapi(oy - G - JH + ly, ny);
                const long long gxy = cb + gx + (long long)nx * gy;
                const bool in = lx >= 1 && lx < je0 - 1 && ly >= 1 && ly < je1 - 1;
                unsigned t0 = 0, x0 = 0, y0 = 0, t1 = 0, x1 = 0, y1 = 0;
                int l = lx + P0 * ly;
                auto plane = [&](int at, unsigned &t, unsigned &x, unsigned &y) {
                    const int *c = scnt + at;
                    const unsigned b0 = c[-1 - P0], b1 = c[-P0], b2 = c[1 - P0], m0 = c[-1], m1 = c[0], m2 = c[1],
                                   u0 = c[P0 - 1], u1 = c[P0], u2 = c[P0 + 1];
                    x = b2 + m2 + u2;
                    y = u0 + u1 + u2;
                    t = b0 + b1 + m0 + m1 + x + u0 + u1;
                };
                if (in) plane(l, t1, x1, y1);
                for (int lz = 0; lz < je2; ++lz, l += P0 * P1) {
                    unsigned t2 = 0, x2 = 0, y2 = 0;
                    if (in && lz + 1 < je2) plane(l + P0 * P1, t2, x2, y2);
                    const unsigned s = t0 + t1 + t2;
                    const unsigned off[3] = {(s - (x0 + x1 + x2)) * kFixBias, (s - (y0 + y1 + y2)) * kFixBias,
                                             (t0 + t1) * kFixBias};
                    const long long gi = gxy + (long long)nx * ny * wrapi(oz - G - JH + lz, nz);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const int h = (int)((unsigned)sJh[c][l] - off[c]), lo = (int)((unsigned)sJl[c][l] - off[c]);
                        if ((h | lo) != 0) atomicAdd(&a.F.J[c][gi], (R)(fmaf((float)h, 65536.0f, (float)lo) * jinv));
                    }
                    t0 = t1; x0 = x1; y0 = y1;
                    t1 = t2; x1 = x2; y1 = y2;
                }
            }
        } else
        for (int l = threadIdx.x; l < nj; l += blockDim.x) {
            const int lx = l % P0, r = l / P0, ly = r % P1, lz = r / P1;
            if (lx >= je0 || ly >= je1) continue;   // pitch padding
            const int gx = wrapi(ox - G - JH + lx, nx);
            const int gy = wrapi(oy - G - JH + ly, ny);
            const int gz = DIM == 3 ? wrapi(oz - G - JH + lz, nz) : 0;
            const long long gi = cb + gx + (long long)nx * (gy + (long long)ny * gz);
            // FP32: contributions of particles that stayed in their cell, per
            // component: the stencil of such a particle with base b covers the
            // cells b + (dx, dy, dz) with dx in {0, 1} and dy, dz in {-1, 0, 1}
            // for J^x (faces 0, 1; cells -1..1), likewise for J^y and J^z, so a
            // cell l received sum_{b in l - stencil} cnt[b] of them
            unsigned nst[3] = {0u, 0u, 0u};
            if (fix5) {
                // l_a = 2 1/2: the stencil of base b covers b + (dx, dy, dz) with
                // dx in {-1, 0, 1} (faces) and dy, dz in {-2, ..., 1} (cells) for
                // J^x, likewise for J^y and J^z; so the bases of word l are
                // l + o, o in {-1, ..., 2} per axis, without the o_a = 2 plane for
                // J^a.  A base is the local cell (in [-G, T + G)) plus the
                // half-offset flag (0 or 1) plus G + JH, so bases lie in
                // [JH, T + 2G + JH] = [JH, je - JH] along each axis: only those
                // indices are read, which keeps every read in the tile.
                bool vx[4], vy[4], vz[4];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    vx[o] = lx + o - 1 >= JH && lx + o - 1 <= je0 - JH;
                    vy[o] = ly + o - 1 >= JH && ly + o - 1 <= je1 - JH;
                    vz[o] = DIM == 3 ? (lz + o - 1 >= JH && lz + o - 1 <= je2 - JH) : o == 1;
                }
                unsigned tot = 0, px = 0, py = 0, pz = 0;   // all, and the o = 2 planes
#pragma unroll
                for (int oz = -1; oz <= (DIM == 3 ? 2 : -1); ++oz)
#pragma unroll
                    for (int oy = -1; oy <= 2; ++oy)
#pragma unroll
                        for (int ox = -1; ox <= 2; ++ox) {
                            const int dz = DIM == 3 ? oz : 0;
                            if (!(vx[ox + 1] && vy[oy + 1] && vz[dz + 1])) continue;
                            const unsigned v = (unsigned)scnt[l + ox + P0 * (oy + P1 * dz)];
                            tot += v;
                            if (ox == 2) px += v;
                            if (oy == 2) py += v;
                            if (DIM == 3 && oz == 2) pz += v;
                        }
                nst[0] = tot - px;
                nst[1] = tot - py;
                nst[2] = tot - pz;
            }
            if constexpr (FIX && ORD != 5) {
                if (lx >= 1 && lx < je0 - 1 && ly >= 1 && ly < je1 - 1 && (DIM == 2 || (lz >= 1 && lz < je2 - 1))) {
                    if (DIM == 3) {
                        unsigned tot = 0, px = 0, py = 0, pz = 0;   // all 27, and the +1 planes
#pragma unroll
                        for (int oz = -1; oz <= 1; ++oz)
#pragma unroll
                            for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
                                for (int ox = -1; ox <= 1; ++ox) {
                                    const unsigned v = (unsigned)scnt[l + ox + P0 * (oy + P1 * oz)];
                                    tot += v;
                                    if (ox == 1) px += v;
                                    if (oy == 1) py += v;
                                    if (oz == 1) pz += v;
                                }
                        nst[0] = tot - px;
                        nst[1] = tot - py;
                        nst[2] = tot - pz;
                    } else {
                        unsigned tot = 0, px = 0, py = 0;
#pragma unroll
                        for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
                            for (int ox = -1; ox <= 1; ++ox) {
                                const unsigned v = (unsigned)scnt[l + ox + P0 * oy];
                                tot += v;
                                if (ox == 1) px += v;
                                if (oy == 1) py += v;
                            }
                        nst[0] = tot - px;
                        nst[1] = tot - py;
                        nst[2] = tot;
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if constexpr (FIX) {
                    const unsigned off = nst[c] * kFixBias;
                    const int h = (int)((unsigned)sJh[c][l] - off), lo = (int)((unsigned)sJl[c][l] - off);
                    if ((h | lo) != 0)
                        atomicAdd(&a.F.J[c][gi], (R)(fmaf((float)h, 65536.0f, (float)lo) * jinv));
                } else {
                    const R v = sJ[c][l];
                    if (v != R(0)) atomicAdd(&a.F.J[c][gi], v);
                }
            }
        }
    }
    __syncthreads();   // the shared tiles are free for the block's next item
}

template <int DIM, typename R, int MODE, class GEO = GeoDyn, int ORD = 3, bool PERM = false, bool ONE = false>
__global__ void __launch_bounds__(block_threads<R, ONE>(), ONE ? 1 : min_blocks<DIM, R, MODE>())
    k_particles(const __grid_constant__ PartArgs<R> a)
{
    if ((int)blockIdx.x >= *a.n_items) return;
    process_item<DIM, R, MODE, GEO, ORD, PERM, block_threads<R, ONE>()>(a, blockIdx.x);
}

// Run of a batch that owns concatenated cell l (run_cell_base has nruns + 1 entries).
__device__ __forceinline__ int find_run(const long long *run_cell_base, int nruns, long long l)
{
    int lo = 0, hi = nruns;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (run_cell_base[mid] <= l) lo = mid; else hi = mid;
    }
    return lo;
}

// One whole step of every run of a batch in one cooperative launch: B half
// step (+ J clear) over all cells, grid barrier, the fused particle work items,
// grid barrier, B half step, grid barrier, E full step.  The grid is sized so
// that all blocks are resident (cooperative launch), which the barriers need.
// PERM: the step right after a sort that left the arrays in place; the work
// items read the particles through the permutation (as k_particles does).
template <int DIM, typename R, class GEO = GeoDyn, bool PERM = false, bool ONE = false>
__global__ void __launch_bounds__(kThreads, ONE ? 1 : min_blocks_persistent<DIM, R, GEO::dyn>()) k_step_persistent(const __grid_constant__ PartArgs<R> a, int nruns,
                                                              const long long *run_cell_base, long long *ant_n,
                                                              int antennas)
{
    cg::grid_group grid = cg::this_grid();
    const long long total = run_cell_base[nruns];
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (long long l = t0; l < total; l += stride) {
        const int r = find_run(run_cell_base, nruns, l);
        yee_b_half_cell<DIM, R>(a.runs[r], a.F, l - run_cell_base[r], 1, ant_n[r]);
    }
    grid.sync();
    const int ni = *a.n_items;
    for (int it = blockIdx.x; it < ni; it += gridDim.x) process_item<DIM, R, 0, GEO, 3, PERM>(a, it);
    grid.sync();
    for (long long l = t0; l < total; l += stride) {
        const int r = find_run(run_cell_base, nruns, l);
        yee_b_half_cell<DIM, R>(a.runs[r], a.F, l - run_cell_base[r], 0, ant_n[r]);
    }
    grid.sync();
    for (long long l = t0; l < total; l += stride) {
        const int r = find_run(run_cell_base, nruns, l);
        yee_e_cell<DIM, R>(a.runs[r], a.F, l - run_cell_base[r], ant_n[r]);
    }
    if (antennas) {   // the antenna clocks advance once every block has read them
        grid.sync();
        if (blockIdx.x == 0)
            for (int r = threadIdx.x; r < nruns; r += blockDim.x) ant_n[r] += 1;
    }
}

// The launch's deposit queues: their capacity, and the shared memory they add to smem.
template <int DIM, typename R, int MODE>
static size_t choose_queue(size_t smem, int nt, int *qcap)
{
    *qcap = kQueueCap;
    if (DIM != 3 || sizeof(R) == 4 || MODE == 1) return smem;
    const size_t more = smem + queue3_bytes<R>(nt);
    if (more > kSmemMax || std::min(2, blocks_per_sm(more)) < std::min(2, blocks_per_sm(smem))) return smem;
    *qcap = kQueueCap3;
    return more;
}

template <int DIM, typename R, int MODE, class GEO = GeoDyn, int ORD = 3>
static cudaError_t launch_t(cudaStream_t st, int max_items, size_t smem, PartArgs<R> a)
{
    if (max_items <= 0) return cudaSuccess;
    if constexpr (GEO::dyn && DIM == 3) {
        constexpr int nt = block_threads<R, true>();
        size_t smem1 = smem_of<R, MODE>(smem, nt);
        if (one_block_per_sm(smem) && smem1 <= kSmemMax) {
            smem1 = choose_queue<DIM, R, MODE>(smem1, nt, &a.qcap);
            if constexpr (MODE == 0 && ORD == 3) {
                if (a.perm) {
                    k_particles<DIM, R, 0, GEO, 3, true, true><<<max_items, nt, smem1, st>>>(a);
                    return cudaGetLastError();
                }
            }
            k_particles<DIM, R, MODE, GEO, ORD, false, true><<<max_items, nt, smem1, st>>>(a);
            return cudaGetLastError();
        }
    }
    smem = choose_queue<DIM, R, MODE>(smem, kThreads, &a.qcap);
    if constexpr (MODE == 0 && ORD == 3) {
        if (a.perm) {   // right after a sort: the kernel that reads through the permutation
            k_particles<DIM, R, 0, GEO, 3, true><<<max_items, kThreads, smem, st>>>(a);
            return cudaGetLastError();
        }
    }
    k_particles<DIM, R, MODE, GEO, ORD><<<max_items, kThreads, smem, st>>>(a);
    return cudaGetLastError();
}

// The shared-memory limit of a particle kernel, of each variant.
template <int DIM, typename R, int MODE, class GEO, int ORD = 3, bool PERM = false>
static cudaError_t set_limit_one(int bytes)
{
    cudaError_t e = allow_smem(k_particles<DIM, R, MODE, GEO, ORD, PERM>, (size_t)bytes);
    if constexpr (GEO::dyn && DIM == 3) {
        if (e == cudaSuccess) e = allow_smem(k_particles<DIM, R, MODE, GEO, ORD, PERM, true>, (size_t)bytes);
    }
    return e;
}

// The shared-memory limit of the fused kernel of a geometry, both variants.
template <int DIM, typename R, class GEO>
static cudaError_t set_limit_fused(int bytes)
{
    cudaError_t e = set_limit_one<DIM, R, 0, GEO>(bytes);
    if (e != cudaSuccess) return e;
    return set_limit_one<DIM, R, 0, GEO, 3, true>(bytes);
}

template <int DIM, typename R, class GEO = GeoDyn>
static cudaError_t persistent_t(cudaStream_t st, size_t smem, int nruns, const long long *run_cell_base,
                                PartArgs<R> a, int *grid_blocks, int launch, long long *ant_n, int antennas)
{
    smem = choose_queue<DIM, R, 0>(smem, kThreads, &a.qcap);
    constexpr bool both = GEO::dyn && DIM == 3;
    auto fn0 = k_step_persistent<DIM, R, GEO, false>;
    auto fn1 = k_step_persistent<DIM, R, GEO, true>;
    if (both && one_block_per_sm(smem)) {
        fn0 = k_step_persistent<DIM, R, GEO, false, both>;
        fn1 = k_step_persistent<DIM, R, GEO, true, both>;
    }
    auto fn = a.perm ? fn1 : fn0;
    cudaError_t e;
    if (*grid_blocks <= 0) {
        // first use (outside any stream capture): shared-memory limit and grid
        // size, the same for both variants (all blocks of either must be resident)
        int dev = 0, sms = 0, per = 1 << 30;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        for (auto f : {fn0, fn1}) {
            e = allow_smem(f, smem);
            if (e != cudaSuccess) return e;
            int pf = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pf, f, kThreads, smem);
            if (e != cudaSuccess) return e;
            per = std::min(per, pf);
        }
        if (per <= 0) return cudaErrorInvalidConfiguration;
        *grid_blocks = sms * per;
    }
    if (!launch) return cudaSuccess;
    void *args[] = {(void *)&a, (void *)&nruns, (void *)&run_cell_base, (void *)&ant_n, (void *)&antennas};
    return cudaLaunchCooperativeKernel((const void *)fn, dim3(*grid_blocks), dim3(kThreads), args, smem, st);
}

// Kernel arguments from the host-side buffers.
template <typename R>
inline PartArgs<R> make_args(WorkItem *items, const int *n_items, const RunDev *runs, const GroupDev *groups,
                             const PoolBuf &P, void *const E[3], void *const B[3], void *const J[3], int *old_cell,
                             void *const old_off[3], int halo, int *err, unsigned *far_list,
                             const PoolBuf *S = nullptr, const unsigned *perm = nullptr)
{
    PartArgs<R> a;
    a.far_list = far_list;
    a.qcap = kQueueCap;
    a.items = items;
    a.n_items = n_items;
    a.runs = runs;
    a.groups = groups;
    a.P.cell = P.cell;
    a.P.id = P.id;
    const PoolBuf &Q = S ? *S : P;
    a.S.cell = Q.cell;
    a.S.id = Q.id;
    a.perm = S ? perm : nullptr;
    for (int c = 0; c < 3; ++c) {
        a.S.off[c] = static_cast<R *>(Q.off[c]);
        a.S.w[c] = static_cast<R *>(Q.w[c]);
        a.P.off[c] = static_cast<R *>(P.off[c]);
        a.P.w[c] = static_cast<R *>(P.w[c]);
        a.F.E[c] = static_cast<R *>(E[c]);
        a.F.B[c] = static_cast<R *>(B[c]);
        a.F.J[c] = static_cast<R *>(J[c]);
        a.old_off[c] = static_cast<R *>(old_off[c]);
    }
    a.old_cell = old_cell;
    a.halo = halo;
    a.err = err;
    return a;
}

// Kernels with a fixed tile geometry (pic_particles_fixed.cu), FP32 fused step
// and persistent batch step.  Each returns false, without launching, when no
// fixed kernel has the grid's geometry.
bool launch_particles_fixed(int dims, cudaStream_t st, int max_items, size_t smem, const PartArgs<float> &a,
                            const int tile[3], int halo, int p0, int p1, cudaError_t *err);
bool launch_persistent_fixed(int dims, cudaStream_t st, size_t smem, int nruns, const long long *run_cell_base,
                             const PartArgs<float> &a, int *grid_blocks, int launch, const int tile[3], int halo,
                             int p0, int p1, long long *ant_n, int antennas, cudaError_t *err);
cudaError_t fixed_set_smem_limit(int dims, size_t bytes);

// Launch and shared-memory limit of the kernels of another stencil (ORD = 5:
// l_a = 2 1/2 in pic_particles_o5.cu; ORD = 4: Eq. wrong1 in pic_particles_w1.cu),
// any tile geometry, both precisions, all three modes.
template <int DIM, typename R, int ORD>
static cudaError_t launch_mode_ord(int mode, cudaStream_t st, int max_items, size_t smem, const PartArgs<R> &a)
{
    switch (mode) {
    case 0: return launch_t<DIM, R, 0, GeoDyn, ORD>(st, max_items, smem, a);
    case 1: return launch_t<DIM, R, 1, GeoDyn, ORD>(st, max_items, smem, a);
    default: return launch_t<DIM, R, 2, GeoDyn, ORD>(st, max_items, smem, a);
    }
}

template <int ORD>
static cudaError_t launch_particles_ord_t(int dims, int prec, int mode, cudaStream_t st, int max_items, size_t smem,
                                          WorkItem *items, const int *n_items, const RunDev *runs,
                                          const GroupDev *groups, const PoolBuf &P, void *const E[3],
                                          void *const B[3], void *const J[3], int *old_cell, void *const old_off[3],
                                          int halo, int *err, unsigned *far_list)
{
    if (prec == 0) {
        auto a = make_args<double>(items, n_items, runs, groups, P, E, B, J, old_cell, old_off, halo, err,
                                     far_list);
        return dims == 3 ? launch_mode_ord<3, double, ORD>(mode, st, max_items, smem, a)
                         : launch_mode_ord<2, double, ORD>(mode, st, max_items, smem, a);
    }
    auto a = make_args<float>(items, n_items, runs, groups, P, E, B, J, old_cell, old_off, halo, err,
                                     far_list);
    return dims == 3 ? launch_mode_ord<3, float, ORD>(mode, st, max_items, smem, a)
                     : launch_mode_ord<2, float, ORD>(mode, st, max_items, smem, a);
}

template <int DIM, typename R, int ORD>
static cudaError_t set_limit_ord(int mode, size_t bytes)
{
    const int b = (int)bytes;
    switch (mode) {
    case 0: return set_limit_one<DIM, R, 0, GeoDyn, ORD>(b);
    case 1: return set_limit_one<DIM, R, 1, GeoDyn, ORD>(b);
    default: return set_limit_one<DIM, R, 2, GeoDyn, ORD>(b);
    }
}

template <int ORD>
static cudaError_t particles_ord_set_smem_limit_t(int dims, int prec, int mode, size_t bytes)
{
    if (dims == 3)
        return prec == 0 ? set_limit_ord<3, double, ORD>(mode, bytes) : set_limit_ord<3, float, ORD>(mode, bytes);
    return prec == 0 ? set_limit_ord<2, double, ORD>(mode, bytes) : set_limit_ord<2, float, ORD>(mode, bytes);
}

cudaError_t launch_particles_o5(int dims, int prec, int mode, cudaStream_t st, int max_items, size_t smem,
                                WorkItem *items, const int *n_items, const RunDev *runs, const GroupDev *groups,
                                const PoolBuf &P, void *const E[3], void *const B[3], void *const J[3],
                                int *old_cell, void *const old_off[3], int halo, int *err, unsigned *far_list,
                                const int tile[3], int p0, int p1);
cudaError_t particles_o5_set_smem_limit(int dims, int prec, int mode, size_t bytes);
cudaError_t launch_particles_w1(int dims, int prec, int mode, cudaStream_t st, int max_items, size_t smem,
                                WorkItem *items, const int *n_items, const RunDev *runs, const GroupDev *groups,
                                const PoolBuf &P, void *const E[3], void *const B[3], void *const J[3],
                                int *old_cell, void *const old_off[3], int halo, int *err, unsigned *far_list);
cudaError_t particles_w1_set_smem_limit(int dims, int prec, int mode, size_t bytes);

}  // namespace pic
