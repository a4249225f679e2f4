// pic_device.cuh -- device-side data structures and per-particle arithmetic of
// the charge-conserving PIC step (Sokolov, arXiv:1101.0809), shared by the
// particle kernels.  Everything here is templated on the dimension (2 = 2D3V
// with an ignorable z, 3 = 3D3V) and on the real type R (float or double).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pic {

// ---------------------------------------------------------------------------
// Device-side descriptors.  A batch holds one or more independent runs; each
// (run, species) pair is a "group" owning a contiguous range of the particle
// pool.  Tiles of all groups share one global numbering (group tile_base + the
// tile's linear index inside its run) that is the sort key.
// ---------------------------------------------------------------------------
// Division of a non-negative int below 2^31 by a fixed divisor d >= 1 as a
// multiply and shift (Granlund and Montgomery, "Division by invariant integers
// using multiplication", 1994, Thm. 4.2): with L = 31 + ceil(log2 d) and
// m = ceil(2^L / d) (at most 2^32), floor(n / d) = (n * m) >> L exactly, and
// n * m < 2^63.
struct DivU31 {
    unsigned long long m;
    int L;
};
inline DivU31 make_divu31(int d)
{
    int c = 0;
    while ((1LL << c) < (long long)d) ++c;
    const int L = 31 + c;
    DivU31 v;
    v.m = (unsigned long long)(((unsigned __int128)1 << L) + (unsigned)d - 1) / (unsigned)d;
    v.L = L;
    return v;
}
__device__ __forceinline__ int divu31(int n, const DivU31 &v)
{
    return (int)(((unsigned long long)(unsigned)n * v.m) >> v.L);
}

// l / d for cell numbers, with inv = ceil(2^64 / d), d >= 2: l inv / 2^64 exceeds the
// quotient by less than l / 2^64, and by less than 1/d while l d < 2^64 (fewer than
// 2^33 cells fit the device, d < 2^31).
inline unsigned long long make_inv(int d) { return ~0ull / (unsigned)d + 1; }
__host__ __device__ __forceinline__ long long div_cells(long long l, unsigned long long inv)
{
#ifdef __CUDA_ARCH__
    return (long long)__umul64hi((unsigned long long)l, inv);
#else
    return (long long)((unsigned __int128)(unsigned long long)l * inv >> 64);
#endif
}

struct RunDev {
    int n[3];             // cells per axis (n[2] = 1 in 2D)
    int tile[3];          // tile extents (tile[2] = 1 in 2D)
    int ntile[3];         // tiles per axis, ceil(n/tile)
    int pitch[2];         // x and y pitch of the shared-memory field and current tiles
    long long cell_base;  // first cell of this run in the concatenated field arrays
    double cN[3];         // Courant numbers c*dt/d_a
    double dt, c;
    double d[3];
    double V;             // cell volume (dx*dy in 2D)
    double rho_bg;        // uniform background charge density
    // plane-wave antenna (include/pic.h): pol 0 none, 1 E_y/B_z, 2 E_z/B_y;
    // the total field starts at the B node x = ant_i0
    int ant_pol, ant_i0;
    double ant_E0, ant_omega, ant_ramp;
    double fpdt;            // 4 pi dt
    float fpdtf;            // 4 pi dt in FP32
    DivU31 div_nx, div_ny;  // division by n[0] and n[1]
    unsigned long long inv_nx, inv_ny;  // the same of cell numbers from 2^31 on (div_cells)
    DivU31 div_t[3];        // division by the tile extents
    float cf, cNf[3];     // c and the Courant numbers in FP32
};

struct GroupDev {
    int run;
    int tile_base;        // global tile id of this group's tile 0
    long long base, n;    // particle range [base, base+n) in the pool
    double qm;            // q/m
    double qp;            // macro charge q_p = weight*q
    double mp;            // macro mass m_p = weight*m
    float jscale;         // fixed-point scale of the FP32 shared current tile (a power of two)
    float jinv;           // 1 / jscale
    // push and deposit prefactors of the group in its run, from the host:
    // hq = (1/2)(q/m) dt; kf[a] = -(1/4)(d_a/dt) q_p/V in 3D, and in 2D
    // kf[0,1] = -(1/2)(d_a/dt) q_p/V, kf[2] = (1/4) q_p/V (see deposit)
    double hq, kf[3];
    float hqf, kff[3], kfsf[3];   // FP32: the same, and kf * jscale
    float rscale, rinv;   // fixed-point scale of the FP32 diagnostics' shared charge tile, 1/rscale
};

struct WorkItem {
    int group;
    int tile;             // tile index inside the run
    long long begin, end; // particle range of this item
    int drifted;          // particles found past the staged tile, summed over the steps since the sort
};

// The sum of WorkItem::drifted with one step's count, held at the largest int: an
// item may go unsorted for any number of steps.
__host__ __device__ __forceinline__ int add_drifted(int sum, int more)
{
    return more > 0x7fffffff - sum ? 0x7fffffff : sum + more;
}

template <typename R>
struct Pool {
    int *cell;
    R *off[3];
    R *w[3];
    int *id;
};

template <typename R>
struct Fields {
    R *E[3];
    R *B[3];
    R *J[3];
};

enum : int { ERR_NONFINITE = 1 };

// 4, 8 or 16 bytes from global to shared memory, both aligned to as much,
// without waiting; complete after cp.async.wait_all of the thread.
template <int BYTES>
__device__ __forceinline__ void copy_async(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES)
                 : "memory");
}

__device__ __forceinline__ int wrapi(int i, int n)
{
    return i < 0 ? i + n : (i >= n ? i - n : i);
}

// ---------------------------------------------------------------------------
// Alternating-order form factor l_a = 1 1/2 (Sec. 4.5): with d the in-cell
// offset of the particle, the lower-order point values at the integer points
// i, i+1 are f = (1-d, d), and the cell integrals at the half-integer points
// i-1/2, i+1/2, i+3/2 (centres of cells i-1, i, i+1) are
// S = ((1-d)^2/2, 3/4 - (1/2-d)^2, d^2/2).
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void form_factor(R d, R f[2], R S[3])
{
    const R h = R(0.5);
    const R e = R(1) - d;
    const R m = h - d;
    f[0] = e;
    f[1] = d;
    S[0] = h * e * e;
    S[1] = R(0.75) - m * m;
    S[2] = h * d * d;
}

// ---------------------------------------------------------------------------
// Two FP32 values in one register pair, and the packed fused multiply-add
// (fma.rn.f32x2): each half is rounded as the scalar operation would be.  The
// FP32 particle kernels are bound by instruction issue beside the
// shared-memory pipe, and the gather and the deposit do every operation on two
// taps or two contributions with the same weight.
// ---------------------------------------------------------------------------
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float a, float b)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lo2(F2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float hi2(F2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// ---------------------------------------------------------------------------
// Field readers.  Offsets (dx, dy, dz) are relative to the particle's cell.
// ---------------------------------------------------------------------------
template <typename R>
struct SmemReader {          // E/B tile with halo in shared memory
    const R *E[3];
    const R *B[3];
    int base, s1, s2;        // index of the particle cell, strides in y and z
    __device__ __forceinline__ R e(int a, int dx, int dy, int dz) const { return E[a][base + dx + s1 * dy + s2 * dz]; }
    __device__ __forceinline__ R b(int a, int dx, int dy, int dz) const { return B[a][base + dx + s1 * dy + s2 * dz]; }
};

template <typename R>
struct GlobalReader {        // periodic global arrays (particles outside their tile's halo)
    const R *E[3];
    const R *B[3];
    long long xi[4], yj[4], zk[4];   // wrapped offsets for relative -1..2 per axis
    __device__ __forceinline__ long long at(int dx, int dy, int dz) const { return xi[dx + 1] + yj[dy + 1] + zk[dz + 1]; }
    __device__ __forceinline__ R e(int a, int dx, int dy, int dz) const { return E[a][at(dx, dy, dz)]; }
    __device__ __forceinline__ R b(int a, int dx, int dy, int dz) const { return B[a][at(dx, dy, dz)]; }
};

// ---------------------------------------------------------------------------
// Gather (Sec. 2 interpolation sums with alpha of Eq. alphax and beta of
// Eq. betax).  Along its own axis an E component uses f, along the others S;
// a B component uses S along its own axis and f along the others.  2D drops
// every z factor (it sums to one).
// ---------------------------------------------------------------------------
// WITH_B = false leaves Bp unset (for callers that read E alone, whose registers
// are too few for the packed form).
template <int DIM, bool WITH_B = true, typename R, class Rd>
__device__ __forceinline__ void gather(const Rd &rd, const R fx[2], const R Sx[3], const R fy[2], const R Sy[3],
                                       const R fz[2], const R Sz[3], R Ep[3], R Bp[3])
{
    if constexpr (DIM == 3 && sizeof(R) == 4 && WITH_B) {
        // as below, the two sums u and v of a component (the two points of the axis
        // where its weights are f) packed: 128^3 cells of 32 + 32 particles, 12 steps,
        // 100.8 ms, 101.4 unpacked; the slab 14.7 and 14.8; in 2D no difference
        F2 x[3], y[3], z[3], gy[2], gz[2];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            x[q] = pack2(Sx[q], Sx[q]);
            y[q] = pack2(Sy[q], Sy[q]);
            z[q] = pack2(Sz[q], Sz[q]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            gy[q] = pack2(fy[q], fy[q]);
            gz[q] = pack2(fz[q], fz[q]);
        }
        F2 u;
        auto end = [&](const R f[2]) { return f[0] * lo2(u) + f[1] * hi2(u); };
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            F2 t = mul2(y[0], pack2(rd.e(0, 0, -1, c - 1), rd.e(0, 1, -1, c - 1)));
            t = fma2(y[1], pack2(rd.e(0, 0, 0, c - 1), rd.e(0, 1, 0, c - 1)), t);
            t = fma2(y[2], pack2(rd.e(0, 0, 1, c - 1), rd.e(0, 1, 1, c - 1)), t);
            u = c ? fma2(z[c], t, u) : mul2(z[c], t);
        }
        Ep[0] = end(fx);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            F2 t = mul2(x[0], pack2(rd.e(1, -1, 0, c - 1), rd.e(1, -1, 1, c - 1)));
            t = fma2(x[1], pack2(rd.e(1, 0, 0, c - 1), rd.e(1, 0, 1, c - 1)), t);
            t = fma2(x[2], pack2(rd.e(1, 1, 0, c - 1), rd.e(1, 1, 1, c - 1)), t);
            u = c ? fma2(z[c], t, u) : mul2(z[c], t);
        }
        Ep[1] = end(fy);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            F2 t = mul2(x[0], pack2(rd.e(2, -1, b - 1, 0), rd.e(2, -1, b - 1, 1)));
            t = fma2(x[1], pack2(rd.e(2, 0, b - 1, 0), rd.e(2, 0, b - 1, 1)), t);
            t = fma2(x[2], pack2(rd.e(2, 1, b - 1, 0), rd.e(2, 1, b - 1, 1)), t);
            u = b ? fma2(y[b], t, u) : mul2(y[b], t);
        }
        Ep[2] = end(fz);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            F2 t = mul2(x[0], pack2(rd.b(0, -1, b, 0), rd.b(0, -1, b, 1)));
            t = fma2(x[1], pack2(rd.b(0, 0, b, 0), rd.b(0, 0, b, 1)), t);
            t = fma2(x[2], pack2(rd.b(0, 1, b, 0), rd.b(0, 1, b, 1)), t);
            u = b ? fma2(gy[b], t, u) : mul2(gy[b], t);
        }
        Bp[0] = end(fz);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            F2 t = mul2(y[0], pack2(rd.b(1, 0, -1, c), rd.b(1, 1, -1, c)));
            t = fma2(y[1], pack2(rd.b(1, 0, 0, c), rd.b(1, 1, 0, c)), t);
            t = fma2(y[2], pack2(rd.b(1, 0, 1, c), rd.b(1, 1, 1, c)), t);
            u = c ? fma2(gz[c], t, u) : mul2(gz[c], t);
        }
        Bp[1] = end(fx);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            F2 t = mul2(gy[0], pack2(rd.b(2, 0, 0, c - 1), rd.b(2, 1, 0, c - 1)));
            t = fma2(gy[1], pack2(rd.b(2, 0, 1, c - 1), rd.b(2, 1, 1, c - 1)), t);
            u = c ? fma2(z[c], t, u) : mul2(z[c], t);
        }
        Bp[2] = end(fx);
    } else if constexpr (DIM == 2 && sizeof(R) == 4 && WITH_B) {
        F2 x[3], y[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            x[q] = pack2(Sx[q], Sx[q]);
            y[q] = pack2(Sy[q], Sy[q]);
        }
        auto end = [&](const R f[2], F2 u) { return f[0] * lo2(u) + f[1] * hi2(u); };
        auto three = [&](const F2 w[3], F2 a, F2 b, F2 c) { return fma2(w[2], c, fma2(w[1], b, mul2(w[0], a))); };
        Ep[0] = end(fx, three(y, pack2(rd.e(0, 0, -1, 0), rd.e(0, 1, -1, 0)), pack2(rd.e(0, 0, 0, 0), rd.e(0, 1, 0, 0)),
                              pack2(rd.e(0, 0, 1, 0), rd.e(0, 1, 1, 0))));
        Ep[1] = end(fy, three(x, pack2(rd.e(1, -1, 0, 0), rd.e(1, -1, 1, 0)), pack2(rd.e(1, 0, 0, 0), rd.e(1, 0, 1, 0)),
                              pack2(rd.e(1, 1, 0, 0), rd.e(1, 1, 1, 0))));
        // E^z: S along both axes, the rows -1 and 0 packed
        const F2 r = three(x, pack2(rd.e(2, -1, -1, 0), rd.e(2, -1, 0, 0)), pack2(rd.e(2, 0, -1, 0), rd.e(2, 0, 0, 0)),
                           pack2(rd.e(2, 1, -1, 0), rd.e(2, 1, 0, 0)));
        Ep[2] = Sy[0] * lo2(r) + Sy[1] * hi2(r) +
                Sy[2] * (Sx[0] * rd.e(2, -1, 1, 0) + Sx[1] * rd.e(2, 0, 1, 0) + Sx[2] * rd.e(2, 1, 1, 0));
        Bp[0] = end(fy, three(x, pack2(rd.b(0, -1, 0, 0), rd.b(0, -1, 1, 0)), pack2(rd.b(0, 0, 0, 0), rd.b(0, 0, 1, 0)),
                              pack2(rd.b(0, 1, 0, 0), rd.b(0, 1, 1, 0))));
        Bp[1] = end(fx, three(y, pack2(rd.b(1, 0, -1, 0), rd.b(1, 1, -1, 0)), pack2(rd.b(1, 0, 0, 0), rd.b(1, 1, 0, 0)),
                              pack2(rd.b(1, 0, 1, 0), rd.b(1, 1, 1, 0))));
        Bp[2] = end(fx, fma2(pack2(fy[1], fy[1]), pack2(rd.b(2, 0, 1, 0), rd.b(2, 1, 1, 0)),
                             mul2(pack2(fy[0], fy[0]), pack2(rd.b(2, 0, 0, 0), rd.b(2, 1, 0, 0)))));
    } else if (DIM == 3) {
        // One axis at a time, the one that leaves fewest sums first: 26 operations for
        // a component of E and 18 for one of B, 132 in all instead of the 164 of a
        // weight product per row (3 percent of an FP64 step at 48^3 cells and 16 + 16
        // particles each).  Component after component, so that few sums are live at once.
        R u = 0, v = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            u += Sz[c] * (Sy[0] * rd.e(0, 0, -1, c - 1) + Sy[1] * rd.e(0, 0, 0, c - 1) + Sy[2] * rd.e(0, 0, 1, c - 1));
            v += Sz[c] * (Sy[0] * rd.e(0, 1, -1, c - 1) + Sy[1] * rd.e(0, 1, 0, c - 1) + Sy[2] * rd.e(0, 1, 1, c - 1));
        }
        Ep[0] = fx[0] * u + fx[1] * v;
        u = v = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            u += Sz[c] * (Sx[0] * rd.e(1, -1, 0, c - 1) + Sx[1] * rd.e(1, 0, 0, c - 1) + Sx[2] * rd.e(1, 1, 0, c - 1));
            v += Sz[c] * (Sx[0] * rd.e(1, -1, 1, c - 1) + Sx[1] * rd.e(1, 0, 1, c - 1) + Sx[2] * rd.e(1, 1, 1, c - 1));
        }
        Ep[1] = fy[0] * u + fy[1] * v;
        u = v = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            u += Sy[b] * (Sx[0] * rd.e(2, -1, b - 1, 0) + Sx[1] * rd.e(2, 0, b - 1, 0) + Sx[2] * rd.e(2, 1, b - 1, 0));
            v += Sy[b] * (Sx[0] * rd.e(2, -1, b - 1, 1) + Sx[1] * rd.e(2, 0, b - 1, 1) + Sx[2] * rd.e(2, 1, b - 1, 1));
        }
        Ep[2] = fz[0] * u + fz[1] * v;
        if (!WITH_B) return;
        u = v = 0;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            u += fy[b] * (Sx[0] * rd.b(0, -1, b, 0) + Sx[1] * rd.b(0, 0, b, 0) + Sx[2] * rd.b(0, 1, b, 0));
            v += fy[b] * (Sx[0] * rd.b(0, -1, b, 1) + Sx[1] * rd.b(0, 0, b, 1) + Sx[2] * rd.b(0, 1, b, 1));
        }
        Bp[0] = fz[0] * u + fz[1] * v;
        u = v = 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            u += fz[c] * (Sy[0] * rd.b(1, 0, -1, c) + Sy[1] * rd.b(1, 0, 0, c) + Sy[2] * rd.b(1, 0, 1, c));
            v += fz[c] * (Sy[0] * rd.b(1, 1, -1, c) + Sy[1] * rd.b(1, 1, 0, c) + Sy[2] * rd.b(1, 1, 1, c));
        }
        Bp[1] = fx[0] * u + fx[1] * v;
        u = v = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            u += Sz[c] * (fy[0] * rd.b(2, 0, 0, c - 1) + fy[1] * rd.b(2, 0, 1, c - 1));
            v += Sz[c] * (fy[0] * rd.b(2, 1, 0, c - 1) + fy[1] * rd.b(2, 1, 1, c - 1));
        }
        Bp[2] = fx[0] * u + fx[1] * v;
    } else {
        R ex = 0, ey = 0, ez = 0, bx = 0, by = 0, bz = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            ex += Sy[b] * (fx[0] * rd.e(0, 0, b - 1, 0) + fx[1] * rd.e(0, 1, b - 1, 0));
            ez += Sy[b] * (Sx[0] * rd.e(2, -1, b - 1, 0) + Sx[1] * rd.e(2, 0, b - 1, 0) + Sx[2] * rd.e(2, 1, b - 1, 0));
            by += Sy[b] * (fx[0] * rd.b(1, 0, b - 1, 0) + fx[1] * rd.b(1, 1, b - 1, 0));
        }
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            ey += fy[b] * (Sx[0] * rd.e(1, -1, b, 0) + Sx[1] * rd.e(1, 0, b, 0) + Sx[2] * rd.e(1, 1, b, 0));
            bx += fy[b] * (Sx[0] * rd.b(0, -1, b, 0) + Sx[1] * rd.b(0, 0, b, 0) + Sx[2] * rd.b(0, 1, b, 0));
            bz += fy[b] * (fx[0] * rd.b(2, 0, b, 0) + fx[1] * rd.b(2, 1, b, 0));
        }
        Ep[0] = ex; Ep[1] = ey; Ep[2] = ez;
        Bp[0] = bx; Bp[1] = by; Bp[2] = bz;
    }
}

// ---------------------------------------------------------------------------
// Relativistic push of the Appendix (Eq. 1): e = (q dt/2m) E; w~ = w + e;
// b = (q dt/2m) B / sqrt(w~^2 + c^2); w_n = w~ + w~ x b;
// w' = w~ + e + 2 (w_n x b)/(1 + b^2).   hq = q dt/(2m).
// ---------------------------------------------------------------------------
// The reciprocal of sqrt(x), a quotient by sqrt(x) and the quotient 2/(1 + b^2).  In
// FP64 by CUDA's rsqrt, whose error is at most 0.51 ulp (measured over 2e6 values):
// 1/sqrt(x) with its two roundings reached 1.49, and a quotient by sqrt(x) has two
// either way (a rsqrt(x) 1.46 ulp at most, a/sqrt(x) 1.47).  An FP64 instruction
// occupies its pipe for 16 cycles per warp: 17.4 ms for 4 steps at 48^3 cells and
// 16 + 16 particles each, 17.8 by root and quotient.  In FP32 the hardware reciprocal square root and a fast
// reciprocal, whose few-ulp errors lie far below the FP32 form's tolerance and
// replace the longer IEEE division and square-root sequences.
__device__ __forceinline__ double rsqrt_r(double x) { return rsqrt(x); }
__device__ __forceinline__ float rsqrt_r(float x) { return rsqrtf(x); }
__device__ __forceinline__ double div_sqrt(double a, double x) { return a * rsqrt(x); }
__device__ __forceinline__ float div_sqrt(float a, float x) { return a * rsqrtf(x); }
__device__ __forceinline__ double two_over(double x) { return 2.0 / x; }
__device__ __forceinline__ float two_over(float x) { return __fdividef(2.0f, x); }

template <typename R>
__device__ __forceinline__ void boris(R w[3], const R Ep[3], const R Bp[3], R hq, R c2)
{
    const R e0 = hq * Ep[0], e1 = hq * Ep[1], e2 = hq * Ep[2];
    const R t0 = w[0] + e0, t1 = w[1] + e1, t2 = w[2] + e2;
    const R s = div_sqrt(hq, t0 * t0 + t1 * t1 + t2 * t2 + c2);
    const R b0 = s * Bp[0], b1 = s * Bp[1], b2 = s * Bp[2];
    const R n0 = t0 + (t1 * b2 - t2 * b1);
    const R n1 = t1 + (t2 * b0 - t0 * b2);
    const R n2 = t2 + (t0 * b1 - t1 * b0);
    const R f = two_over(R(1) + b0 * b0 + b1 * b1 + b2 * b2);
    w[0] = t0 + e0 + f * (n1 * b2 - n2 * b1);
    w[1] = t1 + e1 + f * (n2 * b0 - n0 * b2);
    w[2] = t2 + e2 + f * (n0 * b1 - n1 * b0);
}

// ---------------------------------------------------------------------------
// Offset-to-cell renormalization after a move by delta (|delta| < 1): returns
// the cell shift k and the new offset o' in [0, 1) with cell + o' = old cell +
// o + delta.  The float version forms o + delta - k with two error-free
// TwoSum steps (Knuth) and rounds once, so o' is the float nearest to the exact
// value, as a double-precision renormalization followed by one rounding would
// give, without a single double-precision instruction.  An offset that rounds
// to 1 moves to the next cell with offset 0.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int renormalize(float o, float delta, float &out)
{
    const float s = __fadd_rn(o, delta);
    const float bv = __fsub_rn(s, o);
    const float err1 = __fadd_rn(__fsub_rn(o, __fsub_rn(s, bv)), __fsub_rn(delta, bv));
    const float k = floorf(s);
    const float t = __fsub_rn(s, k);
    const float bt = __fsub_rn(t, s);
    const float err2 = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bt)), __fsub_rn(-k, bt));
    float r = __fadd_rn(t, __fadd_rn(err1, err2));
    int ki = (int)k;
    if (r < 0.f) {
        ki -= 1;
        r = __fadd_rn(r, 1.0f);
    }
    if (r >= 1.f) {
        ki += 1;
        r = __fsub_rn(r, 1.0f);
    }
    out = r;
    return ki;
}

__device__ __forceinline__ int renormalize(double o, double delta, double &out)
{
    const double s = o + delta;
    const double k = floor(s);
    double r = s - k;
    int ki = (int)k;
    if (r >= 1.0) {
        ki += 1;
        r -= 1.0;
    }
    out = r;
    return ki;
}

// ---------------------------------------------------------------------------
// Virtual-path current (Sec. 3.2, Eq. current; Appendix step 2d).  Per axis,
// with the old cloud on cells -1..1 around the old cell and the new one on
// s-1..s+1 (s in {-1,0,1} the cell shift), the window is four cells starting at
// lo = -1 + min(s, 0).  Pp = dF(x^{n+1}) + dF(x^n) and Pm = dF(x^{n+1}) - dF(x^n)
// per window cell, and D[q] = F_f(x^{n+1}) - F_f(x^n) = sum_{w <= q} Pm[w] at the
// face f = lo + q + 1 (q = 0..2; the face after the window has D = 0).
// ---------------------------------------------------------------------------
template <typename R>
struct AxisWin {
    R Pp[4], Pm[4], D[3];
    int lo;
};

// Pm = dF(x^{n+1}) - dF(x^n) on the cells -1..1 of a particle that stayed in
// its cell along this axis (offsets d0 -> d1), in the factored form of the
// differences of the l_a = 1 1/2 weights,
//   (1-d1)^2/2 - (1-d0)^2/2 = -(1/2) dl (2 - d0 - d1),
//   (1/2-d0)^2 - (1/2-d1)^2 =  dl (1 - d0 - d1),
//   d1^2/2 - d0^2/2          =  (1/2) dl (d0 + d1),       dl = d1 - d0,
// which vanishes exactly for a particle at rest and keeps its relative accuracy
// for small displacements (the plain differences cancel).
template <typename R>
__device__ __forceinline__ void still_pm(R d0, R d1, R pm[3])
{
    const R dl = d1 - d0;
    const R sm = d0 + d1;
    pm[0] = R(-0.5) * dl * (R(2) - sm);
    pm[1] = dl * (R(1) - sm);
    pm[2] = R(0.5) * dl * sm;
}

template <typename R>
__device__ __forceinline__ void axis_window(R d0, R d1, int s, AxisWin<R> &a)
{
    R f0[2], S0[3], f1[2], S1[3];
    form_factor(d0, f0, S0);
    form_factor(d1, f1, S1);
    const bool neg = s < 0, pos = s > 0;
    const R o0 = neg ? R(0) : S0[0];
    const R o1 = neg ? S0[0] : S0[1];
    const R o2 = neg ? S0[1] : S0[2];
    const R o3 = neg ? S0[2] : R(0);
    const R n0 = pos ? R(0) : S1[0];
    const R n1 = pos ? S1[0] : S1[1];
    const R n2 = pos ? S1[1] : S1[2];
    const R n3 = pos ? S1[2] : R(0);
    a.Pp[0] = n0 + o0; a.Pm[0] = n0 - o0;
    a.Pp[1] = n1 + o1; a.Pm[1] = n1 - o1;
    a.Pp[2] = n2 + o2; a.Pm[2] = n2 - o2;
    a.Pp[3] = n3 + o3; a.Pm[3] = n3 - o3;
    if (s == 0) {   // no shift along this axis: the factored differences
        R pm[3];
        still_pm(d0, d1, pm);
        a.Pm[0] = pm[0];
        a.Pm[1] = pm[1];
        a.Pm[2] = pm[2];
    }
    a.D[0] = a.Pm[0];
    a.D[1] = a.D[0] + a.Pm[1];
    a.D[2] = a.D[1] + a.Pm[2];
    a.lo = neg ? -2 : -1;
}

// The window of a particle that stayed in its cell along this axis (s = 0):
// cells -1..1 of the old cell, interior faces 0 and 1.  The fourth cell and the
// third face carry nothing (zero weight; the closure sum of Pm), and a
// deposit called with the axis' `full` bit clear never reads them.
template <typename R>
__device__ __forceinline__ void axis_window_still(R d0, R d1, AxisWin<R> &a)
{
    // Pp = S(d1) + S(d0): Pp0 = ((1-d0)^2 + (1-d1)^2)/2, Pp2 = (d0^2 + d1^2)/2 and
    // Pp1 = 2 - Pp0 - Pp2 (the cell integrals sum to one); Pm in the factored
    // form of still_pm with h = (d1 - d0)/2 and s = d0 + d1: Pm0 = h (s - 2),
    // Pm2 = h s, Pm1 = -(Pm0 + Pm2); the face sums D0 = Pm0, D1 = -Pm2.
    const R e0 = R(1) - d0, e1 = R(1) - d1;
    a.Pp[0] = R(0.5) * (e0 * e0 + e1 * e1);
    a.Pp[2] = R(0.5) * (d0 * d0 + d1 * d1);
    a.Pp[1] = (R(2) - a.Pp[0]) - a.Pp[2];
    a.Pp[3] = R(0);
    const R h = R(0.5) * (d1 - d0), sm = d0 + d1;
    a.Pm[0] = h * (sm - R(2));
    a.Pm[2] = h * sm;
    a.Pm[1] = -(a.Pm[0] + a.Pm[2]);
    a.Pm[3] = R(0);
    a.D[0] = a.Pm[0];
    a.D[1] = -a.Pm[2];
    a.D[2] = R(0);
    a.lo = -1;
}

// Current accumulators; offsets are relative to the particle's OLD cell.
template <typename R>
struct SmemAcc {
    R *J[3];
    int base, s1, s2;
    // adds kp * t
    __device__ __forceinline__ void add(int a, int dx, int dy, int dz, R kp, R t) const
    {
        atomicAdd(&J[a][base + dx + s1 * dy + s2 * dz], kp * t);
    }
    // kp0 * t0 at (dx, dy, dz) and kp1 * t1 one cell on along axis ax
    __device__ __forceinline__ void add2(int a, int dx, int dy, int dz, int ax, R kp0, R kp1, R t0, R t1) const
    {
        add(a, dx, dy, dz, kp0, t0);
        add(a, dx + (ax == 0), dy + (ax == 1), dz + (ax == 2), kp1, t1);
    }
};

// FP32 form: the shared current tile accumulates in integer fixed point.
// Shared-memory float atomics run as compare-and-swap loops on this GPU while
// 32-bit integer atomics are native.  A contribution is the product kp*t, where
// the caller's prefactor kp carries a power-of-two scale: q = kp*t (|q| <= 2^33
// for every possible contribution; the host sets the scale).  It is split into
// hi = rint(q/2^16) and lo = rint(q - hi*2^16) (|lo| <= 2^15), both taken from
// the 1.5*2^23 magic-number addition, with the product formed inside the fused
// multiply-adds: magic + hi = fma(kp/2^16, t, magic), then the exact constant
// magic - hi*2^16 = fma(magic + hi, -2^16, magic*(2^16 + 1)) (at most 18
// significant bits), and magic + lo = fma(kp, t, magic - hi*2^16), rounded once
// to an integer because it lies in [2^23, 2^24).  The two integer sums are exact and stay below 2^31 for up to
// 2^13 particles per block; the block converts hi*2^16 + lo back once.
// The words added are the bit patterns of magic + hi and magic + lo, i.e.
// kFixBias + hi and kFixBias + lo.  With SUB the bias is taken off before each
// atomic; without it the block takes N * kFixBias off each word once before the
// flush, N being the number of contributions the word received (known for the
// fixed stencil of a particle that stayed in its cell; integer sums wrap
// modulo 2^32, so the order does not matter).
constexpr unsigned kFixBias = 0x4B400000u;
template <bool SUB>
struct FixedAccT {
    int *hi[3];
    int *lo[3];
    int base, s1, s2;
    __device__ __forceinline__ void add(int a, int dx, int dy, int dz, float kp, float t) const
    {
        const float magic = 12582912.0f;   // 1.5 * 2^23
        const float th = fmaf(kp * (1.0f / 65536.0f), t, magic);   // magic + hi
        const float ch = fmaf(th, -65536.0f, magic * 65537.0f);      // magic - hi * 2^16, exact
        const float tl = fmaf(kp, t, ch);                            // magic + lo, one rounding
        const int idx = base + dx + s1 * dy + s2 * dz;
        atomicAdd(&hi[a][idx], SUB ? __float_as_int(th) - (int)kFixBias : __float_as_int(th));
        atomicAdd(&lo[a][idx], SUB ? __float_as_int(tl) - (int)kFixBias : __float_as_int(tl));
    }
    // The same for two contributions, packed: 128^3 cells of 32 + 32 particles, 12
    // steps, 100.8 ms, 102.9 one by one; 64^3 of 32 + 32 with l_a = 2 1/2, 6 steps, 16.3 and
    // 16.8; the slab 14.7 and 15.2.  (Packing the gather of l_a = 2 1/2 as well cost 1
    // percent.)
    __device__ __forceinline__ void add2(int a, int dx, int dy, int dz, int ax, float kp0, float kp1, float t0,
                                         float t1) const
    {
        const float magic = 12582912.0f, s16 = 1.0f / 65536.0f;
        const F2 t = pack2(t0, t1);
        const F2 th = fma2(pack2(kp0 * s16, kp1 * s16), t, pack2(magic, magic));
        const F2 ch = fma2(th, pack2(-65536.0f, -65536.0f), pack2(magic * 65537.0f, magic * 65537.0f));
        const F2 tl = fma2(pack2(kp0, kp1), t, ch);
        const int i0 = base + dx + s1 * dy + s2 * dz, i1 = i0 + (ax == 0 ? 1 : ax == 1 ? s1 : s2);
        const int off = SUB ? (int)kFixBias : 0;
        atomicAdd(&hi[a][i0], __float_as_int(lo2(th)) - off);
        atomicAdd(&hi[a][i1], __float_as_int(hi2(th)) - off);
        atomicAdd(&lo[a][i0], __float_as_int(lo2(tl)) - off);
        atomicAdd(&lo[a][i1], __float_as_int(hi2(tl)) - off);
    }
};
using FixedAcc = FixedAccT<true>;

// Current accumulator on the periodic global arrays for one particle's windows:
// the wrapped offsets of the window's NW cells along each axis (from lo) are
// formed once, so that a contribution costs one index sum and one atomic.
template <typename R, int NW>
struct GlobalAcc {
    R *J[3];
    long long xw[NW], yw[NW], zw[NW];
    int lox, loy, loz;
    __device__ __forceinline__ void set(long long cb, int i, int j, int k, int nx, int ny, int nz, int lx, int ly,
                                        int lz, bool three)
    {
        lox = lx;
        loy = ly;
        loz = three ? lz : 0;
#pragma unroll
        for (int m = 0; m < NW; ++m) {
            xw[m] = cb + wrapi(i + lox + m, nx);
            yw[m] = (long long)nx * wrapi(j + loy + m, ny);
            zw[m] = three ? (long long)nx * ny * wrapi(k + loz + m, nz) : 0;
        }
    }
    __device__ __forceinline__ void add(int a, int dx, int dy, int dz, R kp, R t) const
    {
        atomicAdd(&J[a][xw[dx - lox] + yw[dy - loy] + zw[dz - loz]], kp * t);
    }
    __device__ __forceinline__ void add2(int a, int dx, int dy, int dz, int ax, R kp0, R kp1, R t0, R t1) const
    {
        add(a, dx, dy, dz, kp0, t0);
        add(a, dx + (ax == 0), dy + (ax == 1), dz + (ax == 2), kp1, t1);
    }
};

// Deposit one particle.  kf[a] = -(1/4)(d_a/dt) q_p/V in 3D and -(1/2)(d_a/dt) q_p/V
// (a = x, y) with kf[2] = (1/4) q_p/V in 2D (reading of Eq. current summed
// over the ignorable z: xi^x = -(1/2)(dx/dt) D_x Pp_y, xi^z = (1/4) u_z [Pp Pp + Pm Pm/3]).
// Bit a of `full` is clear when no particle handled by the warp changed cell
// along axis a: then every window's fourth cell along a carries zero weight and
// its third face only the closure sum of Pm (zero up to rounding; the window
// of an unshifted particle has two interior faces), and those contributions are
// skipped.  The flag is warp-uniform, so the skip is a uniform branch.
// only (warp-uniform): the one component to deposit, or -1 for all three.
template <int DIM, typename R, class Acc>
__device__ __forceinline__ void deposit(const Acc &acc, const AxisWin<R> &X, const AxisWin<R> &Y, const AxisWin<R> &Z,
                                        const R kf[3], R uz, int full, int only = -1)
{
    const R third = R(1) / R(3);
    const bool fx = full & 1, fy = full & 2, fz = full & 4;
    if (DIM == 3) {
        if (only < 0 || only == 0) {
#pragma unroll
            for (int wz = 0; wz < 4; ++wz) {
                if (wz == 3 && !fz) continue;
#pragma unroll
                for (int wy = 0; wy < 4; ++wy) {
                    if (wy == 3 && !fy) continue;
                    const R T = Y.Pp[wy] * Z.Pp[wz] + third * Y.Pm[wy] * Z.Pm[wz];
                    acc.add2(0, X.lo + 1, Y.lo + wy, Z.lo + wz, 0, kf[0] * X.D[0], kf[0] * X.D[1], T, T);
                    if (fx) acc.add(0, X.lo + 3, Y.lo + wy, Z.lo + wz, kf[0] * X.D[2], T);
                }
            }
        }
        if (only < 0 || only == 1) {
#pragma unroll
            for (int wz = 0; wz < 4; ++wz) {
                if (wz == 3 && !fz) continue;
#pragma unroll
                for (int wx = 0; wx < 4; ++wx) {
                    if (wx == 3 && !fx) continue;
                    const R T = X.Pp[wx] * Z.Pp[wz] + third * X.Pm[wx] * Z.Pm[wz];
                    acc.add2(1, X.lo + wx, Y.lo + 1, Z.lo + wz, 1, kf[1] * Y.D[0], kf[1] * Y.D[1], T, T);
                    if (fy) acc.add(1, X.lo + wx, Y.lo + 3, Z.lo + wz, kf[1] * Y.D[2], T);
                }
            }
        }
        if (only < 0 || only == 2) {
#pragma unroll
            for (int wy = 0; wy < 4; ++wy) {
                if (wy == 3 && !fy) continue;
#pragma unroll
                for (int wx = 0; wx < 4; ++wx) {
                    if (wx == 3 && !fx) continue;
                    const R T = X.Pp[wx] * Y.Pp[wy] + third * X.Pm[wx] * Y.Pm[wy];
                    acc.add2(2, X.lo + wx, Y.lo + wy, Z.lo + 1, 2, kf[2] * Z.D[0], kf[2] * Z.D[1], T, T);
                    if (fz) acc.add(2, X.lo + wx, Y.lo + wy, Z.lo + 3, kf[2] * Z.D[2], T);
                }
            }
        }
    } else {
        if (only < 0 || only == 0) {
#pragma unroll
            for (int wy = 0; wy < 4; ++wy) {
                if (wy == 3 && !fy) continue;
                const R t = kf[0] * Y.Pp[wy];
                acc.add2(0, X.lo + 1, Y.lo + wy, 0, 0, t, t, X.D[0], X.D[1]);
                if (fx) acc.add(0, X.lo + 3, Y.lo + wy, 0, t, X.D[2]);
            }
        }
        if (only < 0 || only == 1) {
#pragma unroll
            for (int wx = 0; wx < 4; ++wx) {
                if (wx == 3 && !fx) continue;
                const R t = kf[1] * X.Pp[wx];
                acc.add2(1, X.lo + wx, Y.lo + 1, 0, 1, t, t, Y.D[0], Y.D[1]);
                if (fy) acc.add(1, X.lo + wx, Y.lo + 3, 0, t, Y.D[2]);
            }
        }
        const R kz = kf[2] * uz;
        if (only < 0 || only == 2) {
#pragma unroll
            for (int wy = 0; wy < 4; ++wy) {
                if (wy == 3 && !fy) continue;
                R T[4];
#pragma unroll
                for (int wx = 0; wx < 4; ++wx) T[wx] = X.Pp[wx] * Y.Pp[wy] + third * X.Pm[wx] * Y.Pm[wy];
                acc.add2(2, X.lo, Y.lo + wy, 0, 0, kz, kz, T[0], T[1]);
                acc.add(2, X.lo + 2, Y.lo + wy, 0, kz, T[2]);
                if (fx) acc.add(2, X.lo + 3, Y.lo + wy, 0, kz, T[3]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Alternating-order form factor l_a = 2 1/2 (Sec. 4.5).  The base index is
// ib = int(x_p + 1/2) with d = x_p + 1/2 - ib; the point values f = f^(2) at
// the integer points ib-1, ib, ib+1 are ((1-d)^2/2, 3/4 - (1/2-d)^2, d^2/2) and
// the cell integrals S = f^(3) over the cells ib-2 .. ib+1 (centres
// ib-3/2 .. ib+3/2) are the cubic B-spline values
//   ((1-d)^3/6, (4 - 6d^2 + 3d^3)/6, (1 + 3d + 3d^2 - 3d^3)/6, d^3/6),
// the second and third being the paper's (2-d)^3/6 - 2(1-d)^3/3 and
// (1+d)^3/6 - 2d^3/3 multiplied out.  From the stored (cell, offset o):
// ib = cell + (o >= 1/2), d = o + 1/2 - (o >= 1/2).
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ int split5(R o, R &d)
{
    const int up = o >= R(0.5) ? 1 : 0;
    d = up ? o - R(0.5) : o + R(0.5);
    return up;
}

template <typename R>
__device__ __forceinline__ void form_factor5(R d, R f[3], R S[4])
{
    const R h = R(0.5), s6 = R(1) / R(6);
    const R e = R(1) - d, m = h - d, d2 = d * d;
    f[0] = h * e * e;
    f[1] = R(0.75) - m * m;
    f[2] = h * d2;
    S[0] = s6 * e * e * e;
    S[1] = s6 * (R(4) + d2 * (R(3) * d - R(6)));
    S[2] = s6 * (R(1) + R(3) * d * (R(1) + d - d2));
    S[3] = s6 * d2 * d;
}

// Gather with l_a = 2 1/2 (Eqs. alphax, betax with f^(2) and f^(3)); reader
// offsets are relative to the base index ib: f index a sits at a - 1, S index
// b at b - 2.  2D drops every z factor.
template <int DIM, typename R, class Rd>
__device__ __forceinline__ void gather5(const Rd &rd, const R fx[3], const R Sx[4], const R fy[3], const R Sy[4],
                                        const R fz[3], const R Sz[4], R Ep[3], R Bp[3])
{
    constexpr int NZS = DIM == 3 ? 4 : 1, NZF = DIM == 3 ? 3 : 1;
    R ex = 0, ey = 0, ez = 0, bx = 0, by = 0, bz = 0;
    // The z planes are a loop, not unrolled: unrolled, the 252 taps of the
    // 3D gather need more than the 128 registers of two blocks per SM and spill.
#pragma unroll 1
    for (int c = 0; c < NZS; ++c) {   // S along z: E^x, E^y, B^z
        const R wz = DIM == 3 ? (c == 0 ? Sz[0] : c == 1 ? Sz[1] : c == 2 ? Sz[2] : Sz[3]) : R(1);
        const int oz = DIM == 3 ? c - 2 : 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const R t = fx[0] * rd.e(0, -1, b - 2, oz) + fx[1] * rd.e(0, 0, b - 2, oz) + fx[2] * rd.e(0, 1, b - 2, oz);
            ex += Sy[b] * wz * t;
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R t = Sx[0] * rd.e(1, -2, b - 1, oz) + Sx[1] * rd.e(1, -1, b - 1, oz) +
                        Sx[2] * rd.e(1, 0, b - 1, oz) + Sx[3] * rd.e(1, 1, b - 1, oz);
            ey += fy[b] * wz * t;
            const R u = fx[0] * rd.b(2, -1, b - 1, oz) + fx[1] * rd.b(2, 0, b - 1, oz) + fx[2] * rd.b(2, 1, b - 1, oz);
            bz += fy[b] * wz * u;
        }
    }
#pragma unroll 1
    for (int c = 0; c < NZF; ++c) {   // f along z: E^z, B^x, B^y
        const R wz = DIM == 3 ? (c == 0 ? fz[0] : c == 1 ? fz[1] : fz[2]) : R(1);
        const int oz = DIM == 3 ? c - 1 : 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const R t = Sx[0] * rd.e(2, -2, b - 2, oz) + Sx[1] * rd.e(2, -1, b - 2, oz) +
                        Sx[2] * rd.e(2, 0, b - 2, oz) + Sx[3] * rd.e(2, 1, b - 2, oz);
            ez += Sy[b] * wz * t;
            const R u = fx[0] * rd.b(1, -1, b - 2, oz) + fx[1] * rd.b(1, 0, b - 2, oz) + fx[2] * rd.b(1, 1, b - 2, oz);
            by += Sy[b] * wz * u;
        }
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R t = Sx[0] * rd.b(0, -2, b - 1, oz) + Sx[1] * rd.b(0, -1, b - 1, oz) +
                        Sx[2] * rd.b(0, 0, b - 1, oz) + Sx[3] * rd.b(0, 1, b - 1, oz);
            bx += fy[b] * wz * t;
        }
    }
    Ep[0] = ex; Ep[1] = ey; Ep[2] = ez;
    Bp[0] = bx; Bp[1] = by; Bp[2] = bz;
}

// Gather of the comparison scheme of Eq. wrong1 (Sec. 5, the "conventional"
// uniform-order l = 2 interpolation): the l_a = 1 1/2 cell integrals S at the
// cells -1..1 of the particle's cell, and at the integer points -1..2 the mean
// of the two neighbouring cell integrals, g = (S0/2, (S0+S1)/2, (S1+S2)/2, S2/2).
// Reader offsets are relative to the cell.  2D drops every z factor.
template <typename R>
__device__ __forceinline__ void wrong1_points(const R S[3], R g[4])
{
    const R h = R(0.5);
    g[0] = h * S[0];
    g[1] = h * (S[0] + S[1]);
    g[2] = h * (S[1] + S[2]);
    g[3] = h * S[2];
}

template <int DIM, typename R, class Rd>
__device__ __forceinline__ void gather_w1(const Rd &rd, const R Sx[3], const R Sy[3], const R Sz[3], R Ep[3],
                                          R Bp[3])
{
    R gx[4], gy[4], gz[4];
    wrong1_points(Sx, gx);
    wrong1_points(Sy, gy);
    wrong1_points(Sz, gz);
    constexpr int NZS = DIM == 3 ? 3 : 1, NZG = DIM == 3 ? 4 : 1;
    R ex = 0, ey = 0, ez = 0, bx = 0, by = 0, bz = 0;
    // The z planes are a loop, not unrolled: unrolled, the 132 taps of the
    // 3D gather need more than the 128 registers of two blocks per SM and spill.
#pragma unroll 1
    for (int c = 0; c < NZS; ++c) {   // S along z: E^x, E^y, B^z
        const R wz = DIM == 3 ? (c == 0 ? Sz[0] : c == 1 ? Sz[1] : Sz[2]) : R(1);
        const int oz = DIM == 3 ? c - 1 : 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R t = gx[0] * rd.e(0, -1, b - 1, oz) + gx[1] * rd.e(0, 0, b - 1, oz) +
                        gx[2] * rd.e(0, 1, b - 1, oz) + gx[3] * rd.e(0, 2, b - 1, oz);
            ex += Sy[b] * wz * t;
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const R t = Sx[0] * rd.e(1, -1, b - 1, oz) + Sx[1] * rd.e(1, 0, b - 1, oz) + Sx[2] * rd.e(1, 1, b - 1, oz);
            ey += gy[b] * wz * t;
            const R u = gx[0] * rd.b(2, -1, b - 1, oz) + gx[1] * rd.b(2, 0, b - 1, oz) +
                        gx[2] * rd.b(2, 1, b - 1, oz) + gx[3] * rd.b(2, 2, b - 1, oz);
            bz += gy[b] * wz * u;
        }
    }
#pragma unroll 1
    for (int c = 0; c < NZG; ++c) {   // g along z: E^z, B^x, B^y
        const R wz = DIM == 3 ? (c == 0 ? gz[0] : c == 1 ? gz[1] : c == 2 ? gz[2] : gz[3]) : R(1);
        const int oz = DIM == 3 ? c - 1 : 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R t = Sx[0] * rd.e(2, -1, b - 1, oz) + Sx[1] * rd.e(2, 0, b - 1, oz) + Sx[2] * rd.e(2, 1, b - 1, oz);
            ez += Sy[b] * wz * t;
            const R u = gx[0] * rd.b(1, -1, b - 1, oz) + gx[1] * rd.b(1, 0, b - 1, oz) +
                        gx[2] * rd.b(1, 1, b - 1, oz) + gx[3] * rd.b(1, 2, b - 1, oz);
            by += Sy[b] * wz * u;
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const R t = Sx[0] * rd.b(0, -1, b - 1, oz) + Sx[1] * rd.b(0, 0, b - 1, oz) + Sx[2] * rd.b(0, 1, b - 1, oz);
            bx += gy[b] * wz * t;
        }
    }
    Ep[0] = ex; Ep[1] = ey; Ep[2] = ez;
    Bp[0] = bx; Bp[1] = by; Bp[2] = bz;
}

template <typename R>
struct GlobalReader5 {       // periodic global arrays, offsets -2..2 from the base index
    const R *E[3];
    const R *B[3];
    long long xi[5], yj[5], zk[5];
    __device__ __forceinline__ long long at(int dx, int dy, int dz) const { return xi[dx + 2] + yj[dy + 2] + zk[dz + 2]; }
    __device__ __forceinline__ R e(int a, int dx, int dy, int dz) const { return E[a][at(dx, dy, dz)]; }
    __device__ __forceinline__ R b(int a, int dx, int dy, int dz) const { return B[a][at(dx, dy, dz)]; }
};

// Deposit window of one axis with l_a = 2 1/2: the cells lo .. lo+4 relative to
// the old base index (lo = -2, or -3 when the base index moved down), the old
// and new cell integrals laid on it, Pp/Pm = new +- old, and the partial sums
// D[q] = sum_{w <= q} Pm[w] at the faces lo+q+1 (q = 0..3; the face after the
// last cell carries the closure sum only).
template <typename R>
struct AxisWin5 {
    R Pp[5], Pm[5], D[4];
    int lo;
};

template <typename R>
__device__ __forceinline__ void axis_window5(R d0, R d1, int s, AxisWin5<R> &a)
{
    R f0[3], S0[4], f1[3], S1[4];
    form_factor5(d0, f0, S0);
    form_factor5(d1, f1, S1);
    const bool neg = s < 0, pos = s > 0;
    R o[5], n[5];
#pragma unroll
    for (int w = 0; w < 5; ++w) {
        o[w] = neg ? (w == 0 ? R(0) : S0[w - 1]) : (w == 4 ? R(0) : S0[w]);
        n[w] = pos ? (w == 0 ? R(0) : S1[w - 1]) : (w == 4 ? R(0) : S1[w]);
    }
#pragma unroll
    for (int w = 0; w < 5; ++w) {
        a.Pp[w] = n[w] + o[w];
        a.Pm[w] = n[w] - o[w];
    }
    a.D[0] = a.Pm[0];
#pragma unroll
    for (int q = 1; q < 4; ++q) a.D[q] = a.D[q - 1] + a.Pm[q];
    a.lo = neg ? -3 : -2;
}

// Deposit of one particle with l_a = 2 1/2 (Eq. current on the 5-cell windows;
// the prefactors kf as for deposit()).  Bit a of `full` clear: no particle of
// the warp moved its base index along a, so the fifth window cell and the
// fourth face (the closure) are skipped.
template <int DIM, typename R, class Acc>
__device__ __forceinline__ void deposit5(const Acc &acc, const AxisWin5<R> &X, const AxisWin5<R> &Y,
                                         const AxisWin5<R> &Z, const R kf[3], R uz, int full, int only = -1)
{
    const R third = R(1) / R(3);
    const bool fx = full & 1, fy = full & 2, fz = full & 4;
    if (DIM == 3) {
        if (only < 0 || only == 0) {
#pragma unroll
            for (int wz = 0; wz < 5; ++wz) {
                if (wz == 4 && !fz) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {   // two cells of the axis at a time
                    const int wy = 2 * h;
                    const R T0 = Y.Pp[wy] * Z.Pp[wz] + third * Y.Pm[wy] * Z.Pm[wz];
                    const R T1 = Y.Pp[wy + 1] * Z.Pp[wz] + third * Y.Pm[wy + 1] * Z.Pm[wz];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q == 3 && !fx) continue;
                        acc.add2(0, X.lo + 1 + q, Y.lo + wy, Z.lo + wz, 1, kf[0] * X.D[q], kf[0] * X.D[q], T0, T1);
                    }
                }
                if (fy) {
                    const int wy = 4;
                    const R T = Y.Pp[wy] * Z.Pp[wz] + third * Y.Pm[wy] * Z.Pm[wz];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q == 3 && !fx) continue;
                        acc.add(0, X.lo + 1 + q, Y.lo + wy, Z.lo + wz, kf[0] * X.D[q], T);
                    }
                }
            }
        }
        if (only < 0 || only == 1) {
#pragma unroll
            for (int wz = 0; wz < 5; ++wz) {
                if (wz == 4 && !fz) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {   // two cells of the axis at a time
                    const int wx = 2 * h;
                    const R T0 = X.Pp[wx] * Z.Pp[wz] + third * X.Pm[wx] * Z.Pm[wz];
                    const R T1 = X.Pp[wx + 1] * Z.Pp[wz] + third * X.Pm[wx + 1] * Z.Pm[wz];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q == 3 && !fy) continue;
                        acc.add2(1, X.lo + wx, Y.lo + 1 + q, Z.lo + wz, 0, kf[1] * Y.D[q], kf[1] * Y.D[q], T0, T1);
                    }
                }
                if (fx) {
                    const int wx = 4;
                    const R T = X.Pp[wx] * Z.Pp[wz] + third * X.Pm[wx] * Z.Pm[wz];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q == 3 && !fy) continue;
                        acc.add(1, X.lo + wx, Y.lo + 1 + q, Z.lo + wz, kf[1] * Y.D[q], T);
                    }
                }
            }
        }
        if (only < 0 || only == 2) {
#pragma unroll
            for (int wy = 0; wy < 5; ++wy) {
                if (wy == 4 && !fy) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {   // two cells of the axis at a time
                    const int wx = 2 * h;
                    const R T0 = X.Pp[wx] * Y.Pp[wy] + third * X.Pm[wx] * Y.Pm[wy];
                    const R T1 = X.Pp[wx + 1] * Y.Pp[wy] + third * X.Pm[wx + 1] * Y.Pm[wy];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q == 3 && !fz) continue;
                        acc.add2(2, X.lo + wx, Y.lo + wy, Z.lo + 1 + q, 0, kf[2] * Z.D[q], kf[2] * Z.D[q], T0, T1);
                    }
                }
                if (fx) {
                    const int wx = 4;
                    const R T = X.Pp[wx] * Y.Pp[wy] + third * X.Pm[wx] * Y.Pm[wy];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q == 3 && !fz) continue;
                        acc.add(2, X.lo + wx, Y.lo + wy, Z.lo + 1 + q, kf[2] * Z.D[q], T);
                    }
                }
            }
        }
    } else {
        if (only < 0 || only == 0) {
#pragma unroll
            for (int wy = 0; wy < 5; ++wy) {
                if (wy == 4 && !fy) continue;
                const R t = kf[0] * Y.Pp[wy];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q == 3 && !fx) continue;
                    acc.add(0, X.lo + 1 + q, Y.lo + wy, 0, t, X.D[q]);
                }
            }
        }
        if (only < 0 || only == 1) {
#pragma unroll
            for (int wx = 0; wx < 5; ++wx) {
                if (wx == 4 && !fx) continue;
                const R t = kf[1] * X.Pp[wx];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q == 3 && !fy) continue;
                    acc.add(1, X.lo + wx, Y.lo + 1 + q, 0, t, Y.D[q]);
                }
            }
        }
        const R kz = kf[2] * uz;
        if (only < 0 || only == 2) {
#pragma unroll
            for (int wy = 0; wy < 5; ++wy) {
                if (wy == 4 && !fy) continue;
#pragma unroll
                for (int wx = 0; wx < 5; ++wx) {
                    if (wx == 4 && !fx) continue;
                    const R T = X.Pp[wx] * Y.Pp[wy] + third * X.Pm[wx] * Y.Pm[wy];
                    acc.add(2, X.lo + wx, Y.lo + wy, 0, kz, T);
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// 3D deposit (l_a = 1 1/2) of a particle whose cell moved along one axis only,
// written for that axis, A, and the two after it, B and C, so that the lanes of a
// warp may hold different axes: strides, prefactors and component arrays are the
// lane's.  B and C have three cells and two faces, A four and three: 75
// contributions instead of 144.  J[c]: the component along A, B, C; b0: the first
// cell of all three windows; s: strides.  only: as for deposit().
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void deposit_one_axis(R *const J[3], const AxisWin<R> &A, const AxisWin<R> &B,
                                                 const AxisWin<R> &C, const R kf[3], int b0, const int s[3], int only)
{
    const R third = R(1) / R(3);
    if (only < 0 || only == 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const R T = B.Pp[b] * C.Pp[c] + third * B.Pm[b] * C.Pm[c];
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    atomicAdd(J[0] + b0 + (1 + q) * s[0] + b * s[1] + c * s[2], kf[0] * A.D[q] * T);
            }
    }
    if (only < 0 || only == 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const R T = A.Pp[a] * C.Pp[c] + third * A.Pm[a] * C.Pm[c];
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    atomicAdd(J[1] + b0 + a * s[0] + (1 + q) * s[1] + c * s[2], kf[1] * B.D[q] * T);
            }
    }
    if (only < 0 || only == 2) {
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const R T = A.Pp[a] * B.Pp[b] + third * A.Pm[a] * B.Pm[b];
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    atomicAdd(J[2] + b0 + a * s[0] + b * s[1] + (1 + q) * s[2], kf[2] * C.D[q] * T);
            }
    }
}

// ---------------------------------------------------------------------------
// Yee updates of one cell l of run rn (Appendix, Eqs. updateB and escheme,
// completed cyclically; in 2D every z difference vanishes).
//   B half step:  Bx[i,j,k] -= (c_y/2)(Ez[i,j,k]-Ez[i,j-1,k]) - (c_z/2)(Ey[i,j,k]-Ey[i,j,k-1])
//                 By[i,j,k] -= (c_z/2)(Ex[i,j,k]-Ex[i,j,k-1]) - (c_x/2)(Ez[i,j,k]-Ez[i-1,j,k])
//                 Bz[i,j,k] -= (c_x/2)(Ey[i,j,k]-Ey[i-1,j,k]) - (c_y/2)(Ex[i,j,k]-Ex[i,j-1,k])
//   E full step:  Ex += -4 pi dt Jx + c_y(Bz[i,j+1,k]-Bz[i,j,k]) - c_z(By[i,j,k+1]-By[i,j,k])
//                 Ey += -4 pi dt Jy + c_z(Bx[i,j,k+1]-Bx[i,j,k]) - c_x(Bz[i+1,j,k]-Bz[i,j,k])
//                 Ez += -4 pi dt Jz + c_x(By[i+1,j,k]-By[i,j,k]) - c_y(Bx[i,j+1,k]-Bx[i,j,k])
// With zero_j the B pass also clears J for the coming deposit.
// ---------------------------------------------------------------------------
// The antenna's incident field at x (cell units) and time t (include/pic.h).
__device__ __forceinline__ double antenna_field(const RunDev &rn, double x, double t)
{
    const double tau = t - (x - rn.ant_i0) * rn.d[0] / rn.c;
    if (tau <= 0.0) return 0.0;
    double g = 1.0;
    if (tau < rn.ant_ramp) {
        const double s = sin(1.5707963267948966 * tau / rn.ant_ramp);
        g = s * s;
    }
    return rn.ant_E0 * g * sin(rn.ant_omega * tau);
}

// v + k f, rounded as the precision's other field sums are.
__device__ __forceinline__ double add_incident(double v, double k, double f) { return fma(k, f, v); }
__device__ __forceinline__ float add_incident(float v, double k, double f) { return v + (float)(k * f); }

// The cell indices of cell l of a run.  Without quotients, which set the Yee kernels'
// time (256x64x64 cells FP32: 20.9 us per B half step and 24.0 us per E step, 48 and
// 60 bytes per cell), and in 64 bits, since a run without particles may have 2^31
// cells and more.
__host__ __device__ __forceinline__ void yee_ijk(const RunDev &rn, long long l, int &i, int &j, int &k)
{
    const long long r = div_cells(l, rn.inv_nx);
    i = (int)(l - r * rn.n[0]);
    k = (int)div_cells(r, rn.inv_ny);
    j = (int)(r - (long long)k * rn.n[1]);
}

// The B half step's new values at a cell, h = c dt/(2 d): the fused multiply-adds
// are written out, so that the two passes and the one pass round alike and a
// run's fields do not depend on how its steps are split into calls.
template <int DIM, typename R>
__device__ __forceinline__ R yee_bx(R b, R hy, R hz, R ez, R ez_j, R ey, R ey_k)
{
    b = fma(-hy, ez - ez_j, b);
    return DIM == 3 ? fma(hz, ey - ey_k, b) : b;
}
template <int DIM, typename R>
__device__ __forceinline__ R yee_by(R b, R hx, R hz, R ez, R ez_i, R ex, R ex_k)
{
    b = fma(hx, ez - ez_i, b);
    return DIM == 3 ? fma(-hz, ex - ex_k, b) : b;
}
template <typename R>
__device__ __forceinline__ R yee_bz(R b, R hx, R hy, R ey, R ey_i, R ex, R ex_j)
{
    return fma(hy, ex - ex_j, fma(-hx, ey - ey_i, b));
}

// ant_n: the antenna clock of the run (E steps since the antenna was set).
template <int DIM, typename R>
__device__ __forceinline__ void yee_b_half_cell(const RunDev &rn, const Fields<R> &F, long long l, int zero_j,
                                                long long ant_n)
{
    const int nx = rn.n[0], ny = rn.n[1], nz = rn.n[2];
    int i, j, k;
    yee_ijk(rn, l, i, j, k);
    const long long p = rn.cell_base + l;
    const long long pim = p + (i == 0 ? nx - 1 : -1);
    const long long pjm = p + (long long)nx * (j == 0 ? ny - 1 : -1);
    const bool f32 = sizeof(R) == 4;
    const R hx = f32 ? R(0.5f * rn.cNf[0]) : R(0.5 * rn.cN[0]), hy = f32 ? R(0.5f * rn.cNf[1]) : R(0.5 * rn.cN[1]);
    const R hz = f32 ? R(0.5f * rn.cNf[2]) : R(0.5 * rn.cN[2]);
    const long long pkm = DIM == 3 ? p + (long long)nx * ny * (k == 0 ? nz - 1 : -1) : p;
    const R ex = F.E[0][p], ey = F.E[1][p], ez = F.E[2][p];
    const R bx = yee_bx<DIM>(F.B[0][p], hy, hz, ez, F.E[2][pjm], ey, DIM == 3 ? F.E[1][pkm] : R(0));
    R by = yee_by<DIM>(F.B[1][p], hx, hz, ez, F.E[2][pim], ex, DIM == 3 ? F.E[0][pkm] : R(0));
    R bz = yee_bz(F.B[2][p], hx, hy, ey, F.E[1][pim], ex, F.E[0][pjm]);
    if (rn.ant_pol != 0 && i == rn.ant_i0) {
        // the scattered-field E node at x = i0 - 1/2 lacks the incident wave
        const double h = 0.5 * rn.cN[0], f = antenna_field(rn, rn.ant_i0 - 0.5, ant_n * rn.dt);
        if (rn.ant_pol == 1) bz = add_incident(bz, h, f); else by = add_incident(by, -h, f);
    }
    F.B[0][p] = bx;
    F.B[1][p] = by;
    F.B[2][p] = bz;
    if (zero_j) {
        F.J[0][p] = R(0);
        F.J[1][p] = R(0);
        F.J[2][p] = R(0);
    }
}

// The E step's new values at a cell from B (own cell and its + neighbours).
template <int DIM, typename R>
__device__ __forceinline__ void yee_e_values(const RunDev &rn, const R e0[3], const R J[3], R bx, R by, R bz, R bz_j,
                                             R by_k, R bz_i, R bx_k, R by_i, R bx_j, int i, long long ant_n, R e[3])
{
    const bool f32 = sizeof(R) == 4;
    const R cx = f32 ? R(rn.cNf[0]) : R(rn.cN[0]), cy = f32 ? R(rn.cNf[1]) : R(rn.cN[1]);
    const R fp = f32 ? R(rn.fpdtf) : R(rn.fpdt);
    e[0] = fma(cy, bz_j - bz, fma(-fp, J[0], e0[0]));
    e[1] = fma(-cx, bz_i - bz, fma(-fp, J[1], e0[1]));
    e[2] = fma(-cy, bx_j - bx, fma(cx, by_i - by, fma(-fp, J[2], e0[2])));
    if (DIM == 3) {
        const R cz = f32 ? R(rn.cNf[2]) : R(rn.cN[2]);
        e[0] = fma(-cz, by_k - by, e[0]);
        e[1] = fma(cz, bx_k - bx, e[1]);
    }
    if (rn.ant_pol != 0 && i == rn.ant_i0 - 1) {
        // the scattered-field E node at x = i0 - 1/2 sees the total-field B node at
        // x = i0, whose incident part (B_z = E_inc, B_y = -E_inc) comes off
        const double f = antenna_field(rn, rn.ant_i0, (ant_n + 0.5) * rn.dt);
        if (rn.ant_pol == 1) e[1] = add_incident(e[1], rn.cN[0], f); else e[2] = add_incident(e[2], rn.cN[0], f);
    }
}

template <int DIM, typename R>
__device__ __forceinline__ void yee_e_cell(const RunDev &rn, const Fields<R> &F, long long l, long long ant_n)
{
    const int nx = rn.n[0], ny = rn.n[1], nz = rn.n[2];
    int i, j, k;
    yee_ijk(rn, l, i, j, k);
    const long long p = rn.cell_base + l;
    const long long pip = p + (i == nx - 1 ? -(nx - 1) : 1);
    const long long pjp = p + (long long)nx * (j == ny - 1 ? -(ny - 1) : 1);
    const long long pkp = DIM == 3 ? p + (long long)nx * ny * (k == nz - 1 ? -(nz - 1) : 1) : p;
    const R e0[3] = {F.E[0][p], F.E[1][p], F.E[2][p]}, J[3] = {F.J[0][p], F.J[1][p], F.J[2][p]};
    R e[3];
    yee_e_values<DIM, R>(rn, e0, J, F.B[0][p], F.B[1][p], F.B[2][p], F.B[2][pjp], DIM == 3 ? F.B[1][pkp] : R(0),
                         F.B[2][pip], DIM == 3 ? F.B[0][pkp] : R(0), F.B[1][pip], F.B[0][pjp], i, ant_n, e);
    F.E[0][p] = e[0];
    F.E[1][p] = e[1];
    F.E[2][p] = e[2];
}

// The second B half step and the E step in one pass, from the fields F to the
// fields O (E and B of F stay as they are, so no cell sees a neighbour's new
// value): a cell's thread forms the new B at its own cell and the six values
// that its E needs at the + neighbours, with the arithmetic of the two passes.
template <int DIM, typename R>
__device__ __forceinline__ void yee_b_half_e_cell(const RunDev &rn, const Fields<R> &F, const Fields<R> &O, long long l,
                                                  long long ant_n)
{
    const int nx = rn.n[0], ny = rn.n[1], nz = rn.n[2];
    int i, j, k;
    yee_ijk(rn, l, i, j, k);
    const long long p = rn.cell_base + l;
    const bool f32 = sizeof(R) == 4;
    const R hx = f32 ? R(0.5f * rn.cNf[0]) : R(0.5 * rn.cN[0]), hy = f32 ? R(0.5f * rn.cNf[1]) : R(0.5 * rn.cN[1]);
    const R hz = f32 ? R(0.5f * rn.cNf[2]) : R(0.5 * rn.cN[2]);
    // offsets to the neighbours along each axis
    const long long im = i == 0 ? nx - 1 : -1, ip = i == nx - 1 ? -(nx - 1) : 1;
    const long long jm = (long long)nx * (j == 0 ? ny - 1 : -1), jp = (long long)nx * (j == ny - 1 ? -(ny - 1) : 1);
    const long long nxy = (long long)nx * ny;
    const long long km = DIM == 3 ? nxy * (k == 0 ? nz - 1 : -1) : 0;
    const long long kp = DIM == 3 ? nxy * (k == nz - 1 ? -(nz - 1) : 1) : 0;
    // the new B of the cell at q whose neighbours below are at qi, qj, qk
    auto nbx = [&](long long q, long long qj, long long qk) {
        return yee_bx<DIM>(F.B[0][q], hy, hz, F.E[2][q], F.E[2][qj], DIM == 3 ? F.E[1][q] : R(0),
                           DIM == 3 ? F.E[1][qk] : R(0));
    };
    auto nby = [&](long long q, long long qi, long long qk) {
        return yee_by<DIM>(F.B[1][q], hx, hz, F.E[2][q], F.E[2][qi], DIM == 3 ? F.E[0][q] : R(0),
                           DIM == 3 ? F.E[0][qk] : R(0));
    };
    auto nbz = [&](long long q, long long qi, long long qj) {
        return yee_bz(F.B[2][q], hx, hy, F.E[1][q], F.E[1][qi], F.E[0][q], F.E[0][qj]);
    };
    R bx = nbx(p, p + jm, p + km), by = nby(p, p + im, p + km), bz = nbz(p, p + im, p + jm);
    R bx_j = nbx(p + jp, p, p + jp + km), bz_j = nbz(p + jp, p + jp + im, p);
    R by_i = nby(p + ip, p, p + ip + km), bz_i = nbz(p + ip, p, p + ip + jm);
    R bx_k = R(0), by_k = R(0);
    if (DIM == 3) {
        bx_k = nbx(p + kp, p + kp + jm, p);
        by_k = nby(p + kp, p + kp + im, p);
    }
    if (rn.ant_pol != 0 && (i == rn.ant_i0 || i + 1 == rn.ant_i0)) {
        // the scattered-field E node at x = i0 - 1/2 lacks the incident wave
        // (1 <= i0 < nx, so the + neighbour along x at i0 is not across the wrap)
        const double h = 0.5 * rn.cN[0], f = antenna_field(rn, rn.ant_i0 - 0.5, ant_n * rn.dt);
        const bool z = rn.ant_pol == 1;
        auto add = [&](R &v) { v = add_incident(v, z ? h : -h, f); };
        if (i == rn.ant_i0) {
            if (z) { add(bz); add(bz_j); } else { add(by); add(by_k); }
        } else {
            if (z) add(bz_i); else add(by_i);
        }
    }
    const R e0[3] = {F.E[0][p], F.E[1][p], F.E[2][p]}, J[3] = {F.J[0][p], F.J[1][p], F.J[2][p]};
    R e[3];
    yee_e_values<DIM, R>(rn, e0, J, bx, by, bz, bz_j, by_k, bz_i, bx_k, by_i, bx_j, i, ant_n, e);
    O.B[0][p] = bx;
    O.B[1][p] = by;
    O.B[2][p] = bz;
    O.E[0][p] = e[0];
    O.E[1][p] = e[1];
    O.E[2][p] = e[2];
}

}  // namespace pic
