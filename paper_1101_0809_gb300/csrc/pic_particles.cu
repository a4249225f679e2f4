// pic_particles.cu -- launchers of the per-particle kernels (pic_particles.cuh)
// with the tile geometry read at run time, the shared-memory sizing, and the
// particle loader and pool copy.
#include "pic_particles.cuh"

namespace pic {

template <int DIM, typename R>
static cudaError_t launch_mode(int mode, cudaStream_t st, int max_items, size_t smem, const PartArgs<R> &a)
{
    switch (mode) {
    case 0: return launch_t<DIM, R, 0>(st, max_items, smem, a);
    case 1: return launch_t<DIM, R, 1>(st, max_items, smem, a);
    default: return launch_t<DIM, R, 2>(st, max_items, smem, a);
    }
}

size_t particles_smem_bytes(int dims, int prec, int mode, int tx, int ty, int tz, int halo, int p0, int p1,
                            int order2)
{
    (void)tx;   // the x and y extents enter through the pitches (p0, p1 cover the widest tile)
    (void)ty;
    const size_t es = prec == 0 ? sizeof(double) : sizeof(float);
    // l_a = 2 1/2 reaches one cell further in both tiles; the gather of
    // Eq. wrong1 (order2 = 4) in the field tile only
    const int fext = order2 == 3 ? 0 : 1, jext = order2 == 5 ? 1 : 0;
    const long long fe = (long long)p0 * p1 * (dims == 3 ? tz + 2 * (halo + 1 + fext) : 1);
    const long long je = (long long)p0 * p1 * (dims == 3 ? tz + 2 * (halo + 2 + jext) : 1);
    size_t b = 0;
    if (mode != 2) b += 6 * fe * es;
    // current tile (+ per-cell counts in FP32), the warps' deposit queues and one count per warp
    if (mode != 1)
        b += (prec == 0 ? 24 : 28) * je + (size_t)(kThreads / 32) * (kQueueCap * (kQueueVals * es + sizeof(int)) + sizeof(int));
    return b;
}

template <int DIM, typename R>
static cudaError_t set_limit_t(int mode, size_t bytes)
{
    const int b = (int)bytes;
    switch (mode) {
    case 0: return set_limit_fused<DIM, R, GeoDyn>(b);
    case 1: return set_limit_one<DIM, R, 1, GeoDyn>(b);
    default: return set_limit_one<DIM, R, 2, GeoDyn>(b);
    }
}

cudaError_t particles_set_smem_limit(int dims, int prec, int mode, size_t bytes, int order2)
{
    if (order2 == 5) return particles_o5_set_smem_limit(dims, prec, mode, bytes);
    if (order2 == 4) return particles_w1_set_smem_limit(dims, prec, mode, bytes);
    if (prec != 0 && mode == 0) {
        const cudaError_t e = fixed_set_smem_limit(dims, bytes);
        if (e != cudaSuccess) return e;
    }
    if (dims == 3) return prec == 0 ? set_limit_t<3, double>(mode, bytes) : set_limit_t<3, float>(mode, bytes);
    return prec == 0 ? set_limit_t<2, double>(mode, bytes) : set_limit_t<2, float>(mode, bytes);
}


cudaError_t launch_particles(int dims, int prec, int mode, cudaStream_t st, WorkItem *items,
                             const int *n_items, int max_items, const RunDev *runs, const GroupDev *groups,
                             const PoolBuf &P, void *const E[3], void *const B[3], void *const J[3],
                             int *old_cell, void *const old_off[3], int halo, int max_tile_x, int max_tile_y,
                             int max_tile_z, int *err, unsigned *far_list, int p0, int p1, int order2,
                             const PoolBuf *src, const unsigned *perm)
{
    if (perm && (mode != 0 || order2 != 3)) return cudaErrorInvalidValue;   // read through perm: fused l_a = 1 1/2 only
    const size_t smem =
        particles_smem_bytes(dims, prec, mode, max_tile_x, max_tile_y, max_tile_z, halo, p0, p1, order2);
    if (order2 == 5) {
        const int tile[3] = {max_tile_x, max_tile_y, max_tile_z};
        return launch_particles_o5(dims, prec, mode, st, max_items, smem, items, n_items, runs, groups, P, E, B, J,
                                   old_cell, old_off, halo, err, far_list, tile, p0, p1);
    }
    if (order2 == 4)
        return launch_particles_w1(dims, prec, mode, st, max_items, smem, items, n_items, runs, groups, P, E, B, J,
                                   old_cell, old_off, halo, err, far_list);
    if (prec == 0) {
        auto a = make_args<double>(items, n_items, runs, groups, P, E, B, J, old_cell, old_off, halo, err, far_list, src,
                                    perm);
        return dims == 3 ? launch_mode<3, double>(mode, st, max_items, smem, a)
                         : launch_mode<2, double>(mode, st, max_items, smem, a);
    }
    auto a = make_args<float>(items, n_items, runs, groups, P, E, B, J, old_cell, old_off, halo, err, far_list, src,
                                    perm);
    if (mode == 0) {
        const int tile[3] = {max_tile_x, max_tile_y, max_tile_z};
        cudaError_t e = cudaSuccess;
        if (launch_particles_fixed(dims, st, max_items, smem, a, tile, halo, p0, p1, &e)) return e;
    }
    return dims == 3 ? launch_mode<3, float>(mode, st, max_items, smem, a)
                     : launch_mode<2, float>(mode, st, max_items, smem, a);
}

cudaError_t launch_step_persistent(int dims, int prec, cudaStream_t st, WorkItem *items, const int *n_items,
                                   const RunDev *runs, const GroupDev *groups, const PoolBuf &P, void *const E[3],
                                   void *const B[3], void *const J[3], int halo, int tx, int ty, int tz, int *err,
                                   unsigned *far_list, int nruns, const long long *run_cell_base, int *grid_blocks, int launch, int p0,
                                   int p1, long long *ant_n, int antennas, const PoolBuf *src, const unsigned *perm)
{
    void *none[3] = {nullptr, nullptr, nullptr};
    const size_t smem = particles_smem_bytes(dims, prec, 0, tx, ty, tz, halo, p0, p1);
    if (prec == 0) {
        auto a = make_args<double>(items, n_items, runs, groups, P, E, B, J, nullptr, none, halo, err, far_list, src, perm);
        return dims == 3 ? persistent_t<3, double>(st, smem, nruns, run_cell_base, a, grid_blocks, launch, ant_n, antennas)
                         : persistent_t<2, double>(st, smem, nruns, run_cell_base, a, grid_blocks, launch, ant_n, antennas);
    }
    auto a = make_args<float>(items, n_items, runs, groups, P, E, B, J, nullptr, none, halo, err, far_list, src, perm);
    const int tile[3] = {tx, ty, tz};
    cudaError_t e = cudaSuccess;
    if (launch_persistent_fixed(dims, st, smem, nruns, run_cell_base, a, grid_blocks, launch, tile, halo, p0, p1,
                                ant_n, antennas, &e))
        return e;
    return dims == 3 ? persistent_t<3, float>(st, smem, nruns, run_cell_base, a, grid_blocks, launch, ant_n, antennas)
                     : persistent_t<2, float>(st, smem, nruns, run_cell_base, a, grid_blocks, launch, ant_n, antennas);
}

// ---------------------------------------------------------------------------
// Loader: absolute normalized FP64 positions -> (cell, offset) of the pool's
// precision, periodic wrap into [0, N); an offset that rounds to 1 moves to the
// next cell with offset 0.  Momenta are converted; id = index in the call.
// ---------------------------------------------------------------------------
// With REC (FP32) the particle is written as one record (LoadRec), for the sort's
// gather.  A position already in (0, N) is taken as it is: the wrap would
// subtract N * floor(x / N) = 0, and its FP64 quotient set the kernel's time
// (16e6 particles: 1.66 ms with it; their 80 bytes each are 0.19 ms of memory).
__device__ __forceinline__ double wrap_position(double x, double N)
{
    if (x > 0.0 && x < N) return x;   // (-0.0 becomes 0.0 below)
    x -= N * floor(x / N);
    if (x >= N) x -= N;
    if (x < 0.0) x = 0.0;
    return x;
}

template <int DIM>
__device__ __forceinline__ void put_record(void *rec, long long q, int cell, int id, const float of[3], const float w[3])
{
    if constexpr (DIM == 3) {
        int4 *r = reinterpret_cast<int4 *>(static_cast<LoadRec<3> *>(rec) + q);
        r[0] = make_int4(cell, id, __float_as_int(of[0]), __float_as_int(of[1]));
        reinterpret_cast<float4 *>(r)[1] = make_float4(of[2], w[0], w[1], w[2]);
    } else {
        static_cast<LoadRec<2> *>(rec)[q] = {cell, id, {of[0], of[1]}, {w[0], w[1], w[2]}};
    }
}

template <typename R, int DIM, bool REC>
__global__ void k_load(long long n, const double *x0, const double *x1, const double *x2, const double *w0,
                       const double *w1, const double *w2, int nx, int ny, int nz, PoolBuf P, void *rec,
                       long long base)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= n) return;
    const double xs[3] = {x0[p], x1[p], DIM == 3 ? x2[p] : 0.0};
    const double ws[3] = {w0[p], w1[p], w2[p]};
    const int nn[3] = {nx, ny, nz};
    int ci[3] = {0, 0, 0};
    R of[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const double x = wrap_position(xs[a], (double)nn[a]);
        int c = (int)floor(x);
        if (c >= nn[a]) c = nn[a] - 1;
        R o = (R)(x - (double)c);
        if (o >= R(1)) {
            o = R(0);
            c = c + 1 == nn[a] ? 0 : c + 1;
        }
        ci[a] = c;
        of[a] = o;
    }
    const int cell = ci[0] + nx * (ci[1] + ny * ci[2]);
    P.cell[base + p] = cell;
    if constexpr (REC) {
        const float w[3] = {(float)ws[0], (float)ws[1], (float)ws[2]};
        put_record<DIM>(rec, base + p, cell, (int)p, of, w);
    } else {
#pragma unroll
        for (int a = 0; a < DIM; ++a) static_cast<R *>(P.off[a])[base + p] = of[a];
#pragma unroll
        for (int a = 0; a < 3; ++a) static_cast<R *>(P.w[a])[base + p] = (R)ws[a];
        P.id[base + p] = (int)p;
    }
}

template <int DIM>
static void load_t(int prec, cudaStream_t st, unsigned nb, int nt, long long n, const double *x0, const double *x1,
                   const double *x2, const double *w0, const double *w1, const double *w2, int nx, int ny, int nz,
                   const PoolBuf &P, void *rec, long long base)
{
    if (prec == 0)
        k_load<double, DIM, false><<<nb, nt, 0, st>>>(n, x0, x1, x2, w0, w1, w2, nx, ny, nz, P, nullptr, base);
    else if (rec)
        k_load<float, DIM, true><<<nb, nt, 0, st>>>(n, x0, x1, x2, w0, w1, w2, nx, ny, nz, P, rec, base);
    else
        k_load<float, DIM, false><<<nb, nt, 0, st>>>(n, x0, x1, x2, w0, w1, w2, nx, ny, nz, P, nullptr, base);
}

cudaError_t launch_load(int prec, cudaStream_t st, long long n, const double *x0, const double *x1,
                        const double *x2, const double *w0, const double *w1, const double *w2, int dims, int nx,
                        int ny, int nz, const PoolBuf &P, long long base, void *rec)
{
    if (n <= 0) return cudaSuccess;
    const int nt = 256;
    const unsigned nb = (unsigned)((n + nt - 1) / nt);
    if (dims == 3)
        load_t<3>(prec, st, nb, nt, n, x0, x1, x2, w0, w1, w2, nx, ny, nz, P, rec, base);
    else
        load_t<2>(prec, st, nb, nt, n, x0, x1, x2, w0, w1, w2, nx, ny, nz, P, rec, base);
    return cudaGetLastError();
}

// A range of an FP32 pool into records, for a load that keeps other groups.
template <int DIM>
__global__ void k_copy_pool_rec(long long n, PoolBuf S, long long sb, int *cell, void *rec, long long db)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= n) return;
    auto at = [&](void *v) { return static_cast<const float *>(v)[sb + p]; };
    const int c = S.cell[sb + p];
    if (cell + db != S.cell + sb) cell[db + p] = c;
    const float of[3] = {at(S.off[0]), at(S.off[1]), DIM == 3 ? at(S.off[2]) : 0.f};
    const float w[3] = {at(S.w[0]), at(S.w[1]), at(S.w[2])};
    put_record<DIM>(rec, db + p, c, S.id[sb + p], of, w);
}

cudaError_t launch_copy_pool_rec(cudaStream_t st, const PoolBuf &src, long long sb, int *dst_cell, void *rec,
                                 long long db, long long n, int dims)
{
    if (n <= 0) return cudaSuccess;
    const int nt = 256;
    const unsigned nb = (unsigned)((n + nt - 1) / nt);
    if (dims == 3)
        k_copy_pool_rec<3><<<nb, nt, 0, st>>>(n, src, sb, dst_cell, rec, db);
    else
        k_copy_pool_rec<2><<<nb, nt, 0, st>>>(n, src, sb, dst_cell, rec, db);
    return cudaGetLastError();
}

// Device-to-device copy of a range of pool entries (used when the pool is re-laid out).
template <typename R>
__global__ void k_copy_pool(long long n, const int *sc, const R *so0, const R *so1, const R *so2, const R *sw0,
                            const R *sw1, const R *sw2, const int *sid, int *dc, R *do0, R *do1, R *do2, R *dw0,
                            R *dw1, R *dw2, int *did)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= n) return;
    dc[p] = sc[p];
    do0[p] = so0[p];
    do1[p] = so1[p];
    if (do2) do2[p] = so2[p];
    dw0[p] = sw0[p];
    dw1[p] = sw1[p];
    dw2[p] = sw2[p];
    did[p] = sid[p];
}

cudaError_t launch_copy_pool(int prec, cudaStream_t st, const PoolBuf &src, long long sb, const PoolBuf &dst,
                             long long db, long long n)
{
    if (n <= 0) return cudaSuccess;
    const int nt = 256;
    const unsigned nb = (unsigned)((n + nt - 1) / nt);
    if (prec == 0) {
        auto S = [&](void *p) { return p ? (double *)p + sb : nullptr; };
        auto D = [&](void *p) { return p ? (double *)p + db : nullptr; };
        k_copy_pool<double><<<nb, nt, 0, st>>>(n, src.cell + sb, S(src.off[0]), S(src.off[1]), S(src.off[2]),
                                               S(src.w[0]), S(src.w[1]), S(src.w[2]), src.id + sb, dst.cell + db,
                                               D(dst.off[0]), D(dst.off[1]), D(dst.off[2]), D(dst.w[0]),
                                               D(dst.w[1]), D(dst.w[2]), dst.id + db);
    } else {
        auto S = [&](void *p) { return p ? (float *)p + sb : nullptr; };
        auto D = [&](void *p) { return p ? (float *)p + db : nullptr; };
        k_copy_pool<float><<<nb, nt, 0, st>>>(n, src.cell + sb, S(src.off[0]), S(src.off[1]), S(src.off[2]),
                                              S(src.w[0]), S(src.w[1]), S(src.w[2]), src.id + sb, dst.cell + db,
                                              D(dst.off[0]), D(dst.off[1]), D(dst.off[2]), D(dst.w[0]),
                                              D(dst.w[1]), D(dst.w[2]), dst.id + db);
    }
    return cudaGetLastError();
}

}  // namespace pic
