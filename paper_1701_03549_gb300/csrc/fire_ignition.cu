// Ignition-point search (the paper's Sec. 3 experiment with the ignition
// treated as unknown) on the device, with its C ABI (include/fire.h).
//
// Reading (identical to the test oracle's, implemented independently):
//  * the target's burnt cells span rows [r0, r1] and columns [c0, c1];
//  * lattice point (a, b) sits at row r0 + floor((2a+1)(r1-r0+1) / (2 LH))
//    and column c0 + floor((2b+1)(c1-c0+1) / (2 LW));
//  * its candidate ignition is the burnable burnt cell nearest to it
//    (squared distance, ties to the lower row-major index);
//  * candidate c = a LW + b is simulated reps times with seeds
//    seed + c reps + r; its fitness is the replicate mean;
//  * the ensemble is the candidates with fitness <= cutoff (else the best,
//    ties to the lower index); the estimate is the mean and sample standard
//    deviation of their x = column and y = row.
#include "fire_internal.h"

using namespace fire;

namespace {

// Bounding box of the target's burnt cells: bbox = {r0, r1, c0, c1}.
__global__ void k_target_bbox(MapDev m, int *bbox)
{
    const int nw = m.ntiles * 32;
    for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < nw;
         w += gridDim.x * blockDim.x) {
        const uint32_t t = m.tgt[w];
        if (!t) continue;
        const int k = w >> 5, ti = k / m.TW, tj = k - ti * m.TW;
        const int R = ti * 32 + (w & 31);
        const int cmin = tj * 32 + (__ffs(t) - 1);
        const int cmax = tj * 32 + (31 - __clz(t));
        atomicMin(&bbox[0], R);
        atomicMax(&bbox[1], R);
        atomicMin(&bbox[2], cmin);
        atomicMax(&bbox[3], cmax);
    }
}

// Row-major index of the burnable burnt cell nearest to (R, C), a cell of the
// map: least (squared distance, index), one block of 256 threads cooperating
// (all call it); 0xffffffff when the target has no burnable cell.  The distance
// can exceed 32 bits on wide maps, so the pair is compared field by field.
//
// The tiles are searched in square rings around the point's tile, in batches
// that double, until no farther ring can hold a cell as near as the best one:
// every cell of ring r is at least 32 (r - 1) + 1 rows or columns away.  A
// batch is the map's part of one square less that of the square inside: up to
// four rectangles of tiles, so that no tile is visited twice and none outside
// the map (whole rings, on 32 x 131072 with the target at the far end, were 2e9
// words a point instead of 131072).  A warp takes a tile, four at a time for
// the loads' latency, a lane its row word; of a word only the nearest cell on
// either side counts.  fire_snap_ignitions on one GB300, against a walk over
// every word of the map (ms, that walk in brackets): 256 points on 1024 x 1024
// inside a scar 0.056 (0.143), target in the far corner 0.054 (0.064); 4096 x
// 4096, far corner 0.20 (0.47); 16 points on 32 x 131072, far end 0.079 (0.139;
// by whole rings 1434).
__device__ uint32_t block_nearest(const MapDev &m, long long R, long long C)
{
    constexpr int kWarps = 8;
    unsigned long long bd = ~0ull;
    uint32_t bi = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = (int)(R >> 5), u0 = (int)(C >> 5);
    const int last = max(max(t0, m.TH - 1 - t0), max(u0, m.TW - 1 - u0));
    // rings of this batch; up to 64 tiles all at once, eight a warp
    int r0 = 0, r1 = m.ntiles <= 64 ? last : 1;
    for (;;) {
        r1 = min(r1, last);
        // the batch's rows and columns of tiles, and those of the square inside
        const int i0 = max(t0 - r1, 0), i1 = min(t0 + r1, m.TH - 1);
        const int j0 = max(u0 - r1, 0), j1 = min(u0 + r1, m.TW - 1);
        const int a0 = r0 ? t0 - r0 + 1 : i1 + 1, a1 = r0 ? t0 + r0 - 1 : i1;
        const int b0 = u0 - r0 + 1, b1 = u0 + r0 - 1;
#pragma unroll 1
        for (int side = 0; side < (r0 ? 4 : 1); ++side) {   // above (or all), below, left, right
            const int p0 = side == 0 ? i0 : side == 1 ? max(a1 + 1, i0) : max(a0, i0);
            const int p1 = side == 0 ? min(a0 - 1, i1) : side == 1 ? i1 : min(a1, i1);
            const int q0 = side == 3 ? max(b1 + 1, j0) : j0;
            const int q1 = side == 2 ? min(b0 - 1, j1) : j1;
            const int h = p1 - p0 + 1, w = q1 - q0 + 1;
            if (h <= 0 || w <= 0) continue;
            int i = warp / w, j = warp - i * w;
            const int di = kWarps / w, dj = kWarps - di * w;
            while (i < h) {
                uint32_t t[4];
                int ti[4], tj[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    ti[k] = p0 + i;
                    tj[k] = q0 + j;
                    t[k] = i < h ? m.tgt[(ti[k] * m.TW + tj[k]) * 32 + lane] : 0u;
                    i += di;
                    j += dj;
                    if (j >= w) j -= w, ++i;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (!t[k]) continue;
                    const uint32_t v = t[k] & ~m.blk[(ti[k] * m.TW + tj[k]) * 32 + lane];
                    const long long Rw = ti[k] * 32 + lane;
                    // columns up to C, and from C on
                    const int c = (int)min(max(C - tj[k] * 32, -1ll), 32ll);
                    const uint32_t le = c < 0 ? 0u : (c >= 31 ? v : v & ((2u << c) - 1u));
                    const uint32_t ge = c <= 0 ? v : (c > 31 ? 0u : v & ~((1u << c) - 1u));
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t x = e ? ge : le;
                        if (!x) continue;
                        const long long Cc = tj[k] * 32 + (e ? __ffs(x) - 1 : 31 - __clz(x));
                        const unsigned long long d = (unsigned long long)(
                            (Rw - R) * (Rw - R) + (Cc - C) * (Cc - C));
                        const uint32_t idx = (uint32_t)(Rw * m.W + Cc);
                        if (d < bd || (d == bd && idx < bi)) {
                            bd = d;
                            bi = idx;
                        }
                    }
                }
            }
        }
        if (r1 == last) break;
        // the best of the block so far, a lower bound of the next ring's cells
        const unsigned long long near = 32ull * r1 + 1ull;
        if (__syncthreads_or(bd < near * near)) break;
        r0 = r1 + 1;
        r1 = 2 * r1 + 1;
    }
    __shared__ unsigned long long rd[256];
    __shared__ uint32_t ri[256];
    rd[threadIdx.x] = bd;
    ri[threadIdx.x] = bi;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            const unsigned long long d2 = rd[threadIdx.x + s];
            const uint32_t i2 = ri[threadIdx.x + s];
            if (d2 < rd[threadIdx.x] ||
                (d2 == rd[threadIdx.x] && i2 < ri[threadIdx.x])) {
                rd[threadIdx.x] = d2;
                ri[threadIdx.x] = i2;
            }
        }
        __syncthreads();
    }
    const uint32_t best = rd[0] == ~0ull ? 0xffffffffu : ri[0];
    __syncthreads();   // the arrays may be reused by the next call
    return best;
}

// One block (256 threads) per lattice point: nearest burnable burnt cell.
__global__ void k_snap(MapDev m, const int *__restrict__ bbox, int LH, int LW,
                       int32_t *__restrict__ cells, int *__restrict__ fail)
{
    const int cidx = blockIdx.x;
    const int a = cidx / LW, b = cidx - a * LW;
    const int r0 = bbox[0], r1 = bbox[1], c0 = bbox[2], c1 = bbox[3];
    const long long R = r0 + ((2LL * a + 1) * (r1 - r0 + 1)) / (2LL * LH);
    const long long C = c0 + ((2LL * b + 1) * (c1 - c0 + 1)) / (2LL * LW);
    const uint32_t best = block_nearest(m, R, C);
    if (threadIdx.x == 0) {
        if (best == 0xffffffffu) {
            atomicOr(fail, 1);
            cells[2 * cidx] = cells[2 * cidx + 1] = 0;
        } else {
            cells[2 * cidx] = (int32_t)(best / (uint32_t)m.W);
            cells[2 * cidx + 1] = (int32_t)(best % (uint32_t)m.W);
        }
    }
}

// A coordinate gene clamped to [0, hi] (a NaN counts as 0) and rounded half
// up.
__device__ __forceinline__ long long gene_coord(double v, int hi)
{
    const double c = v >= 0.0 ? (v > (double)hi ? (double)hi : v) : 0.0;
    return (long long)floor(__dadd_rn(c, 0.5));
}

// One block (256 threads) per individual: the ignition cell of its x
// (column) and y (row) genes, written to its reps simulations.
__global__ void k_snap_genes(MapDev m, int G, int gx, int gy,
                             const double *__restrict__ genes, int reps,
                             fire_cell *__restrict__ ign, int *__restrict__ fail)
{
    const long long j = blockIdx.x;
    const long long C = gene_coord(genes[j * G + gx], m.W - 1);
    const long long R = gene_coord(genes[j * G + gy], m.H - 1);
    const uint32_t best = block_nearest(m, R, C);
    fire_cell cell;
    cell.row = best == 0xffffffffu ? 0 : (int32_t)(best / (uint32_t)m.W);
    cell.col = best == 0xffffffffu ? 0 : (int32_t)(best % (uint32_t)m.W);
    if (best == 0xffffffffu && threadIdx.x == 0) atomicOr(fail, 1);
    for (int r = threadIdx.x; r < reps; r += blockDim.x) ign[j * reps + r] = cell;
}

__global__ void k_ign_batch(int L, int reps, const int32_t *__restrict__ cells,
                            const double *__restrict__ beta, uint64_t seed,
                            fire_params *__restrict__ params,
                            fire_cell *__restrict__ ign,
                            uint64_t *__restrict__ seeds)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L * reps) return;
    const int c = i / reps;
    fire_params p;
    for (int j = 0; j < 5; ++j) p.b[j] = beta[j];
    params[i] = p;
    ign[i].row = cells[2 * c];
    ign[i].col = cells[2 * c + 1];
    seeds[i] = seed + (uint64_t)i;   // = seed + c reps + r
}

// Ensemble estimate (one block of 256).  Coordinates are whole numbers, so
// their sums are exact in any order; the sums of squared deviations are added
// in index order by one thread each, from shared memory (one thread that read
// and decided everything took 525 us for 1024 candidates).  Candidates outside
// the ensemble add +0, which changes no sum.
__global__ void __launch_bounds__(256)
    k_ign_ensemble(int L, const double *__restrict__ fm,
                   const int32_t *__restrict__ cells, double cutoff,
                   double *__restrict__ xy)
{
    __shared__ unsigned long long red[3][256];
    const int i = threadIdx.x;
    unsigned long long k = 0, sx = 0, sy = 0;
    for (int c = i; c < L; c += 256)
        if (fm[c] <= cutoff) {
            k++;
            sx += (unsigned long long)cells[2 * c + 1];
            sy += (unsigned long long)cells[2 * c];
        }
    red[0][i] = k;
    red[1][i] = sx;
    red[2][i] = sy;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (i < s)
            for (int j = 0; j < 3; ++j) red[j][i] += red[j][i + s];
        __syncthreads();
    }
    k = red[0][0];
    sx = red[1][0];
    sy = red[2][0];
    __syncthreads();
    if (k == 0) {
        // the candidate of least fitness (NaN last), ties to the lower index
        __shared__ int cand[256];
        int b = -1;
        auto better = [&](int c, int d) {
            const double fc = fm[c], fd = fm[d];
            const bool nc = fc != fc, nd = fd != fd;
            if (nc != nd) return nd;
            if (!nc && fc != fd) return fc < fd;
            return c < d;
        };
        for (int c = i; c < L; c += 256)
            if (b < 0 || better(c, b)) b = c;
        cand[i] = b;
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if (i < s && cand[i + s] >= 0 && (cand[i] < 0 || better(cand[i + s], cand[i])))
                cand[i] = cand[i + s];
            __syncthreads();
        }
        if (i == 0) {
            xy[0] = (double)cells[2 * cand[0] + 1];
            xy[1] = 0.0;
            xy[2] = (double)cells[2 * cand[0]];
            xy[3] = 0.0;
        }
        return;
    }
    const double mean[2] = {__ddiv_rn((double)sx, (double)k),
                            __ddiv_rn((double)sy, (double)k)};
    __shared__ double sq[2][256];
    double v = 0.0;
    for (int c0 = 0; c0 < L; c0 += 256) {
        const int c = c0 + i;
        const bool in = c < L && fm[c] <= cutoff;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const double d = in ? __dsub_rn((double)cells[2 * c + (a ? 0 : 1)], mean[a]) : 0.0;
            sq[a][i] = __dmul_rn(d, d);
        }
        __syncthreads();
        if (i == 0 || i == 32)
            for (int j = 0; j < min(256, L - c0); ++j) v = __dadd_rn(v, sq[i >> 5][j]);
        __syncthreads();
    }
    if (i == 0 || i == 32) {
        const int a = i >> 5;
        xy[2 * a] = mean[a];
        xy[2 * a + 1] = k > 1 ? __dsqrt_rn(__ddiv_rn(v, (double)(k - 1))) : 0.0;
    }
}

}  // namespace

extern "C" int ignition_search(fire_ctx *ctx, const fire_map *map,
                               const fire_params *params, int lat_h, int lat_w,
                               int reps, uint64_t seed, int kind, double cutoff,
                               uint32_t flags, double *fitness_map,
                               int32_t *cells, double xy_mean_sd[4])
{
    FIRE_NVTX("ignition_search");
    if (!ctx) return FIRE_EINVAL;
    if (!valid_map(map) || !params || lat_h <= 0 || lat_w <= 0 || reps <= 0 ||
        (kind != 0 && kind != 1) || !fitness_map || !xy_mean_sd)
        return set_err(ctx, FIRE_EINVAL, "bad ignition_search arguments");
    const long long Lll = (long long)lat_h * lat_w;
    if (Lll * reps > 0x7fffffffll)
        return set_err(ctx, FIRE_EINVAL, "lattice x replicates too large");
    int rc = ensure_device(ctx);
    if (rc) return rc;
    const bool dev = flags & FIRE_DEVICE_PTRS;
    const int L = (int)Lll, n = L * reps;
    // scratch layout
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += round16(bytes); return o; };
    const size_t o_bbox = take(16), o_fail = take(16), o_cells = take((size_t)L * 8);
    const size_t o_beta = take(40), o_par = take((size_t)n * sizeof(fire_params));
    const size_t o_ign = take((size_t)n * sizeof(fire_cell));
    const size_t o_seed = take((size_t)n * 8), o_res = take((size_t)n * sizeof(fire_result));
    const size_t o_fit = take((size_t)n * 8), o_fm = take((size_t)L * 8);
    const size_t o_xy = take(32);
    rc = grow_device(ctx, &ctx->staging, &ctx->staging_bytes, off, "ignition search");
    if (rc) return rc;
    char *base = (char *)ctx->staging;
    int *dbbox = (int *)(base + o_bbox);
    int *dfail = (int *)(base + o_fail);
    int32_t *dcells = (int32_t *)(base + o_cells);
    double *dbeta = (double *)(base + o_beta);
    fire_params *dpar = (fire_params *)(base + o_par);
    fire_cell *dign = (fire_cell *)(base + o_ign);
    uint64_t *dseed = (uint64_t *)(base + o_seed);
    fire_result *dres = (fire_result *)(base + o_res);
    double *dfit = (double *)(base + o_fit);
    double *dfm = (double *)(base + o_fm);
    double *dxy = (double *)(base + o_xy);
    cudaStream_t st = ctx->stream;
    const int init[4] = {0x7fffffff, -1, 0x7fffffff, -1};
    CUDA_TRY(ctx, cudaMemcpyAsync(dbbox, init, 16, cudaMemcpyHostToDevice, st), "bbox init");
    CUDA_TRY(ctx, cudaMemsetAsync(dfail, 0, 4, st), "fail init");
    CUDA_TRY(ctx, cudaMemcpyAsync(dbeta, params->b, 40,
                                  dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                  st), "params copy");
    k_target_bbox<<<152 * 4, 256, 0, st>>>(map->dev, dbbox);
    int hbbox[4];
    CUDA_TRY(ctx, cudaMemcpyAsync(hbbox, dbbox, 16, cudaMemcpyDeviceToHost, st), "bbox D2H");
    CUDA_TRY(ctx, cudaStreamSynchronize(st), "bbox sync");
    if (hbbox[1] < 0) return set_err(ctx, FIRE_EINVAL, "the map's target is empty");
    k_snap<<<L, 256, 0, st>>>(map->dev, dbbox, lat_h, lat_w, dcells, dfail);
    k_ign_batch<<<(n + 255) / 256, 256, 0, st>>>(L, reps, dcells, dbeta, seed, dpar,
                                                  dign, dseed);
    CUDA_TRY(ctx, cudaGetLastError(), "ignition set-up kernels");
    int hfail = 0;
    CUDA_TRY(ctx, cudaMemcpyAsync(&hfail, dfail, 4, cudaMemcpyDeviceToHost, st), "fail D2H");
    CUDA_TRY(ctx, cudaStreamSynchronize(st), "snap sync");
    if (hfail) return set_err(ctx, FIRE_EINVAL, "the target has no burnable burnt cell");
    rc = fire_simulate_batch(ctx, map, n, dpar, dign, dseed, 0, FIRE_DEVICE_PTRS, dres,
                             nullptr);
    if (rc) return rc;
    rc = fire_fitness(ctx, dres, n, kind, FIRE_DEVICE_PTRS, dfit);
    if (rc) return rc;
    rc = fire_group_mean(ctx, dfit, L, reps, FIRE_DEVICE_PTRS, dfm);
    if (rc) return rc;
    k_ign_ensemble<<<1, 256, 0, st>>>(L, dfm, dcells, cutoff, dxy);
    CUDA_TRY(ctx, cudaGetLastError(), "ensemble kernel");
    const cudaMemcpyKind dk = dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    CUDA_TRY(ctx, cudaMemcpyAsync(fitness_map, dfm, (size_t)L * 8, dk, st), "fitness map");
    if (cells)
        CUDA_TRY(ctx, cudaMemcpyAsync(cells, dcells, (size_t)L * 8, dk, st), "cells");
    CUDA_TRY(ctx, cudaMemcpyAsync(xy_mean_sd, dxy, 32, dk, st), "estimate");
    return fire_sync(ctx);
}

extern "C" int fire_snap_ignitions(fire_ctx *ctx, const fire_map *map, int n,
                                   int genes, int gx, int gy,
                                   const double *genes_in, int reps,
                                   uint32_t flags, fire_cell *ignitions)
{
    FIRE_NVTX("fire_snap_ignitions");
    if (!ctx) return FIRE_EINVAL;
    if (!valid_map(map) || n < 0 || genes < 1 || gx < 0 || gx >= genes ||
        gy < 0 || gy >= genes || reps < 1)
        return set_err(ctx, FIRE_EINVAL, "bad fire_snap_ignitions arguments");
    if (map->ctx->device != ctx->device)
        return set_err(ctx, FIRE_EINVAL, "the map was uploaded on another device");
    if (n == 0) return FIRE_OK;
    if (!genes_in || !ignitions) return set_err(ctx, FIRE_EINVAL, "NULL argument");
    if ((long long)n * reps > 0x7fffffffll)
        return set_err(ctx, FIRE_EINVAL, "individuals x replicates too large");
    int rc = ensure_device(ctx);
    if (rc) return rc;
    const bool dev = flags & FIRE_DEVICE_PTRS;
    const size_t bg = round16((size_t)n * genes * 8);
    const size_t bi = round16((size_t)n * reps * sizeof(fire_cell));
    rc = grow_device(ctx, &ctx->staging, &ctx->staging_bytes,
                     16 + (dev ? 0 : bg + bi), "ignition genes");
    if (rc) return rc;
    char *base = (char *)ctx->staging;
    int *dfail = (int *)base;
    const double *dgenes = genes_in;
    fire_cell *dign = ignitions;
    cudaStream_t st = ctx->stream;
    if (!dev) {
        dgenes = (const double *)(base + 16);
        dign = (fire_cell *)(base + 16 + bg);
        CUDA_TRY(ctx, cudaMemcpyAsync((void *)dgenes, genes_in, (size_t)n * genes * 8,
                                      cudaMemcpyHostToDevice, st), "genes H2D");
    }
    CUDA_TRY(ctx, cudaMemsetAsync(dfail, 0, 4, st), "fail init");
    k_snap_genes<<<n, 256, 0, st>>>(map->dev, genes, gx, gy, dgenes, reps, dign, dfail);
    CUDA_TRY(ctx, cudaGetLastError(), "snap kernel");
    if (!dev)
        CUDA_TRY(ctx, cudaMemcpyAsync(ignitions, dign, (size_t)n * reps * sizeof(fire_cell),
                                      cudaMemcpyDeviceToHost, st), "ignitions D2H");
    int hfail = 0;
    CUDA_TRY(ctx, cudaMemcpyAsync(&hfail, dfail, 4, cudaMemcpyDeviceToHost, st), "fail D2H");
    CUDA_TRY(ctx, cudaStreamSynchronize(st), "snap sync");
    if (hfail) return set_err(ctx, FIRE_EINVAL, "the target has no burnable burnt cell");
    return FIRE_OK;
}
