// Set-up of the dense coarse solve: the pseudo-inverse A^+ of the coarsest operator (at most
// 1024 cells), A^+ = (A + c 1 1^T)^-1 - 1 1^T / (c n^2), c = mean(diag) / n, by blocked
// Gauss-Jordan in place without pivoting (the matrix is symmetric positive definite).
//
// A step takes 32 pivots K: P^-1 of the pivot block, the row panel M[K, J] <- P^-1 M[K, J], the
// trailing update M[I, J] <- M[I, J] - M[I, K] M[K, J], and the column panel
// M[I, K] <- -M[I, K] P^-1, M[K, K] <- P^-1 (I, J outside K).
//
// What bounds it: a warp's FP64 FMA occupies its quarter of an SM for 64 clocks on GB300 (two
// FMAs per SM and clock), so the n^3 FMAs take 0.21 ms at n = 512 and 1.6 ms at n = 990 on all SMs, and the
// 32 x 32 pivot block, one serial chain of 32 reciprocals (about 750 clocks a pivot), 12 us per
// step on one SM.  So a step is two launches: the panels, dealt out in 32 x 8 tiles, and the trailing
// update, whose first cluster of four CTAs updates the next pivot block before anything else and
// then inverts it while the other CTAs do the rest.  Four launches per step, the pivot block
// inverted by itself, took 85 us per step; this takes about 20 us (n = 512).  The operations on
// every entry and their order do not depend on the tiling.
#include <cooperative_groups.h>

#include "mg_internal.cuh"

namespace cg = cooperative_groups;

namespace mg {

namespace {

constexpr int kGj = 32;          // pivots per step
constexpr int kPanel = 8;        // columns (rows) of a row (column) panel tile
constexpr int kTileRows = 16;    // rows of a trailing tile, kGj columns
constexpr int kTrailThreads = 512;
constexpr int kTrailCluster = 4;

// M (row-major n x n) = A + c 1 1^T, scal[0] = c; a block takes rows blockIdx.x, + gridDim.x, ...
// and, like every other block, adds up the diagonal (the same tree in each)
__global__ void __launch_bounds__(1024) k_coarse_assemble(Dims d, double ih2, const double *__restrict__ fx,
                                                          const double *__restrict__ fy, const double *__restrict__ fz,
                                                          double *M, double *scal) {
    grid_wait();
    __shared__ double red[1024], dg[1024];
    const int c = threadIdx.x, n = (int)d.n, nxy = (int)d.nxy;
    double diag = 0.0;
    if (c < n) {
        const int r = c / d.nx, i = c - r * d.nx, j = r % d.ny, k = r / d.ny;
        if (i > 0) diag = fma(fx[c], ih2, diag);
        if (i < d.nx - 1) diag = fma(fx[c + 1], ih2, diag);
        if (j > 0) diag = fma(fy[c], ih2, diag);
        if (j < d.ny - 1) diag = fma(fy[c + d.nx], ih2, diag);
        if (k > 0) diag = fma(fz[c], ih2, diag);
        if (k < d.nz - 1) diag = fma(fz[c + nxy], ih2, diag);
    }
    red[c] = dg[c] = diag;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if (c < w) red[c] += red[c + w];
        __syncthreads();
    }
    const double shift = red[0] / n / n;
    if (blockIdx.x == 0 && c == 0) scal[0] = shift;
    if (c >= n) return;
    for (int row = blockIdx.x; row < n; row += gridDim.x) {
        const int r = row / d.nx, i = row - r * d.nx, j = r % d.ny, k = r / d.ny;
        double f = 0.0;
        if (i > 0 && c == row - 1) f = fx[row];
        if (i < d.nx - 1 && c == row + 1) f = fx[row + 1];
        if (j > 0 && c == row - d.nx) f = fy[row];
        if (j < d.ny - 1 && c == row + d.nx) f = fy[row + d.nx];
        if (k > 0 && c == row - nxy) f = fz[row];
        if (k < d.nz - 1 && c == row + nxy) f = fz[row + nxy];
        // an entry is rounded before the shift is added
        M[(i64)row * n + c] = __dadd_rn(c == row ? dg[row] : -__dmul_rn(f, ih2), shift);
    }
}

// the panels of pivots [kb, kb + bs): blocks [0, tiles) take eight columns of the row panel, blocks
// [tiles, 2 tiles) eight rows of the column panel, whose old entries go to C (n x 32)
__global__ void __launch_bounds__(256) k_gj_panels(int n, int kb, int bs, int tiles, double *M,
                                                   const double *__restrict__ Pinv, double *C) {
    grid_wait();
    __shared__ double Pi[kGj][kGj + 1], S[kGj][kPanel + 1];
    const int tid = threadIdx.x;
    for (int e = tid; e < kGj * kGj; e += 256) Pi[e / kGj][e % kGj] = Pinv[e];
    if ((int)blockIdx.x < tiles) {
        const int ty = tid / kPanel, tx = tid % kPanel, j = blockIdx.x * kPanel + tx;
        const bool ok = j < n && (j < kb || j >= kb + bs);
        if (ty < bs) S[ty][tx] = ok ? M[(i64)(kb + ty) * n + j] : 0.0;
        __syncthreads();
        if (ty < bs && ok) {
            double acc = 0.0;
            for (int t = 0; t < bs; ++t) acc = fma(Pi[ty][t], S[t][tx], acc);
            M[(i64)(kb + ty) * n + j] = acc;
        }
        return;
    }
    const int ty = tid / kGj, tx = tid % kGj, i = (blockIdx.x - tiles) * kPanel + ty;
    const bool in = i < n && tx < bs, piv = i >= kb && i < kb + bs;
    const double old = in && !piv ? M[(i64)i * n + kb + tx] : 0.0;
    S[tx][ty] = old;
    if (in && !piv) C[i * kGj + tx] = old;
    __syncthreads();
    if (!in) return;
    if (piv) {
        M[(i64)i * n + kb + tx] = Pi[i - kb][tx];
    } else {
        double acc = 0.0;
        for (int t = 0; t < bs; ++t) acc = fma(S[t][ty], Pi[t][tx], acc);
        M[(i64)i * n + kb + tx] = -acc;
    }
}

// P^-1 of the bs x bs block P by element-wise Gauss-Jordan, P in shared memory (row stride
// kGj + 1), the result row-major in Pinv.  Warp w holds rows w and w + 16, a lane a column; the
// warp of the next pivot's row forms its reciprocal and scaled row ahead of the barrier that
// publishes them, while the other rows are still being updated.
__device__ void pivot_inverse(const double (*P)[kGj + 1], int bs, double (*srow)[kGj], double *srp, double *Pinv) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double a[2] = {P[w][lane], P[w + 16][lane]};
    // scaled row of pivot k, from the value of its row before the step
    auto publish = [&](int k, double v) {
        const double rp = 1.0 / __shfl_sync(0xffffffffu, v, k);
        srow[k & 1][lane] = lane == k ? rp : v * rp;
        if (lane == 0) srp[k & 1] = rp;
    };
    if (w == 0) publish(0, a[0]);
    __syncthreads();
    for (int k = 0; k < bs; ++k) {
        const double s = srow[k & 1][lane], rp = srp[k & 1];
        const int next = k + 1;
        auto step = [&](int q) {
            const double col = __shfl_sync(0xffffffffu, a[q], k);
            // column k: fma(-col, rp, 0) = -col rp, so that every entry costs one FP64 instruction
            const double v = fma(-col, lane == k ? rp : s, lane == k ? 0.0 : a[q]);
            a[q] = w + 16 * q == k ? s : v;
        };
        const int first = (next >> 4) & 1;  // the next pivot's row before the other one
        step(first);
        if (next < bs && w == (next & 15)) publish(next, a[first]);
        step(1 - first);
        __syncthreads();
    }
    Pinv[w * kGj + lane] = a[0];
    Pinv[(w + 16) * kGj + lane] = a[1];
}

// the trailing update of pivots [kb, kb + bs) (none for kb < 0) and the inverse of the next pivot
// block [nb, nb + nbs) (none for nbs = 0).  Cluster 0 updates that block, eight rows per CTA; its first
// CTA inverts it, all the others share the 16 x 32 tiles outside it.
__global__ void __cluster_dims__(kTrailCluster, 1, 1) __launch_bounds__(kTrailThreads)
    k_gj_trailing(int n, int kb, int bs, int nb, int nbs, double *M, const double *__restrict__ C, double *Pinv) {
    grid_wait();
    __shared__ double Cs[kTileRows][kGj], R[kGj][kGj], P[kGj][kGj + 1], srow[2][kGj], srp[2];
    const int tid = threadIdx.x, ty = tid / kGj, tx = tid % kGj;
    // a tile: rows i0 + [0, rows), rows <= kTileRows, of the 32 columns from j0.  fetch loads this
    // thread's entry and its share of C and of the pivot rows, update returns (and stores) the entry
    double fc = 0.0, fr[kGj * kGj / kTrailThreads], fm = 0.0;
    auto fetch = [&](int i0, int rows, int j0) {
        const int i = i0 + ty, j = j0 + tx;
        fc = (ty < rows && i < n && tx < bs) ? C[i * kGj + tx] : 0.0;
        fm = (ty < rows && i < n && j < n) ? M[(i64)i * n + j] : 0.0;
#pragma unroll
        for (int u = 0; u < kGj * kGj / kTrailThreads; ++u) {
            const int t = ty + u * (kTrailThreads / kGj);
            fr[u] = (t < bs && j < n) ? M[(i64)(kb + t) * n + j] : 0.0;
        }
    };
    auto update = [&](int i0, int rows, int j0, auto &&next) {
        Cs[ty][tx] = fc;
#pragma unroll
        for (int u = 0; u < kGj * kGj / kTrailThreads; ++u) R[ty + u * (kTrailThreads / kGj)][tx] = fr[u];
        double acc = fm;
        __syncthreads();
        next();  // the next tile's loads travel during this one's arithmetic
        if (ty < rows) {
            if (bs == kGj) {
#pragma unroll 8
                for (int t = 0; t < kGj; ++t) acc = fma(-Cs[ty][t], R[t][tx], acc);
            } else {
                for (int t = 0; t < bs; ++t) acc = fma(-Cs[ty][t], R[t][tx], acc);
            }
            if (i0 + ty < n && j0 + tx < n) M[(i64)(i0 + ty) * n + j0 + tx] = acc;
        }
        __syncthreads();
        return acc;
    };
    if (nbs > 0 && blockIdx.x < kTrailCluster) {
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();  // the cluster's first CTA is there before the others write its shared memory
        const int r0 = blockIdx.x * 8;  // this CTA's rows of the pivot block
        double v = 0.0;
        if (kb >= 0) {
            fetch(nb + r0, 8, nb);
            v = update(nb + r0, 8, nb, [] {});
        } else if (ty < 8 && nb + r0 + ty < n && nb + tx < n) v = M[(i64)(nb + r0 + ty) * n + nb + tx];
        if (ty < 8) *cl.map_shared_rank(&P[r0 + ty][tx], 0) = v;
        cl.sync();
        if (blockIdx.x == 0) {
            pivot_inverse(P, nbs, srow, srp, Pinv);
            return;
        }
    }
    if (kb < 0) return;
    // row tiles without those of the pivots, column tiles without the pivots' one
    const int tr = (n + kTileRows - 1) / kTileRows, tc = (n + kGj - 1) / kGj;
    const int kr = kb / kTileRows, kn = (bs + kTileRows - 1) / kTileRows, kc = kb / kGj;
    const int w0 = nbs > 0 ? 1 : 0, workers = gridDim.x - w0;
    const int live = (tr - kn) * (tc - 1);
    int q = (int)blockIdx.x - w0, i0 = 0, j0 = 0;
    auto place = [&]() {  // of tile q, the next pivot block's tiles passed over
        for (;; q += workers) {
            if (q >= live) return false;
            const int r = q / (tc - 1), c = q - r * (tc - 1);
            i0 = (r < kr ? r : r + kn) * kTileRows;
            j0 = (c < kc ? c : c + 1) * kGj;
            if (!(nbs > 0 && i0 / kGj * kGj == nb && j0 == nb)) return true;
        }
    };
    bool more = place();
    if (more) fetch(i0, kTileRows, j0);
    while (more) {
        const int ci = i0, cj = j0;
        update(ci, kTileRows, cj, [&] {
            q += workers;
            more = place();
            if (more) fetch(i0, kTileRows, j0);
        });
    }
}

__global__ void k_pinv_finish(int nc, double *M, const double *__restrict__ scal) {
    grid_wait();
    const i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (i64)nc * nc) return;
    M[e] -= 1.0 / (scal[0] * (double)nc * (double)nc);
}

}  // namespace

// CTAs of k_gj_trailing that run at once, one per SM, in whole clusters.  Left to itself the device
// places two CTAs of a cluster on one SM, where they share its FP64 pipe while other SMs idle (the
// update then took twice the time); asking for more than half of an SM's shared memory keeps them apart.
constexpr int kTrailSmem = 118 * 1024;
int trailing_ctas() {
    static const int ctas = [] {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kTrailCluster);
        cfg.blockDim = dim3(kTrailThreads);
        cfg.dynamicSmemBytes = kTrailSmem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kTrailCluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_gj_trailing, &cfg) != cudaSuccess || n < 1) {
            (void)cudaGetLastError();
            return device_sms() / kTrailCluster * kTrailCluster;  // a grid size only
        }
        return n * kTrailCluster;
    }();
    return ctas;
}

// P^-1, the old column panel, the shift
size_t coarse_scratch_doubles(Dims d) { return (size_t)kGj * kGj + (size_t)d.n * kGj + 1; }

void launch_coarse_pinv(cudaStream_t s, Dims d, double ih2, const double *fx, const double *fy, const double *fz,
                        double *M, double *scratch) {
    const int n = (int)d.n, tiles = (n + kPanel - 1) / kPanel;
    double *Pinv = scratch, *C = Pinv + kGj * kGj, *scal = C + (size_t)n * kGj;
    const int sms = device_sms();
    static std::atomic<unsigned long long> opted{0};
    if (!opt_in_smem((const void *)k_gj_trailing, kTrailSmem, opted)) return;
    // fewer CTAs where there are fewer tiles (and at least the pivot cluster)
    const int live = (n + kTileRows - 1) / kTileRows * ((n + kGj - 1) / kGj) + 1, most = trailing_ctas();
    const int grid = live < most ? (live + kTrailCluster - 1) / kTrailCluster * kTrailCluster : most;
    count_launch();
    run_kernel(k_coarse_assemble, n < sms ? n : sms, 1024, 0, s, d, ih2, fx, fy, fz, M, scal);
    count_launch();
    run_kernel(k_gj_trailing, kTrailCluster, kTrailThreads, kTrailSmem, s, n, -1, 0, 0, n < kGj ? n : kGj, M, C, Pinv);
    for (int kb = 0; kb < n; kb += kGj) {
        const int bs = n - kb < kGj ? n - kb : kGj, nb = kb + kGj, left = n - nb;
        const int nbs = left <= 0 ? 0 : (left < kGj ? left : kGj);
        count_launch(2);
        run_kernel(k_gj_panels, 2 * tiles, 256, 0, s, n, kb, bs, tiles, M, Pinv, C);
        run_kernel(k_gj_trailing, grid, kTrailThreads, kTrailSmem, s, n, kb, bs, nb, nbs, M, C, Pinv);
    }
    count_launch();
    run_kernel(k_pinv_finish, (unsigned)(((i64)n * n + 255) / 256), 256, 0, s, n, M, scal);
}

}  // namespace mg
