// Set-up of the dense coarse solve: the pseudo-inverse A^+ of the coarsest operator (at most
// 1024 cells), by block elimination along the longest axis.
//
// Ordered in planes across its longest axis the operator is block tridiagonal: L planes of m
// cells (m <= 101), the blocks between planes diagonal (one face per cell).  With Schur
// complements taken from both ends towards the middle plane,
//     W_k = (A_kk - F W_(k-1) F)^-1   from below,   W_k = (A_kk - F' W_(k+1) F')^-1   from above,
// F the diagonal of face coefficients between the two planes, and in the middle
//     W_mid = (A_mid - both terms + c 1 1^T)^-1,
// which inverts A + c v v^T, v the indicator of the middle plane (the middle Schur complement
// is singular, its null vector the constants; v v^T does not change A^+ r, because a zero-sum
// right-hand side gives v . x = 0).  Each column of that inverse G is one elimination towards
// the middle and one back-substitution outwards with the W_k, and A^+ = P G P with
// P = I - 1 1^T / n, which is G minus its row and column means plus its mean.
//
// What bounds it: GB300 issues two FP64 FMAs per SM and clock, so the n^3 FMAs of inverting the
// n x n matrix itself take 0.21 ms (n = 512) to 1.7 ms (n = 1024) on all SMs, and its launches
// as many again; the plane inverses and substitutions take about L m^3 + 3 n^2 m, a tenth of
// that, but the m pivots of every plane are one serial chain (about 400 clocks each).  Two
// clusters of eight CTAs run the two chains side by side with rows spread over the cluster, and
// the pivot rows travel through distributed shared memory.  Against Gauss-Jordan on A + c 1 1^T
// by blocks of 32 pivots (4 launches per block) a 64^3 projection step (512 coarse cells) went
// from 3.68 to 2.50 ms and an 88 x 80 x 72 one (990 coarse cells) from 10.4 to 7.2 ms; the error of
// A^+ r against extended precision went from 2.3e-14 to 1.3e-15 (drop and film, 8^3).
#include <cooperative_groups.h>

#include "mg_internal.cuh"

namespace cg = cooperative_groups;

namespace mg {

namespace {

constexpr int kCl = 8;      // CTAs per cluster
constexpr int kPb = 8;      // pivots per step (rows of one CTA)
constexpr int kMaxM = 104;  // cells per plane, rounded up to kPb: m <= 1024^(2/3) < 102
constexpr int kSlots = 16;  // rows per CTA: ceil(kMaxM / (kCl * kPb)) * kPb

// the coarsest level seen as L planes of m = n0 x n1 cells across its longest axis
struct CoarseGeo {
    int m, L, mid, n0, n1, n;
    int s0, s1, sk;              // natural strides of the in-plane axes and of the block axis
    const double *f0, *f1, *fk;  // low faces along them
    double ih2;
};

__device__ __forceinline__ int nat_of(const CoarseGeo &g, int k, int q) {
    const int v = q / g.n0, u = q - v * g.n0;
    return k * g.sk + v * g.s1 + u * g.s0;
}

// sum of the interior faces of cell q of plane k, times ih2
__device__ double diag_of(const CoarseGeo &g, int k, int q) {
    const int v = q / g.n0, u = q - v * g.n0, c = nat_of(g, k, q);
    double s = 0.0;
    if (u > 0) s += g.f0[c] * g.ih2;
    if (u < g.n0 - 1) s += g.f0[c + g.s0] * g.ih2;
    if (v > 0) s += g.f1[c] * g.ih2;
    if (v < g.n1 - 1) s += g.f1[c + g.s1] * g.ih2;
    if (k > 0) s += g.fk[c] * g.ih2;
    if (k < g.L - 1) s += g.fk[c + g.sk] * g.ih2;
    return s;
}

// entry (q, j) of plane k's diagonal block
__device__ double entry_of(const CoarseGeo &g, int k, int q, int j) {
    if (j == q) return diag_of(g, k, q);
    const int v = q / g.n0, u = q - v * g.n0, c = nat_of(g, k, q);
    if (u > 0 && j == q - 1) return -g.f0[c] * g.ih2;
    if (u < g.n0 - 1 && j == q + 1) return -g.f0[c + g.s0] * g.ih2;
    if (v > 0 && j == q - g.n0) return -g.f1[c] * g.ih2;
    if (v < g.n1 - 1 && j == q + g.n0) return -g.f1[c + g.s1] * g.ih2;
    return 0.0;
}

// inverse of the bs x bs block P (rows of stride ld) by one warp, without pivoting (P is
// symmetric positive definite): lane l holds entries (l / 8, l % 8) and (l / 8 + 4, l % 8); the
// block is padded with the identity
__device__ __forceinline__ void warp_inv8(const double *P, int ld, int bs, double *out) {
    const int l = threadIdx.x & 31, c = l & 7, r0 = l >> 3, r1 = r0 + 4;
    double a0 = (r0 < bs && c < bs) ? P[r0 * ld + c] : (r0 == c ? 1.0 : 0.0);
    double a1 = (r1 < bs && c < bs) ? P[r1 * ld + c] : (r1 == c ? 1.0 : 0.0);
#pragma unroll
    for (int k = 0; k < kPb; ++k) {
        const int rl = (k & 3) * 8;  // lanes of row k
        const double src = k < 4 ? a0 : a1;
        const double rp = recip64(__shfl_sync(0xffffffffu, src, rl + k));
        const double rowc = __shfl_sync(0xffffffffu, src, rl + c);
        const double c0 = __shfl_sync(0xffffffffu, a0, r0 * 8 + k), c1 = __shfl_sync(0xffffffffu, a1, r0 * 8 + k);
        const double s = c == k ? rp : rowc * rp;
        a0 = r0 == k ? s : (c == k ? -c0 * rp : fma(-c0, s, a0));
        a1 = r1 == k ? s : (c == k ? -c1 * rp : fma(-c1, s, a1));
    }
    out[r0 * 8 + c] = a0;
    out[r1 * 8 + c] = a1;
}

// W_k of the planes below the middle (cluster 0) and above it (cluster 1), or, with `middle`,
// of the middle plane (one cluster).  Row block j of 8 rows lives in CTA j % 8; a step takes
// one row block as pivots: its owner inverts the 8 x 8 pivot block, and after the cluster
// barrier every CTA fetches that inverse and the pivot rows and updates its own rows,
//     M_ij <- M_ij - (M_iK P^-1) M_Kj,   M_iK <- -M_iK P^-1,   M_Kj <- P^-1 M_Kj,   M_KK <- P^-1.
// Every loop has a fixed count; the only waits are block and cluster barriers.
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(256) k_coarse_planes(CoarseGeo g, double *W, int middle) {
    __shared__ double M[kSlots][kMaxM];
    __shared__ double own[2][kPb][kMaxM];  // pivot rows of the steps this CTA owns, read by the others
    __shared__ double ownP[2][kPb * kPb];
    __shared__ double R[kPb][kMaxM], P[kPb * kPb];
    __shared__ double fl[kMaxM], fh[kMaxM];
    __shared__ double shift;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), side = blockIdx.x / kCl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m = g.m, mp = (m + kPb - 1) / kPb * kPb, nb = mp / kPb;
    auto row_of = [&](int s) { return ((s / kPb) * kCl + rank) * kPb + s % kPb; };
    const int planes = middle ? 1 : (side == 0 ? g.mid : g.L - 1 - g.mid);
    int buf = 0;  // alternates over all steps: a buffer is rewritten two cluster barriers after its readers' step
    for (int t = 0; t < planes; ++t) {
        const int k = middle ? g.mid : (side == 0 ? t : g.L - 1 - t);
        // faces to the eliminated neighbours, and the shift of the middle plane
        const bool lo = middle ? k > 0 : (side == 0 && t > 0);
        const bool hi = middle ? k < g.L - 1 : (side == 1 && t > 0);
        for (int q = tid; q < m; q += 256) {
            const int c = nat_of(g, k, q);
            fl[q] = lo ? g.fk[c] * g.ih2 : 0.0;
            fh[q] = hi ? g.fk[c + g.sk] * g.ih2 : 0.0;
        }
        if (middle && warp == 0) {
            double s = 0.0;
            for (int q = lane; q < m; q += 32) s += diag_of(g, k, q);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) shift = s / m / m;
        }
        __syncthreads();
        for (int e = tid; e < kSlots * mp; e += 256) {
            const int s = e / mp, j = e - s * mp, q = row_of(s);
            double v = 0.0;
            if (q < m && j < m) {
                v = entry_of(g, k, q, j);
                if (middle) {
                    const i64 o = (i64)q * m + j, mm = (i64)m * m;
                    if (lo) v -= fl[q] * W[(k - 1) * mm + o] * fl[j];
                    if (hi) v -= fh[q] * W[(k + 1) * mm + o] * fh[j];
                    v += shift;
                } else if (t > 0) {  // this CTA's rows of the neighbour's inverse are still in M
                    v -= side == 0 ? fl[q] * M[s][j] * fl[j] : fh[q] * M[s][j] * fh[j];
                }
            }
            M[s][j] = v;
        }
        __syncthreads();
        for (int kb = 0; kb < nb; ++kb) {
            const int k0 = kb * kPb, bs = min(kPb, m - k0), owner = kb % kCl;
            if (rank == owner) {
                const int s0 = (kb / kCl) * kPb;
                if (warp == 0) warp_inv8(&M[s0][k0], kMaxM, bs, ownP[buf]);
                for (int e = tid; e < kPb * mp; e += 256) own[buf][e / mp][e % mp] = M[s0 + e / mp][e % mp];
            }
            cl.sync();
            const double *src = cl.map_shared_rank(&own[buf][0][0], owner);
            const double *srcP = cl.map_shared_rank(&ownP[buf][0], owner);
            for (int e = tid; e < kPb * mp; e += 256) R[e / mp][e % mp] = src[(e / mp) * kMaxM + e % mp];
            if (tid < kPb * kPb) P[tid] = srcP[tid];
            __syncthreads();
            for (int s = warp; s < kSlots; s += 8) {
                const int q = row_of(s);
                if (q >= m) continue;  // the same for the whole warp
                const bool piv = q >= k0 && q < k0 + kPb;
                // coefficients of the pivot rows: T = M_iK P^-1, for a pivot row -P^-1's row
                double T[kPb];
#pragma unroll
                for (int a = 0; a < kPb; ++a) T[a] = 0.0;
                if (piv) {
#pragma unroll
                    for (int a = 0; a < kPb; ++a) T[a] = -P[(q - k0) * kPb + a];
                } else {
                    double mine = 0.0;
                    if (lane < kPb) {
#pragma unroll
                        for (int a = 0; a < kPb; ++a) mine = fma(M[s][k0 + a], P[a * kPb + lane], mine);
                    }
#pragma unroll
                    for (int a = 0; a < kPb; ++a) T[a] = __shfl_sync(0xffffffffu, mine, a);
                }
                __syncwarp();  // every lane has read M[s][k0..k0+7] before it is overwritten
                for (int j = lane; j < mp; j += 32) {
                    double v;
                    if (j >= k0 && j < k0 + kPb) {
                        v = 0.0;
#pragma unroll
                        for (int a = 0; a < kPb; ++a) v = (j - k0 == a) ? -T[a] : v;
                        if (j >= m) v = 0.0;
                    } else {
                        v = piv ? 0.0 : M[s][j];
#pragma unroll
                        for (int a = 0; a < kPb; ++a) v = fma(-T[a], R[a][j], v);
                    }
                    M[s][j] = v;
                }
            }
            __syncthreads();
            buf ^= 1;
        }
        for (int e = tid; e < kSlots * m; e += 256) {
            const int s = e / m, j = e - s * m, q = row_of(s);
            if (q < m) W[(i64)k * m * m + (i64)q * m + j] = M[s][j];
        }
        __syncthreads();  // M is read above and rewritten for the next plane
    }
    cl.sync();  // no CTA leaves while another may still read its shared memory
}

// Columns of G, four of one plane per CTA: elimination from their plane to the middle, then
// substitution outwards to both ends.  A thread takes one row i and a part of the sum over t of
// a plane product (W is symmetric: row t is read along i, coalesced, from L2); the parts are
// added in a fixed order.  G's column c goes to row c of M (G is symmetric) and its mean to cm.
constexpr int kCols = 4;
__global__ void __launch_bounds__(256) k_coarse_columns(CoarseGeo g, const double *__restrict__ W, double *M,
                                                        double *cm) {
    __shared__ double X[1024 * kCols];  // W_k y_k of the planes passed, then x (plane order)
    __shared__ double v[kMaxM * kCols], red[256 * kCols];
    const int tid = threadIdx.x, m = g.m, ng = (m + kCols - 1) / kCols;
    const int j = blockIdx.x / ng, q0 = (blockIdx.x - j * ng) * kCols;
    const int iw = (m + 31) / 32 * 32, parts = 256 / iw;
    const int i = tid % iw, part = tid / iw, per = (m + parts - 1) / parts;
    const bool act = part < parts && i < m;
    // X_k = W_k v (+ the X_k already there)
    auto plane_product = [&](int k, bool add) {
        double a[kCols] = {0.0, 0.0, 0.0, 0.0};
        if (act) {
            const double *w = W + (i64)k * m * m + i;
            const int t1 = min(m, (part + 1) * per);
#pragma unroll 4
            for (int t = part * per; t < t1; ++t) {
                const double wt = w[(i64)t * m];
#pragma unroll
                for (int c = 0; c < kCols; ++c) a[c] = fma(wt, v[t * kCols + c], a[c]);
            }
#pragma unroll
            for (int c = 0; c < kCols; ++c) red[(part * iw + i) * kCols + c] = a[c];
        }
        __syncthreads();
        for (int e = tid; e < m * kCols; e += 256) {
            double s = 0.0;
            for (int p = 0; p < parts; ++p) s += red[p * iw * kCols + e];
            const int o = k * m * kCols + e;
            X[o] = add ? X[o] + s : s;
        }
        __syncthreads();
    };
    // v = F X_k, F the faces between plane k and plane kn
    auto step = [&](int k, int kn) {
        for (int e = tid; e < m * kCols; e += 256) {
            const int q = e / kCols;
            v[e] = g.fk[nat_of(g, max(k, kn), q)] * g.ih2 * X[k * m * kCols + e];
        }
        __syncthreads();
    };
    for (int e = tid; e < m * kCols; e += 256) v[e] = (e / kCols == q0 + e % kCols) ? 1.0 : 0.0;
    __syncthreads();
    for (int k = j; k != g.mid;) {
        const int kn = k < g.mid ? k + 1 : k - 1;
        plane_product(k, false);
        step(k, kn);
        k = kn;
    }
    plane_product(g.mid, false);
    for (int k = g.mid - 1; k >= 0; --k) {
        step(k + 1, k);
        plane_product(k, j < g.mid && k >= j);
    }
    for (int k = g.mid + 1; k < g.L; ++k) {
        step(k - 1, k);
        plane_product(k, j > g.mid && k <= j);
    }
    for (int c = 0; c < kCols && q0 + c < m; ++c) {
        const int col = nat_of(g, j, q0 + c);
        double s = 0.0;
        for (int e = tid; e < g.n; e += 256) {
            const double x = X[e * kCols + c];
            M[(i64)col * g.n + nat_of(g, e / m, e % m)] = x;
            s += x;
        }
        red[tid] = s;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if (tid < w) red[tid] += red[tid + w];
            __syncthreads();
        }
        if (tid == 0) cm[col] = red[0] / g.n;
        __syncthreads();
    }
}

// A^+ = P G P: row blockIdx.x of G minus its mean, the column means and plus the mean of all
__global__ void __launch_bounds__(256) k_coarse_center(int n, double *M, const double *__restrict__ cm) {
    __shared__ double red[256];
    const int tid = threadIdx.x, r = blockIdx.x;
    double s = 0.0;
    for (int e = tid; e < n; e += 256) s += cm[e];
    red[tid] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (tid < w) red[tid] += red[tid + w];
        __syncthreads();
    }
    const double mean = red[0] / n, own = cm[r];
    for (int e = tid; e < n; e += 256) M[(i64)r * n + e] -= (own - mean) + cm[e];
}

}  // namespace

// W_k of every plane (n m doubles) and the column means (n)
size_t coarse_scratch_doubles(Dims d) {
    const int L = d.nx > d.ny ? (d.nx > d.nz ? d.nx : d.nz) : (d.ny > d.nz ? d.ny : d.nz);
    return (size_t)d.n * (size_t)(d.n / L) + (size_t)d.n;
}

void launch_coarse_pinv(cudaStream_t s, Dims d, double ih2, const double *fx, const double *fy, const double *fz,
                        double *M, double *scratch) {
    CoarseGeo g;
    const int nxy = (int)d.nxy;
    if (d.nz >= d.nx && d.nz >= d.ny) g = CoarseGeo{nxy, d.nz, 0, d.nx, d.ny, 0, 1, d.nx, nxy, fx, fy, fz, ih2};
    else if (d.ny >= d.nx) g = CoarseGeo{d.nx * d.nz, d.ny, 0, d.nx, d.nz, 0, 1, nxy, d.nx, fx, fz, fy, ih2};
    else g = CoarseGeo{d.ny * d.nz, d.nx, 0, d.ny, d.nz, 0, d.nx, nxy, 1, fy, fz, fx, ih2};
    g.n = (int)d.n;
    g.mid = g.L / 2;
    double *W = scratch, *cm = scratch + (size_t)g.n * g.m;
    count_launch(4);
    k_coarse_planes<<<2 * kCl, 256, 0, s>>>(g, W, 0);
    k_coarse_planes<<<kCl, 256, 0, s>>>(g, W, 1);
    k_coarse_columns<<<g.L * ((g.m + kCols - 1) / kCols), 256, 0, s>>>(g, W, M, cm);
    k_coarse_center<<<g.n, 256, 0, s>>>(g.n, M, cm);
}

}  // namespace mg
