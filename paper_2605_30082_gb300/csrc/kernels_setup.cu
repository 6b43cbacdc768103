// Set-up kernels: density mixing (Eq. (5)), face coefficients, coarsening,
// inverse diagonals, precision copies, CSF faces and RHS assembly.  All FP64, one thread per cell (these run once per
// density field, not inside the V-cycle).
#include "mg_internal.cuh"

namespace mg {

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(i64 n) { return (unsigned)((n + kThreads - 1) / kThreads); }

struct FracArgs {
    const double *f[4];
    double drho[4];  // rho_q - rho_last
    double rho_last;
    int nfrac;
};

// Eq. (5) in the form rho_last + sum_q (rho_q - rho_last) f_q: one FMA per fraction (the
// literal sum_q rho_q f_q + rho_last (1 - sum_q f_q) takes 2 nfrac + 1 FP64 operations, which
// bound this kernel by the FP64 pipe); equal in exact arithmetic, within a few units in the
// last place in FP64.  Four cells per thread, all loads before the arithmetic, 16 bytes each
// where every array is on such a boundary (VEC): one cell per thread, the fractions one after another, took
// 181 us at 256^3 with two of them (24 bytes a cell, 59 us), now 61 us.
constexpr int kDensThreads = 256;
template <int NF, bool VEC>
__global__ void __launch_bounds__(kDensThreads) k_density(i64 n, FracArgs a, double *rho) {
    grid_wait();
    constexpr int kPer = VEC ? 2 : 4;  // loads per array and thread
    using V = typename std::conditional<VEC, double2, double>::type;
    const i64 nv = VEC ? n / 2 : n, m0 = (i64)blockIdx.x * (kPer * kDensThreads) + threadIdx.x;
    V f[NF][kPer];
#pragma unroll
    for (int q = 0; q < NF; ++q)
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const i64 m = m0 + u * kDensThreads;
            if (m < nv) f[q][u] = reinterpret_cast<const V *>(a.f[q])[m];
        }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const i64 m = m0 + u * kDensThreads;
        if (m >= nv) continue;
        if constexpr (VEC) {
            double2 r = make_double2(a.rho_last, a.rho_last);
#pragma unroll
            for (int q = 0; q < NF; ++q) r = make_double2(fma(a.drho[q], f[q][u].x, r.x), fma(a.drho[q], f[q][u].y, r.y));
            reinterpret_cast<double2 *>(rho)[m] = r;
        } else {
            double r = a.rho_last;
#pragma unroll
            for (int q = 0; q < NF; ++q) r = fma(a.drho[q], f[q][u], r);
            rho[m] = r;
        }
    }
    if (VEC && (n & 1) && m0 == 0) {  // the last cell of an odd number
        double r = a.rho_last;
#pragma unroll
        for (int q = 0; q < NF; ++q) r = fma(a.drho[q], a.f[q][n - 1], r);
        rho[n - 1] = r;
    }
}
template <int NF>
void run_density(cudaStream_t s, i64 n, const FracArgs &a, double *rho) {
    bool vec = (reinterpret_cast<uintptr_t>(rho) & 15) == 0;
    for (int q = 0; q < NF; ++q) vec = vec && (reinterpret_cast<uintptr_t>(a.f[q]) & 15) == 0;
    const unsigned nb = (unsigned)((n + 4 * kDensThreads - 1) / (4 * kDensThreads));
    run_kernel(vec ? k_density<NF, true> : k_density<NF, false>, nb, kDensThreads, 0, s, n, a, rho);
}

// 0 < v <= 1.79e308, tested on the bit pattern (positive doubles order like their bits, NaN and
// infinity lie above the bound, negative values and zero at or below 0): no FP64 comparison
__device__ __forceinline__ bool good_positive(double v) {
    const long long u = __double_as_longlong(v);
    return u > 0 && u <= 0x7fefdcf158adbb99ll;
}

// v / 2 for v = 0 or normal with a normal result (exponent field above 1): one integer subtraction
// from the exponent field instead of an FP64 multiplication; otherwise the multiplication, in a function of its own:
// in line the compiler computes it for every value (the faces of 256^3 190 us, so 101)
__device__ __noinline__ double half_slow(double v) { return 0.5 * v; }
__device__ __forceinline__ double half_of(double v) {
    const long long u = __double_as_longlong(v);
    const int e = (int)((u >> 52) & 0x7ff);
    if (e > 1 && e < 0x7ff) return __longlong_as_double(u - (1ll << 52));
    return half_slow(v);
}

// s = 1/rho per cell, validating rho (finite and > 0)
__global__ void k_inv_rho(i64 n, const double *__restrict__ rho, double *sinv, unsigned *err) {
    grid_wait();
    const i64 m = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n) return;
    const double r = rho[m];
    if (!good_positive(r)) {
        atomicOr(err, 1u);
        sinv[m] = 1.0;
        return;
    }
    sinv[m] = recip64(r);
}

// the same for even nx and 16-byte boundaries, two cells per thread, with the FP32 copies of a mixed handle (s32 in
// the level's layout, optionally s2 as pairs of FP32 numbers hi + lo = s to about 2^-48) in the same
// pass: 256^3 122 + 90 us apart, now 122 us (its FP64 arithmetic)
__global__ void k_inv_rho_pack(Lay L, const double *__restrict__ rho, double *sinv, float *s32, float2 *s2, unsigned *err) {
    grid_wait();
    const i64 m = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= L.half) return;
    const double2 r = reinterpret_cast<const double2 *>(rho)[m];
    const bool g0 = good_positive(r.x), g1 = good_positive(r.y);
    if (!g0 || !g1) atomicOr(err, 1u);
    const double2 v = make_double2(g0 ? recip64(r.x) : 1.0, g1 ? recip64(r.y) : 1.0);
    reinterpret_cast<double2 *>(sinv)[m] = v;
    const unsigned row = (unsigned)m / (unsigned)L.hx;
    const bool red_first = ((row % (unsigned)L.ny + row / (unsigned)L.ny) & 1) == 0;
    const float h0 = d2f_rn(v.x), h1 = d2f_rn(v.y);
    s32[m] = red_first ? h0 : h1;
    s32[L.half + m] = red_first ? h1 : h0;
    if (s2)
        reinterpret_cast<float4 *>(s2)[m] = make_float4(h0, d2f_rn(v.x - f2d_exact(h0)), h1, d2f_rn(v.y - f2d_exact(h1)));
}

// beta on the low faces: 1 / harmonic mean of the two densities = (s_L + s_R) / 2; blocks take
// rows (grid y, strided), threads the cells of a row
__global__ void k_faces_from_s(Dims d, const double *__restrict__ sv, double *fx, double *fy, double *fz) {
    grid_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= d.nx) return;
    const i64 rows = (i64)d.ny * d.nz;
    for (i64 row = blockIdx.y; row < rows; row += gridDim.y) {
        const int j = (int)((unsigned)row % (unsigned)d.ny), k = (int)((unsigned)row / (unsigned)d.ny);  // rows < 2^31
        const i64 c = row * d.nx + i;
        const double sc = sv[c];
        fx[c] = i > 0 ? half_of(sv[c - 1] + sc) : 0.0;
        fy[c] = j > 0 ? half_of(sv[c - d.nx] + sc) : 0.0;
        fz[c] = k > 0 ? half_of(sv[c - d.nxy] + sc) : 0.0;
    }
}

// the same for even nx, two cells per thread: 16-byte loads and stores (the x - 1 value of the
// pair's first cell is one scalar load, from the line the neighbouring lane reads); the same
// additions in the same order as k_faces_from_s, so bitwise the same faces
__global__ void k_faces_from_s2(Dims d, const double *__restrict__ sv, double *fx, double *fy, double *fz) {
    grid_wait();
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= d.nx) return;
    const i64 rows = (i64)d.ny * d.nz;
    auto ld2 = [](const double *q) { return *reinterpret_cast<const double2 *>(q); };
    auto st2 = [](double *q, double a, double b) { *reinterpret_cast<double2 *>(q) = make_double2(a, b); };
    for (i64 row = blockIdx.y; row < rows; row += gridDim.y) {
        const int j = (int)((unsigned)row % (unsigned)d.ny), k = (int)((unsigned)row / (unsigned)d.ny);  // rows < 2^31
        const i64 c = row * d.nx + i;
        // all loads at once (at a wall the cell itself)
        const double2 sc = ld2(sv + c), sy = ld2(sv + (j > 0 ? c - d.nx : c)), sz = ld2(sv + (k > 0 ? c - d.nxy : c));
        const double sl = sv[i > 0 ? c - 1 : c];
        st2(fx + c, i > 0 ? half_of(sl + sc.x) : 0.0, half_of(sc.x + sc.y));
        st2(fy + c, j > 0 ? half_of(sy.x + sc.x) : 0.0, j > 0 ? half_of(sy.y + sc.y) : 0.0);
        st2(fz + c, k > 0 ? half_of(sz.x + sc.x) : 0.0, k > 0 ? half_of(sz.y + sc.y) : 0.0);
    }
}

__global__ void k_faces_from_api(Dims d, const double *__restrict__ bx, const double *__restrict__ by,
                                 const double *__restrict__ bz, double *fx, double *fy, double *fz,
                                 unsigned *err) {
    grid_wait();
    i64 c = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.n) return;
    const unsigned cu_ = (unsigned)c, ru_ = cu_ / (unsigned)d.nx;  // c < 2^32: 32-bit divisions
    int i = (int)(cu_ - ru_ * (unsigned)d.nx);
    int j = (int)(ru_ % (unsigned)d.ny);
    int k = (int)(ru_ / (unsigned)d.ny);
    double vx = 0.0, vy = 0.0, vz = 0.0;
    if (i > 0) vx = bx[((i64)k * d.ny + j) * (d.nx + 1) + i];
    if (j > 0) vy = by[((i64)k * (d.ny + 1) + j) * d.nx + i];
    if (k > 0) vz = bz[c];  // (nz+1, ny, nx): plane k starts at k*nxy
    if ((i > 0 && !good_positive(vx)) || (j > 0 && !good_positive(vy)) ||
        (k > 0 && !good_positive(vz)))
        atomicOr(err, 1u);
    fx[c] = vx;
    fy[c] = vy;
    fz[c] = vz;
}

__global__ void k_faces_to_api(Dims d, const double *__restrict__ fx, const double *__restrict__ fy,
                               const double *__restrict__ fz, double *bx, double *by, double *bz) {
    grid_wait();
    i64 c = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.n) return;
    const unsigned cu_ = (unsigned)c, ru_ = cu_ / (unsigned)d.nx;  // c < 2^32: 32-bit divisions
    int i = (int)(cu_ - ru_ * (unsigned)d.nx);
    int j = (int)(ru_ % (unsigned)d.ny);
    int k = (int)(ru_ / (unsigned)d.ny);
    i64 ax = ((i64)k * d.ny + j) * (d.nx + 1) + i;
    i64 ay = ((i64)k * (d.ny + 1) + j) * d.nx + i;
    bx[ax] = i > 0 ? fx[c] : 0.0;
    by[ay] = j > 0 ? fy[c] : 0.0;
    bz[c] = k > 0 ? fz[c] : 0.0;
    if (i == d.nx - 1) bx[ax + 1] = 0.0;
    if (j == d.ny - 1) by[ay + d.nx] = 0.0;
    if (k == d.nz - 1) bz[c + d.nxy] = 0.0;
}

__global__ void k_invdiag(Dims d, const double *__restrict__ fx, const double *__restrict__ fy,
                          const double *__restrict__ fz, double *invd64, i64 invd_half, double *diag) {
    grid_wait();
    i64 c = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.n) return;
    const unsigned cu_ = (unsigned)c, ru_ = cu_ / (unsigned)d.nx;  // c < 2^32: 32-bit divisions
    int i = (int)(cu_ - ru_ * (unsigned)d.nx);
    int j = (int)(ru_ % (unsigned)d.ny);
    int k = (int)(ru_ / (unsigned)d.ny);
    // order x-, x+, y-, y+, z-, z+ (low faces of i=0 etc. are stored as 0)
    double s = fx[c];
    if (i < d.nx - 1) s += fx[c + 1];
    s += fy[c];
    if (j < d.ny - 1) s += fy[c + d.nx];
    s += fz[c];
    if (k < d.nz - 1 || d.zhi) s += fz[c + d.nxy];  // a slab's face to its ghost plane counts
    // colour by colour (invd_half = n / 2, even nx) or, with invd_half 0, in natural order
    if (invd64) invd64[invd_half ? ((i + j + k) & 1) * invd_half + (c >> 1) : c] = recip64(s);
    if (diag) diag[c] = s;
}

// coarse low face = mean of the 4 fine low faces that tile it; with c32x, .. also rounded to FP32 in the layout L (a
// launch less per array and level)
__global__ void k_coarsen(Dims f, Dims cd, const double *__restrict__ ffx,
                          const double *__restrict__ ffy, const double *__restrict__ ffz,
                          double *cfx, double *cfy, double *cfz, Lay L, float *c32x, float *c32y, float *c32z) {
    grid_wait();
    i64 C = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (C >= cd.n) return;
    const unsigned cu = (unsigned)C, ru = cu / (unsigned)cd.nx;  // C < 2^32: 32-bit divisions
    const int I = (int)(cu - ru * (unsigned)cd.nx);
    const int J = (int)(ru % (unsigned)cd.ny);
    const int K = (int)(ru / (unsigned)cd.ny);
    i64 base = ((i64)(2 * K) * f.ny + 2 * J) * f.nx + 2 * I;  // child (0,0,0)
    double sx = 0.0, sy = 0.0, sz = 0.0;
    for (int c = 0; c < 2; ++c)
        for (int b = 0; b < 2; ++b) sx += ffx[base + c * f.nxy + b * f.nx];
    for (int c = 0; c < 2; ++c)
        for (int a = 0; a < 2; ++a) sy += ffy[base + c * f.nxy + a];
    for (int b = 0; b < 2; ++b)
        for (int a = 0; a < 2; ++a) sz += ffz[base + b * f.nx + a];
    sx /= 4.0;
    sy /= 4.0;
    sz /= 4.0;
    cfx[C] = sx;
    cfy[C] = sy;
    cfz[C] = sz;
    if (c32x) {
        const i64 t = L.split ? ((I + J + K) & 1) * L.half + (i64)ru * L.hx + (I >> 1) : C;
        c32x[t] = d2f_rn(sx);
        c32y[t] = d2f_rn(sy);
        c32z[t] = d2f_rn(sz);
    }
}

__global__ void k_to_f32(i64 n, const double *__restrict__ src, float *dst) {
    grid_wait();
    i64 m = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (m < n) dst[m] = (float)src[m];
}

__global__ void k_csf_faces(Dims d, double ih, const double *__restrict__ f,
                            const double *__restrict__ kap, double *cx, double *cy, double *cz) {
    grid_wait();
    i64 c = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.n) return;
    const unsigned cu_ = (unsigned)c, ru_ = cu_ / (unsigned)d.nx;  // c < 2^32: 32-bit divisions
    int i = (int)(cu_ - ru_ * (unsigned)d.nx);
    int j = (int)(ru_ % (unsigned)d.ny);
    int k = (int)(ru_ / (unsigned)d.ny);
    i64 ax = ((i64)k * d.ny + j) * (d.nx + 1) + i;
    i64 ay = ((i64)k * (d.ny + 1) + j) * d.nx + i;
    // the mean's 1/2 goes with ih: four FP64 operations per face, which bound this kernel (256^3: five
    // 484 us, four 420)
    const double fc = f[c], kc = kap[c], ih_2 = 0.5 * ih;
    cx[ax] = i > 0 ? (kap[c - 1] + kc) * (fc - f[c - 1]) * ih_2 : 0.0;
    cy[ay] = j > 0 ? (kap[c - d.nx] + kc) * (fc - f[c - d.nx]) * ih_2 : 0.0;
    cz[c] = k > 0 ? (kap[c - d.nxy] + kc) * (fc - f[c - d.nxy]) * ih_2 : 0.0;
    if (i == d.nx - 1) cx[ax + 1] = 0.0;
    if (j == d.ny - 1) cy[ay + d.nx] = 0.0;
    if (k == d.nz - 1) cz[c + d.nxy] = 0.0;
}

// b = b0 + D u + sigma D(beta csf); D over interior faces, (+high - low)/h; terms optional
__global__ void k_rhs(Dims d, double ih, const double *b0, const double *__restrict__ ux,
                      const double *__restrict__ uy, const double *__restrict__ uz,
                      const double *__restrict__ fx, const double *__restrict__ fy,
                      const double *__restrict__ fz, const double *__restrict__ csx,
                      const double *__restrict__ csy, const double *__restrict__ csz, double sigma,
                      double *b) {
    grid_wait();
    i64 c = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.n) return;
    const unsigned cu_ = (unsigned)c, ru_ = cu_ / (unsigned)d.nx;  // c < 2^32: 32-bit divisions
    int i = (int)(cu_ - ru_ * (unsigned)d.nx);
    int j = (int)(ru_ % (unsigned)d.ny);
    int k = (int)(ru_ / (unsigned)d.ny);
    i64 ax = ((i64)k * d.ny + j) * (d.nx + 1) + i;
    i64 ay = ((i64)k * (d.ny + 1) + j) * d.nx + i;
    double v = b0 ? b0[c] : 0.0;
    if (ux) {
        // (high - low) per axis, wall faces as 0: five FP64 additions and one fused
        // multiply-add per cell
        const double xm = i > 0 ? ux[ax] : 0.0, xp = i < d.nx - 1 ? ux[ax + 1] : 0.0;
        const double ym = j > 0 ? uy[ay] : 0.0, yp = j < d.ny - 1 ? uy[ay + d.nx] : 0.0;
        const double zm = k > 0 ? uz[c] : 0.0, zp = k < d.nz - 1 ? uz[c + d.nxy] : 0.0;
        const double s = ((xp - xm) + (yp - ym)) + (zp - zm);
        v = fma(s, ih, v);
    }
    if (csx) {
        double t = 0.0;
        if (i > 0) t -= fx[c] * csx[ax];
        if (i < d.nx - 1) t += fx[c + 1] * csx[ax + 1];
        if (j > 0) t -= fy[c] * csy[ay];
        if (j < d.ny - 1) t += fy[c + d.nx] * csy[ay + d.nx];
        if (k > 0) t -= fz[c] * csz[c];
        if (k < d.nz - 1) t += fz[c + d.nxy] * csz[c + d.nxy];
        v += sigma * (t * ih);
    }
    b[c] = v;
}

}  // namespace

void launch_density(cudaStream_t s, i64 n, int nfrac, const double *const *frac,
                    const double *rho_phase, double *rho) {
    FracArgs a;
    a.nfrac = nfrac;
    a.rho_last = rho_phase[nfrac];
    for (int q = 0; q < 4; ++q) {
        a.f[q] = q < nfrac ? frac[q] : nullptr;
        a.drho[q] = q < nfrac ? rho_phase[q] - rho_phase[nfrac] : 0.0;
    }
    count_launch();
    if (nfrac == 1) run_density<1>(s, n, a, rho);
    else if (nfrac == 2) run_density<2>(s, n, a, rho);
    else if (nfrac == 3) run_density<3>(s, n, a, rho);
    else run_density<4>(s, n, a, rho);
}

void launch_faces_from_rho(cudaStream_t s, Dims d, const double *rho, double *sinv, double *fx, double *fy,
                           double *fz, unsigned *err, Lay L, float *s32, float2 *s2) {
    count_launch(2);
    auto a16 = [](const void *q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    if (s32 && d.nx % 2 == 0 && a16(rho) && a16(sinv)) {
        run_kernel(k_inv_rho_pack, blocks_for(d.n / 2), kThreads, 0, s, L, rho, sinv, s32, s2, err);
    } else {
        run_kernel(k_inv_rho, blocks_for(d.n), kThreads, 0, s, d.n, rho, sinv, err);
        if (s32) launch_pack_inv_rho(s, L, sinv, s32, s2);
    }
    const i64 rows = (i64)d.ny * d.nz;
    if (d.nx % 2 == 0 && a16(sinv) && a16(fx) && a16(fy) && a16(fz)) {
        const dim3 grd((unsigned)((d.nx / 2 + 127) / 128), (unsigned)(rows < 65535 ? rows : 65535));
        run_kernel(k_faces_from_s2, grd, 128, 0, s, d, sinv, fx, fy, fz);
        return;
    }
    const dim3 grd((unsigned)((d.nx + 127) / 128), (unsigned)(rows < 65535 ? rows : 65535));
    run_kernel(k_faces_from_s, grd, 128, 0, s, d, sinv, fx, fy, fz);
}

void launch_faces_from_api(cudaStream_t s, Dims d, const double *bx, const double *by,
                           const double *bz, double *fx, double *fy, double *fz, unsigned *err) {
    count_launch();
    run_kernel(k_faces_from_api, blocks_for(d.n), kThreads, 0, s, d, bx, by, bz, fx, fy, fz, err);
}

void launch_faces_to_api(cudaStream_t s, Dims d, const double *fx, const double *fy,
                         const double *fz, double *bx, double *by, double *bz) {
    count_launch();
    run_kernel(k_faces_to_api, blocks_for(d.n), kThreads, 0, s, d, fx, fy, fz, bx, by, bz);
}

void launch_invdiag(cudaStream_t s, Dims d, const double *fx, const double *fy, const double *fz,
                    double *invd64, i64 invd_half, double *diag) {
    if (!invd64 && !diag) return;
    count_launch();
    run_kernel(k_invdiag, blocks_for(d.n), kThreads, 0, s, d, fx, fy, fz, invd64, invd_half, diag);
}

void launch_coarsen(cudaStream_t s, Dims fine, const double *ffx, const double *ffy,
                    const double *ffz, double *cfx, double *cfy, double *cfz, Lay L, float *c32x, float *c32y, float *c32z) {
    Dims cd = make_dims(fine.nx / 2, fine.ny / 2, fine.nz / 2);
    count_launch();
    run_kernel(k_coarsen, blocks_for(cd.n), kThreads, 0, s, fine, cd, ffx, ffy, ffz, cfx, cfy, cfz, L,
               c32x, c32y, c32z);
}

void launch_to_f32(cudaStream_t s, i64 n, const double *src, float *dst) {
    count_launch();
    run_kernel(k_to_f32, blocks_for(n), kThreads, 0, s, n, src, dst);
}

void launch_csf_faces(cudaStream_t s, Dims d, double h, const double *f, const double *kappa,
                      double *cx, double *cy, double *cz) {
    count_launch();
    run_kernel(k_csf_faces, blocks_for(d.n), kThreads, 0, s, d, 1.0 / h, f, kappa, cx, cy, cz);
}

void launch_rhs(cudaStream_t s, Dims d, double h, const double *b0, const double *ux, const double *uy,
                const double *uz, const double *fx, const double *fy, const double *fz,
                const double *csfx, const double *csfy, const double *csfz, double sigma,
                double *b) {
    count_launch();
    run_kernel(k_rhs, blocks_for(d.n), kThreads, 0, s, d, 1.0 / h, b0, ux, uy, uz, fx, fy, fz, csfx, csfy,
                                               csfz, sigma, b);
}

}  // namespace mg
