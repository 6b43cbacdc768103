// FP32 V-cycle kernels on colour-split levels.
//
// Storage: an FP32 level with even nx keeps every cell array colour-split: all
// red cells ((x+y+z) even) first, then all black cells, each colour row by row
// with the cell at x stored at k = x >> 1.  Levels with odd nx (possible only on
// the coarsest level) keep the natural layout.  `sto` maps (x, y, z) to the
// storage index in either case.
//
// For a cell of colour c at (k, y, z), x = 2k + p with p = (c + y + z) & 1, the six
// neighbours all have the other colour and sit in the other half at
//   x-1: k + p - 1,   x+1: k + p      (same row)
//   y-1, y+1, z-1, z+1: k             (the rows above, below, before, after)
// so a half sweep reads the other colour with unit-stride, vectorisable loads and
// no shared memory: 4 B of the other colour's x, 8 B of 1/rho (both colours) or
// 12 B of face coefficients, and 4 B of b per updated cell, plus the write.
//
// Coefficients: SFORM uses s = 1/rho per cell and beta_f = (s_c + s_nb)/2 (the
// finest level when the operator came from a density); otherwise the low-face
// arrays fx, fy, fz (beta of the face between a cell and its x-1, y-1, z-1
// neighbour) stored in the same split layout.
//
// Two exact properties of red-black Gauss-Seidel shorten the V-cycle:
//  - after the last pre-smoothing sweep (black last) every black row is solved,
//    so the black residuals are zero and the restriction sums red residuals only;
//  - the first post-smoothing sweep (black first) overwrites every black cell, so
//    the coarse correction only needs to be added to the red cells.
#include "mg_internal.cuh"

namespace mg {

namespace {

constexpr int kThreads = 256;
inline unsigned blocks_for(i64 n) { return (unsigned)((n + kThreads - 1) / kThreads); }

__device__ __forceinline__ i64 sto(const Lay &L, int x, int y, int z) {
    const i64 row = (i64)z * L.ny + y;
    if (!L.split) return row * L.nx + x;
    return ((x + y + z) & 1) * L.half + row * L.hx + (x >> 1);
}

struct Coef32 {
    const float *s;             // SFORM when non-null
    const float *fx, *fy, *fz;  // face form otherwise
};

// ---- generic (scalar, any layout) stencil pieces --------------------------------------
// sum_f beta_f x_nb and sum_f beta_f at cell (x, y, z), SFORM carries a factor 2
__device__ __forceinline__ void stencil_any(const Lay &L, const Coef32 &cf, const float *__restrict__ xv,
                                            int x, int y, int z, float &num, float &den) {
    const bool hx0 = x > 0, hx1 = x < L.nx - 1, hy0 = y > 0, hy1 = y < L.ny - 1, hz0 = z > 0, hz1 = z < L.nz - 1;
    // offsets fit 32 bits; in split storage all six neighbours are of the other colour, two of them at k + p - 1 and
    // k + p of the row (x = 2 k + p)
    const int row = z * L.ny + y, w = L.split ? L.hx : L.nx, c = (int)sto(L, x, y, z);
    const int o = L.split ? (((x + y + z) & 1) ? 0 : (int)L.half) + row * w + (x >> 1) : c;
    const int n1o = L.split ? o + (x & 1) : c + 1;
    // beyond a wall, with weight 0: o, in split storage a cell of the other colour.  Not the cell itself, which a sweep
    // from zero is the first to write: 0 times a NaN left there by a solve that diverged, or by the memory's last owner,
    // would go into this solve and every later one
    const int n0 = hx0 ? n1o - (L.split ? 1 : 2) : o, n1 = hx1 ? n1o : o;
    const int n2 = hy0 ? o - w : o, n3 = hy1 ? o + w : o;
    const int n4 = hz0 ? o - L.ny * w : o, n5 = hz1 ? o + L.ny * w : o;
    float w0, w1, w2, w3, w4, w5;
    if (cf.s) {
        const float sc = cf.s[c];
        w0 = hx0 ? sc + cf.s[n0] : 0.f;
        w1 = hx1 ? sc + cf.s[n1] : 0.f;
        w2 = hy0 ? sc + cf.s[n2] : 0.f;
        w3 = hy1 ? sc + cf.s[n3] : 0.f;
        w4 = hz0 ? sc + cf.s[n4] : 0.f;
        w5 = hz1 ? sc + cf.s[n5] : 0.f;
    } else {
        w0 = cf.fx[c];
        w1 = hx1 ? cf.fx[n1] : 0.f;
        w2 = cf.fy[c];
        w3 = hy1 ? cf.fy[n3] : 0.f;
        w4 = cf.fz[c];
        w5 = hz1 ? cf.fz[n5] : 0.f;
    }
    float nm = w0 * xv[n0];
    nm += w1 * xv[n1];
    nm += w2 * xv[n2];
    nm += w3 * xv[n3];
    nm += w4 * xv[n4];
    nm += w5 * xv[n5];
    num = nm;
    den = ((w0 + w1) + (w2 + w3)) + (w4 + w5);
}

// half sweep of colour `col`, one thread per cell of that colour, any layout
__global__ void k_half_any(Lay L, float h2, Coef32 cf, const float *__restrict__ b, float *xv, int col,
                           int from_zero) {
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, row = t / L.by_half;  // below 2^31
    const int m = (int)(t - row * (unsigned)((L.nx + 1) >> 1));
    const int z = (int)(row / L.by_ny), y = (int)(row - (unsigned)z * L.ny);
    const int x = 2 * m + ((col + y + z) & 1);
    grid_wait();
    if (row >= (unsigned)L.ny * L.nz || x >= L.nx) return;
    float num, den;
    stencil_any(L, cf, xv, x, y, z, num, den);
    if (from_zero) num = 0.f;
    const float hh = cf.s ? 2.f * h2 : h2;
    xv[sto(L, x, y, z)] = __fdividef(hh * b[sto(L, x, y, z)] + num, den);
}

struct Upd {
    double *p;      // natural FP64 solution of the finest level (UPDATE 1)
    float2 *p2;     // natural double-float solution of the finest level (UPDATE 2)
    float alpha;    // scale of the correction, rounded to FP32 on the host
    float shift;    // gauge shift, rounded to FP32 on the host (no FP64 conversion on the device)
};

__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
// double-float (h, l) + t, renormalised (Knuth's TwoSum on the high parts)
__device__ __forceinline__ void df_add(float &h, float &l, float t) {
    float s, e;
    two_sum_f(h, t, s, e);
    e += l;
    h = s + e;
    l = e - (h - s);
}

// pairs of FP32 numbers: one instruction for two cells
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// two cells of a half sweep: (hh b + sum w x) / sum w over the faces x-, x+, y-, y+, z-, z+; SFORM: w = c + a, else w = a
template <bool SFORM, bool FROM_ZERO>
__device__ __forceinline__ void relax2(float hh, f32x2 b, f32x2 c, f32x2 a0, f32x2 a1, f32x2 a2, f32x2 a3, f32x2 a4, f32x2 a5, f32x2 v0,
                                       f32x2 v1, f32x2 v2, f32x2 v3, f32x2 v4, f32x2 v5, float &o0, float &o1) {
    const f32x2 w0 = SFORM ? add2(c, a0) : a0, w1 = SFORM ? add2(c, a1) : a1, w2 = SFORM ? add2(c, a2) : a2;
    const f32x2 w3 = SFORM ? add2(c, a3) : a3, w4 = SFORM ? add2(c, a4) : a4, w5 = SFORM ? add2(c, a5) : a5;
    f32x2 num;
    if (FROM_ZERO) {
        num = mul2(pack2(hh, hh), b);
    } else {
        num = fma2(w0, v0, mul2(w1, v1));
        num = fma2(w2, v2, num);
        num = fma2(w3, v3, num);
        num = fma2(w4, v4, num);
        num = fma2(w5, v5, num);
        num = fma2(pack2(hh, hh), b, num);
    }
    const f32x2 den = add2(add2(add2(w0, w1), add2(w2, w3)), add2(w4, w5));
    float n0, n1, d0, d1;
    unpack2(num, n0, n1);
    unpack2(den, d0, d1);
    o0 = __fdividef(n0, d0);
    o1 = __fdividef(n1, d1);
}

// ---- vectorised half sweep on split levels (hx % 4 == 0) ---------------------------------
// one thread updates 4 consecutive cells (k0..k0+3) of colour col in one row.
// UPDATE (last red half sweep of the finest level): instead of storing the 4 new red values,
// add alpha * x - shift for them and for the 4 black values of the same row positions --
// together the 8 consecutive cells x = 2 k0 .. 2 k0 + 7 -- to the solution: the FP64 one
// (UPDATE 1) or the double-float one (UPDATE 2).
// GHOST: a slab of a decomposed level (L.zlo / L.zhi), its ghost planes as z neighbours
// On levels in L2 the instructions bound it, not the bytes: divisions for the indices, the parity branch of the
// window, selects at walls that few rows have and scalar arithmetic made 224 x 160 x 96 with its adjoint 6.6 ms, not
// 5.6.  Without them it also beats kernels that march planes (face form at 256^3 staged by cp.async, 532 us a V-cycle against
// 522; first sweep from zero, 757 against 754 at 512 x 256 x 256) and, up to 60 M cells, the row-sharing one below.
template <bool SFORM, bool FROM_ZERO, int UPDATE = 0, bool GHOST = false>
__global__ void __launch_bounds__(kThreads, UPDATE == 1 ? 3 : 4) k_half_vec(Lay L, float h2, Coef32 cf, const float *__restrict__ b, float *xv, int col,
                           Upd up = Upd{}) {
    const int hx = L.hx, kv = hx >> 2;
    // black sweeps run from the last plane down: they begin with what the red one left in L2
    const unsigned t = (col ? gridDim.x - 1 - blockIdx.x : blockIdx.x) * blockDim.x + threadIdx.x;
    // thread and row indices stay below 2^31 (at most 2e9 cells)
    const unsigned rowu = t / L.by4;
    // offsets within a level fit 32 bits (a slab's two ghost planes might not)
    using Off = typename std::conditional<GHOST, i64, int>::type;
    const Off row = (Off)rowu;
    const int k0 = (int)(t - rowu * (unsigned)kv) << 2;
    const int z = (int)(rowu / L.by_ny), y = (int)(rowu - (unsigned)z * L.ny);
    grid_wait();
    if (rowu >= (unsigned)L.ny * L.nz) return;
    const int p = (col + y + z) & 1;  // x = 2k + p
    const Off own = (col ? (Off)L.half : 0) + row * hx + k0;
    const Off opp = (col ? 0 : (Off)L.half) + row * hx + k0;
    const bool hy0 = y > 0, hy1 = y < L.ny - 1;
    const bool hz0 = z > 0 || (GHOST && L.zlo), hz1 = z < L.nz - 1 || (GHOST && L.zhi);
    const Off dy = hx, dz = (Off)L.ny * hx;
    const bool edge = p ? k0 + 4 < hx : k0 > 0;  // the window's fifth cell lies in the row
    const Off oe = opp + (p ? 4 : -1);
    const float4 f0 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto ld = [](const float *A, Off off) { return *reinterpret_cast<const float4 *>(A + off); };
    // the other colour's cells left (m) and right (q) of the row's: o shifted by one cell or not, e the fifth.  By
    // selection: the rows of a warp have both parities, and a branch would run both ways
    auto window = [&](const float4 &o, float e, float4 &m, float4 &q) {
        m = make_float4(p ? o.x : e, p ? o.y : o.x, p ? o.z : o.y, p ? o.w : o.z);
        q = make_float4(m.y, m.z, m.w, p ? e : o.w);
    };
    // neighbouring rows, at a wall the row itself: loaded without a branch, put right behind one
    const Off oy0 = hy0 ? opp - dy : opp, oy1 = hy1 ? opp + dy : opp, oz0 = hz0 ? opp - dz : opp, oz1 = hz1 ? opp + dz : opp;
    const bool inner = hy0 && hy1 && hz0 && hz1;
    float4 xm = f0, xp = f0, ym = f0, yp = f0, zm = f0, zp = f0;
    if (!FROM_ZERO) {
        ym = ld(xv, oy0);
        yp = ld(xv, oy1);
        zm = ld(xv, oz0);
        zp = ld(xv, oz1);
        float e = 0.f;
        if (edge) e = xv[oe];
        window(ld(xv, opp), e, xm, xp);
    }
    const float4 bb = ld(b, own);
    float4 w0, w1, w2, w3, w4, w5;  // SFORM: s of the neighbours; a weight is the cell's s plus theirs
    float4 sc = f0;
    if (SFORM) {
        sc = ld(cf.s, own);
        w2 = ld(cf.s, oy0);
        w3 = ld(cf.s, oy1);
        w4 = ld(cf.s, oz0);
        w5 = ld(cf.s, oz1);
        // beyond a wall s = -s of the cell, so that the weight s + s is an exact 0
        float e = p ? -sc.w : -sc.x;
        if (edge) e = cf.s[oe];
        window(ld(cf.s, opp), e, w0, w1);
    } else {
        w0 = ld(cf.fx, own);  // low x face (0 at x = 0)
        float e = 0.f;
        if (edge) e = cf.fx[oe];
        float4 d;
        window(ld(cf.fx, opp), e, d, w1);  // high x face = the x+1 neighbour's low face
        w2 = ld(cf.fy, own);
        w3 = ld(cf.fy, oy1);
        w4 = ld(cf.fz, own);
        w5 = ld(cf.fz, oz1);
    }
    if (!inner) {
        const float4 no = make_float4(-sc.x, -sc.y, -sc.z, -sc.w);  // faces: 0
        if (!hy0) {
            ym = f0;
            if (SFORM) w2 = no;
        }
        if (!hy1) {
            yp = f0;
            w3 = no;
        }
        if (!hz0) {
            zm = f0;
            if (SFORM) w4 = no;
        }
        if (!hz1) {
            zp = f0;
            w5 = no;
        }
    }
    const float hh = SFORM ? 2.f * h2 : h2;
    float out[4];
    auto lo = [](const float4 &q) { return pack2(q.x, q.y); };
    auto hi = [](const float4 &q) { return pack2(q.z, q.w); };
    relax2<SFORM, FROM_ZERO>(hh, lo(bb), lo(sc), lo(w0), lo(w1), lo(w2), lo(w3), lo(w4), lo(w5), lo(xm), lo(xp), lo(ym), lo(yp), lo(zm),
                             lo(zp), out[0], out[1]);
    relax2<SFORM, FROM_ZERO>(hh, hi(bb), hi(sc), hi(w0), hi(w1), hi(w2), hi(w3), hi(w4), hi(w5), hi(xm), hi(xp), hi(ym), hi(yp), hi(zm),
                             hi(zp), out[2], out[3]);
    if (UPDATE == 0) {
        *reinterpret_cast<float4 *>(xv + own) = make_float4(out[0], out[1], out[2], out[3]);
    } else if (UPDATE == 2) {
        const float4 blk = *reinterpret_cast<const float4 *>(xv + opp);
        const float bk[4] = {blk.x, blk.y, blk.z, blk.w};
        const float al = up.alpha, sh = up.shift;
        float2 *pr = up.p2 + (i64)row * L.nx + 2 * k0;
        float4 pvs[4];  // all loads before the first store
#pragma unroll
        for (int v = 0; v < 4; ++v) pvs[v] = *reinterpret_cast<const float4 *>(pr + 2 * v);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            float4 pv = pvs[v];  // (h0, l0, h1, l1)
            const float e0 = p ? bk[v] : out[v], e1 = p ? out[v] : bk[v];
            df_add(pv.x, pv.y, fmaf(al, e0, -sh));
            df_add(pv.z, pv.w, fmaf(al, e1, -sh));
            *reinterpret_cast<float4 *>(pr + 2 * v) = pv;
        }
    } else {
        // red at x = 2k + p, black at x = 2k + 1 - p; same-row black values O[k0..k0+3]
        const float4 blk = *reinterpret_cast<const float4 *>(xv + opp);
        const float bk[4] = {blk.x, blk.y, blk.z, blk.w};
        const float al = up.alpha, sh = up.shift;
        double *pr = up.p + (i64)row * L.nx + 2 * k0;
        double2 pvs[4];  // all loads before the first store
#pragma unroll
        for (int v = 0; v < 4; ++v) pvs[v] = *reinterpret_cast<const double2 *>(pr + 2 * v);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const double2 pv = pvs[v];
            const float e0 = p ? bk[v] : out[v], e1 = p ? out[v] : bk[v];  // cells 2(k0+v) and 2(k0+v)+1
            *reinterpret_cast<double2 *>(pr + 2 * v) =
                make_double2(pv.x + f2d_exact(fmaf(al, e0, -sh)), pv.y + f2d_exact(fmaf(al, e1, -sh)));
        }
    }
}

// ---- row-sharing half sweep -----------------------------------------------------------------
// Row-sharing half sweep for the s-form regular sweep (the finest level's dominant kernel).  A
// block takes a tile of RY rows of W four-cell vectors (RY W = kZrThreads, one vector per
// thread) and marches ZC planes.  The other colour's x and s of the tile's rows and of the rows
// above and below travel by cp.async into a ring of kZrStages planes in shared memory, two planes
// ahead, with the cells' own s and b; every row is fetched once per block and read three times
// (as y - 1, y and y + 1) from there.  A slot is refilled behind the block barrier that ends its plane.
//
// What bounded its predecessor (each thread fetching its own six vectors per plane) was the traffic between L2 and the
// SMs, 36 B per updated cell, and 87 instructions per cell: 215 us per 512^3 half sweep (6.24 TB/s of its 10 B per cell, 0.92 of the copy bandwidth) and, on grids that fit L2, no
// more than 5.3 TB/s.  Sharing rows (28 B at W = 64, RY = 2; 24 B at W = 32, RY = 4), walls folded into
// s (a missing neighbour's s is taken as -s, so that its weight is an exact 0) and packed FP32
// pairs (f32x2) leave it bound by HBM: 194 us by itself, 202 us inside a solve (6.63 TB/s, 0.975 of the copy bandwidth);
// by itself 512 x 512 x 64 38.4 -> 28 us, x 32 19.8 -> 12.7 us.  More rows per block
// (4 of 64 vectors) gave 202 us, one 206 us, three stages 219 us, five 197 us.
//
// Blocks of black sweeps take the planes from above, so that a sweep begins with the planes the one
// before it left in L2 (512 x 512 x 64: 28.4 -> 25.8 us; nothing at 512^3).  Arithmetic as
// k_half_vec: bitwise the same results.
constexpr int kZrThreads = 128, kZrStages = 4, kZrBlocks = 4;  // blocks per SM
constexpr int kZrMaxSmem = 56 * 1024;                            // per block
constexpr i64 kZrCells = 60000000;                               // see run_half_zr
struct ZrTile {
    int w, ry, zc;  // vectors per row, rows and planes of a tile, w ry = kZrThreads
    int pitch;      // row stride in shared memory: whole 128 B lines, as cp.async writes them
    int slot;       // float4 of one plane's slot: ry + 2 rows of x and of s, own s and b, and (rows in
                    // several tiles) the vectors beside the tile's rows
    int used;       // threads with a vector, per mille
};


__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

template <bool GHOST>
__global__ void __launch_bounds__(kZrThreads, kZrBlocks) k_half_zr(Lay L, ZrTile T, float h2, const float *__restrict__ sv,
                                                                   const float *__restrict__ b, float *xv, int col) {
    extern __shared__ float4 ring[];
    grid_wait();
    constexpr int D = kZrStages;
    const int tid = threadIdx.x, lane = tid & 31, hx = L.hx, kv = hx >> 2, pitch = T.pitch;
    const int r = min(tid / T.w, T.ry - 1), v = tid % T.w;  // row and vector in the tile
    const int yb = blockIdx.y * T.ry, vb = blockIdx.x * T.w;
    const bool act = tid < T.ry * T.w && yb + r < L.ny && vb + v < kv;
    const int y = min(yb + r, L.ny - 1), k0 = min(vb + v, kv - 1) << 2;
    const int zb = col ? (int)(gridDim.z - 1 - blockIdx.z) : (int)blockIdx.z;
    const int z0 = zb * T.zc, z1 = min(z0 + T.zc, L.nz);
    const i64 dy = hx, dz = (i64)L.ny * hx;
    const i64 row0 = (i64)y * hx + k0;
    const i64 opp0 = (i64)(1 - col) * L.half + row0, own0 = (i64)col * L.half + row0;
    const bool glo = GHOST && L.zlo, ghi = GHOST && L.zhi;  // a slab's ghost planes are neighbours
    const int zend = L.nz + (ghi ? 1 : 0);                  // planes readable above
    const bool hy0 = y > 0, hy1 = y < L.ny - 1, kl = k0 > 0, kr = k0 + 4 < hx;
    // who fetches the rows and vectors beside the tile
    const bool top = act && r == T.ry - 1 && hy1, bottom = act && r == 0 && hy0;
    const bool left = act && v == 0 && kl, right = act && v == T.w - 1 && kr;
    // whose x - 1 and x + 1 come from a neighbouring lane
    const bool lsh = lane > 0 && v > 0, rsh = lane < 31 && v < T.w - 1;
    const float4 f0 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int nrow = (T.ry + 2) * pitch;  // x rows, then s rows, own s, own b
    float4 *const mine = ring + (r + 1) * pitch + v, *const own = ring + 2 * nrow + tid;
    float4 *const beside = ring + 2 * nrow + 2 * kZrThreads + 4 * r;  // x and s left of the tile's row, right of it
    // plane z into its slot: x and s for plane z1 too, which the last plane reads as z + 1 (what lies
    // beside the grid is not fetched and not read)
    auto issue = [&](int z) {
        if (act && z < zend && z <= z1) {
            float4 *x = mine + (z % D) * T.slot, *s = x + nrow;
            const float *gx = xv + opp0 + (i64)z * dz, *gs = sv + opp0 + (i64)z * dz;
            cp_async16(x, gx);
            cp_async16(s, gs);
            if (z < z1) {
                const i64 w = own0 + (i64)z * dz;
                cp_async16(own + (z % D) * T.slot, sv + w);
                cp_async16(own + (z % D) * T.slot + kZrThreads, b + w);
                if (bottom) {
                    cp_async16(x - pitch, gx - dy);
                    cp_async16(s - pitch, gs - dy);
                }
                if (top) {
                    cp_async16(x + pitch, gx + dy);
                    cp_async16(s + pitch, gs + dy);
                }
                if (left) {
                    cp_async16(beside + (z % D) * T.slot, gx - 4);
                    cp_async16(beside + (z % D) * T.slot + 1, gs - 4);
                }
                if (right) {
                    cp_async16(beside + (z % D) * T.slot + 2, gx + 4);
                    cp_async16(beside + (z % D) * T.slot + 3, gs + 4);
                }
            }
        }
        cp_async_commit();  // one group per plane, empty past the chunk: the counting stays uniform
    };
#pragma unroll
    for (int q = 0; q < D - 1; ++q) issue(z0 + q);
    auto ld = [](const float *A, i64 off) { return *reinterpret_cast<const float4 *>(A + off); };
    const bool below = z0 > 0 || glo;
    float4 xzm = below ? ld(xv, opp0 + (i64)(z0 - 1) * dz) : f0, szm = below ? ld(sv, opp0 + (i64)(z0 - 1) * dz) : f0;
    float4 xzc = f0, szc = f0;
    const float hh = 2.f * h2;
    for (int z = z0; z < z1; ++z) {
        cp_async_wait<D - 3>();  // planes z and z + 1 have landed
        __syncthreads();         // for every thread, and plane z - 1 has been read by all
        issue(z + D - 1);        // into the slot of plane z - 1
        const float4 *x = mine + (z % D) * T.slot, *s = x + nrow;
        const float4 *xn = mine + ((z + 1) % D) * T.slot, *sn = xn + nrow;
        if (z == z0) {
            xzc = *x;
            szc = *s;
        }
        float4 xzp = f0, szp = f0, ym = f0, yp = f0;
        const float4 sc = own[(z % D) * T.slot], bv = own[(z % D) * T.slot + kZrThreads];
        // beyond a wall x = 0 and s = -s of the cell, so that the weight s + s is an exact 0
        const float4 ns = make_float4(-sc.x, -sc.y, -sc.z, -sc.w);
        float4 s2 = ns, s3 = ns, s4 = szm, s5 = ns;
        if (z + 1 < zend) {
            xzp = *xn;
            szp = s5 = *sn;
        }
        if (hy0) {
            ym = x[-pitch];
            s2 = s[-pitch];
        }
        if (hy1) {
            yp = x[pitch];
            s3 = s[pitch];
        }
        if (z == 0 && !glo) s4 = ns;
        // x - 1 and x + 1: the own vector shifted by one cell or not (x = 2k + p)
        float4 xm = xzc, xp = xzc, sm = szc, sp = szc;
        const bool p = (col + y + z) & 1;
        // lanes of one warp may hold rows of both parities: both shuffles
        float xr = __shfl_down_sync(0xffffffffu, xzc.x, 1), sr = __shfl_down_sync(0xffffffffu, szc.x, 1);
        float xl = __shfl_up_sync(0xffffffffu, xzc.w, 1), sl = __shfl_up_sync(0xffffffffu, szc.w, 1);
        if (p) {
            if (!rsh && kr) {
                const float4 *e = beside + (z % D) * T.slot + 2;
                xr = v == T.w - 1 ? e[0].x : x[1].x;
                sr = v == T.w - 1 ? e[1].x : s[1].x;
            }
            if (!kr) {
                xr = 0.f;
                sr = ns.w;
            }
            xp = make_float4(xzc.y, xzc.z, xzc.w, xr);
            sp = make_float4(szc.y, szc.z, szc.w, sr);
        } else {
            if (!lsh && kl) {
                const float4 *e = beside + (z % D) * T.slot;
                xl = v == 0 ? e[0].w : x[-1].w;
                sl = v == 0 ? e[1].w : s[-1].w;
            }
            if (!kl) {
                xl = 0.f;
                sl = ns.x;
            }
            xm = make_float4(xl, xzc.x, xzc.y, xzc.z);
            sm = make_float4(sl, szc.x, szc.y, szc.z);
        }
        float4 out;
        auto lo = [](const float4 &q) { return pack2(q.x, q.y); };
        auto up = [](const float4 &q) { return pack2(q.z, q.w); };
        relax2<true, false>(hh, lo(bv), lo(sc), lo(sm), lo(sp), lo(s2), lo(s3), lo(s4), lo(s5), lo(xm), lo(xp), lo(ym), lo(yp), lo(xzm), lo(xzp),
             out.x, out.y);
        relax2<true, false>(hh, up(bv), up(sc), up(sm), up(sp), up(s2), up(s3), up(s4), up(s5), up(xm), up(xp), up(ym), up(yp), up(xzm), up(xzp),
             out.z, out.w);
        if (act) *reinterpret_cast<float4 *>(xv + own0 + (i64)z * dz) = out;
        xzm = xzc;
        xzc = xzp;
        szm = szc;
        szc = szp;
    }
    cp_async_wait<0>();  // only copies that nothing reads can remain; leave none behind
}

// Tiles of k_half_zr: rows of 64, 32 or 16 vectors (or whole rows of 8), whole 128 B lines each, the widest of those that
// leave the fewest threads beyond the end of a row.
ZrTile zr_tile(const Lay &L) {
    ZrTile T;
    const int kv = L.hx / 4;
    T.w = T.used = 0;
    for (int w = 64; w >= 8; w /= 2) {
        if (w > kv || (w == 8 && kv != 8)) continue;
        const int n = (kv + w - 1) / w, used = 1000 * kv / (n * w);
        if (used > T.used) {
            T.used = used;
            T.w = w;
        }
    }
    if (!T.w) return T;
    T.ry = kZrThreads / T.w;
    T.zc = 16;
    T.pitch = T.w;
    T.slot = 2 * (T.ry + 2) * T.w + 2 * kZrThreads + (kv > T.w ? 4 * T.ry : 0);
    return T;
}

// Whether the s-form regular sweep of L goes to k_half_zr (and its launch): tiles that leave at most a tenth of the threads
// idle, on levels of 60 M cells and more, where it is the one that HBM alone bounds.  (A whole grid of that size has sides
// that are multiples of 64, or its coarsest level would be too large; only a slab's last planes can be part of a tile.)
// V-cycles with it and with k_half_vec: 512^3 2883 against 2965 us, 512 x 512 x 256 1474 against 1508, 256 x 512 x 512
// 1462 against 1496, 1024 x 256 x 256 1485 against 1518;
// 512 x 384 x 256 1136 against 1129, 256^3 411 against 404, 192^3 230 against 193; tiles with more idle threads 448^3 2058 against
// 2005, 576 x 512 x 448 2983 against 2935.
template <bool GHOST>
bool run_half_zr(cudaStream_t s, const Lay &L, float h2, const float *sv, const float *b, float *x, int col) {
    const int kv = L.hx / 4;
    if (L.n < kZrCells) return false;
    const ZrTile T = zr_tile(L);
    if (T.used <= 900) return false;
    static std::atomic<unsigned long long> opted{0};
    if (!opt_in_smem((const void *)k_half_zr<GHOST>, kZrMaxSmem, opted)) return true;  // the caller checks the error
    run_kernel(k_half_zr<GHOST>, dim3((kv + T.w - 1) / T.w, (L.ny + T.ry - 1) / T.ry, (L.nz + T.zc - 1) / T.zc), kZrThreads,
               (size_t)kZrStages * T.slot * sizeof(float4), s, L, T, h2, sv, b, x, col);
    return true;
}

// ---- vectorised red-only residual + restriction (split fine level, hx % 4 == 0) ----------
// The red children of coarse cell (I, J, K) are the red cells at k = I of the 4 fine rows
// (2J + b, 2K + c); one thread handles coarse cells I0..I0+3 of one coarse row.
constexpr int kRrThreads = 64;

// GHOST: the fine level is a slab (L.zlo / L.zhi) and Lc a view of the whole coarse level
// (its arrays at the slab's first coarse plane, an even one)
template <bool SFORM, bool GHOST = false>
__global__ void __launch_bounds__(kRrThreads, 12) k_rr_red_vec(Lay L, Lay Lc, float ih2, Coef32 cf, const float *__restrict__ b,
                             const float *__restrict__ xv, float *bc) {
    grid_wait();
    const int hx = L.hx, kv = hx >> 2;
    const i64 T = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    const i64 crows = (i64)Lc.ny * Lc.nz;
    if (T >= crows * kv) return;
    // thread and row indices stay below 2^31 (at most 2e9 cells): 32-bit divisions, several
    // times cheaper than 64-bit ones
    const unsigned Tu = (unsigned)T, crowu = Tu / L.by4;
    const int k0 = (int)(Tu - crowu * (unsigned)kv) << 2;
    const int K = (int)(crowu / Lc.by_ny), J = (int)(crowu - (unsigned)K * Lc.ny);
    using Off = typename std::conditional<GHOST, i64, int>::type;  // as in k_half_vec
    const Off dy = hx, dz = (Off)L.ny * hx;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
        const int y = 2 * J + (ch & 1), z = 2 * K + (ch >> 1);
        const int p = (ch & 1) ^ (ch >> 1);  // red cells of this row sit at x = 2k + p
        const Off row = (Off)z * L.ny + y;
        const Off own = row * hx + k0;                // red half
        const Off opp = (Off)L.half + row * hx + k0;  // black half
        // half of the neighbours are siblings
        const bool hy0 = (ch & 1) || y > 0, hy1 = !(ch & 1) || y < L.ny - 1;
        const bool hz0 = (ch >> 1) || z > 0 || (GHOST && L.zlo), hz1 = !(ch >> 1) || z < L.nz - 1 || (GHOST && L.zhi);
        const bool xw0 = (p == 0 && k0 == 0), xw1 = (p == 1 && k0 + 4 == hx);
        auto window = [&](const float *O, float (&m)[4], float (&q)[4]) {
            const float4 c4 = *reinterpret_cast<const float4 *>(O + opp);
            if (p) {
                const float e = (k0 + 4 < hx) ? O[opp + 4] : 0.f;
                m[0] = c4.x; m[1] = c4.y; m[2] = c4.z; m[3] = c4.w;
                q[0] = c4.y; q[1] = c4.z; q[2] = c4.w; q[3] = e;
            } else {
                const float e = (k0 > 0) ? O[opp - 1] : 0.f;
                m[0] = e; m[1] = c4.x; m[2] = c4.y; m[3] = c4.z;
                q[0] = c4.x; q[1] = c4.y; q[2] = c4.z; q[3] = c4.w;
            }
        };
        auto ld4 = [&](const float *A, Off off, bool ok, float (&v)[4]) {
            if (ok) {
                const float4 c4 = *reinterpret_cast<const float4 *>(A + off);
                v[0] = c4.x; v[1] = c4.y; v[2] = c4.z; v[3] = c4.w;
            } else {
                v[0] = v[1] = v[2] = v[3] = 0.f;
            }
        };
        float xc[4], xm[4], xp[4], ym[4], yp[4], zm[4], zp[4], bb[4];
        ld4(xv, own, true, xc);
        window(xv, xm, xp);
        ld4(xv, opp - dy, hy0, ym);
        ld4(xv, opp + dy, hy1, yp);
        ld4(xv, opp - dz, hz0, zm);
        ld4(xv, opp + dz, hz1, zp);
        ld4(b, own, true, bb);
        float w0[4], w1[4], w2[4], w3[4], w4[4], w5[4];
        if (SFORM) {
            float sc[4], sm_[4], sp_[4], s2[4], s3[4], s4[4], s5[4];
            ld4(cf.s, own, true, sc);
            window(cf.s, sm_, sp_);
            ld4(cf.s, opp - dy, hy0, s2);
            ld4(cf.s, opp + dy, hy1, s3);
            ld4(cf.s, opp - dz, hz0, s4);
            ld4(cf.s, opp + dz, hz1, s5);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                w0[v] = (v == 0 && xw0) ? 0.f : 0.5f * (sc[v] + sm_[v]);
                w1[v] = (v == 3 && xw1) ? 0.f : 0.5f * (sc[v] + sp_[v]);
                w2[v] = hy0 ? 0.5f * (sc[v] + s2[v]) : 0.f;
                w3[v] = hy1 ? 0.5f * (sc[v] + s3[v]) : 0.f;
                w4[v] = hz0 ? 0.5f * (sc[v] + s4[v]) : 0.f;
                w5[v] = hz1 ? 0.5f * (sc[v] + s5[v]) : 0.f;
            }
        } else {
            float d0[4];
            ld4(cf.fx, own, true, w0);
            window(cf.fx, d0, w1);
            if (xw1) w1[3] = 0.f;
            ld4(cf.fy, own, true, w2);
            ld4(cf.fy, opp + dy, hy1, w3);
            ld4(cf.fz, own, true, w4);
            ld4(cf.fz, opp + dz, hz1, w5);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            float ax = w0[v] * (xc[v] - xm[v]);
            ax += w1[v] * (xc[v] - xp[v]);
            ax += w2[v] * (xc[v] - ym[v]);
            ax += w3[v] * (xc[v] - yp[v]);
            ax += w4[v] * (xc[v] - zm[v]);
            ax += w5[v] * (xc[v] - zp[v]);
            acc[v] += bb[v] - ax * ih2;
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) bc[sto(Lc, k0 + v, J, K)] = acc[v] * 0.125f;
}

// The same with one fine row per thread: lanes v, v + 8, v + 16, v + 24 of a warp take the four fine rows of
// the same four coarse cells, and the first adds the four residuals up in their order.  Levels of up to
// kRrRowCells cells have too few coarse cells to fill the device with k_rr_red_vec, whose threads then
// wait for four rounds of loads: 64^3 2.8 -> 2.1 us (s-form) and 3.2 -> 2.0 us (faces), 96^3 3.4 -> 3.1 and 3.6 -> 2.9;
// 128^3 4.5 against 6.0 us and 512^3 238 against 425 us, where it loads more lines than it uses.
// TAIL: the coarse levels' cluster launch follows, which may come in and copy its contexts meanwhile.
constexpr i64 kRrRowCells = 1000000;
constexpr int kRrRowThreads = 128;
template <bool SFORM, bool TAIL>
__global__ void __launch_bounds__(kRrRowThreads, 6) k_rr_red_row(Lay L, Lay Lc, float ih2, Coef32 cf, const float *__restrict__ b,
                                                                 const float *__restrict__ xv, float *bc) {
    const int hx = L.hx, kv = hx >> 2;
    const unsigned T = blockIdx.x * blockDim.x + threadIdx.x, lane = T & 31, total = (unsigned)Lc.ny * Lc.nz * kv;
    const unsigned vi = (T >> 5) * 8 + (lane & 7), vc = min(vi, total - 1);  // 4-cell vector of the coarse level
    const int ch = lane >> 3;
    const unsigned crow = vc / L.by4;
    const int k0 = (int)(vc - crow * (unsigned)kv) << 2;
    const int K = (int)(crow / Lc.by_ny), J = (int)(crow - (unsigned)K * Lc.ny);
    const int dy = hx, dz = L.ny * hx;
    grid_wait();
    if (TAIL) trigger_next();
    const int y = 2 * J + (ch & 1), z = 2 * K + (ch >> 1);
    const int p = (y + z) & 1;  // red cells of this row sit at x = 2k + p
    const int row = z * L.ny + y;
    const int own = row * hx + k0, opp = (int)L.half + own;
    const bool hy0 = y > 0, hy1 = y < L.ny - 1, hz0 = z > 0, hz1 = z < L.nz - 1;
    const bool xw0 = (p == 0 && k0 == 0), xw1 = (p == 1 && k0 + 4 == hx);
    const bool edge = p ? k0 + 4 < hx : k0 > 0;  // the window's fifth cell lies in the row
    const int eo = p ? 4 : -1;
    auto window = [&](const float *O, float (&m)[4], float (&q)[4]) {
        const float4 c4 = *reinterpret_cast<const float4 *>(O + opp);
        const float e = edge ? O[opp + eo] : 0.f;
        m[0] = p ? c4.x : e; m[1] = p ? c4.y : c4.x; m[2] = p ? c4.z : c4.y; m[3] = p ? c4.w : c4.z;
        q[0] = m[1]; q[1] = m[2]; q[2] = m[3]; q[3] = p ? e : c4.w;
    };
    auto ld4 = [&](const float *A, int off, bool ok, float (&v)[4]) {
        if (ok) {
            const float4 c4 = *reinterpret_cast<const float4 *>(A + off);
            v[0] = c4.x; v[1] = c4.y; v[2] = c4.z; v[3] = c4.w;
        } else {
            v[0] = v[1] = v[2] = v[3] = 0.f;
        }
    };
    float xc[4], xm[4], xp[4], ym[4], yp[4], zm[4], zp[4], bb[4];
    ld4(xv, own, true, xc);
    window(xv, xm, xp);
    ld4(xv, opp - dy, hy0, ym);
    ld4(xv, opp + dy, hy1, yp);
    ld4(xv, opp - dz, hz0, zm);
    ld4(xv, opp + dz, hz1, zp);
    ld4(b, own, true, bb);
    float w0[4], w1[4], w2[4], w3[4], w4[4], w5[4];
    if (SFORM) {
        float sc[4], sm_[4], sp_[4], s2[4], s3[4], s4[4], s5[4];
        ld4(cf.s, own, true, sc);
        window(cf.s, sm_, sp_);
        ld4(cf.s, opp - dy, hy0, s2);
        ld4(cf.s, opp + dy, hy1, s3);
        ld4(cf.s, opp - dz, hz0, s4);
        ld4(cf.s, opp + dz, hz1, s5);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            w0[v] = (v == 0 && xw0) ? 0.f : 0.5f * (sc[v] + sm_[v]);
            w1[v] = (v == 3 && xw1) ? 0.f : 0.5f * (sc[v] + sp_[v]);
            w2[v] = hy0 ? 0.5f * (sc[v] + s2[v]) : 0.f;
            w3[v] = hy1 ? 0.5f * (sc[v] + s3[v]) : 0.f;
            w4[v] = hz0 ? 0.5f * (sc[v] + s4[v]) : 0.f;
            w5[v] = hz1 ? 0.5f * (sc[v] + s5[v]) : 0.f;
        }
    } else {
        float d0[4];
        ld4(cf.fx, own, true, w0);
        window(cf.fx, d0, w1);
        if (xw1) w1[3] = 0.f;
        ld4(cf.fy, own, true, w2);
        ld4(cf.fy, opp + dy, hy1, w3);
        ld4(cf.fz, own, true, w4);
        ld4(cf.fz, opp + dz, hz1, w5);
    }
    float acc[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        // the sum of products in the order k_rr_red_vec forms it
        float ax = fmaf(w0[v], xc[v] - xm[v], w1[v] * (xc[v] - xp[v]));
        ax = fmaf(w2[v], xc[v] - ym[v], ax);
        ax = fmaf(w3[v], xc[v] - yp[v], ax);
        ax = fmaf(w4[v], xc[v] - zm[v], ax);
        ax = fmaf(w5[v], xc[v] - zp[v], ax);
        const float r = fmaf(-ax, ih2, bb[v]);
        const float r1 = __shfl_down_sync(0xffffffffu, r, 8), r2 = __shfl_down_sync(0xffffffffu, r, 16);
        const float r3 = __shfl_down_sync(0xffffffffu, r, 24);
        acc[v] = ((r + r1) + r2) + r3;
    }
    if (vi >= total || ch) return;
#pragma unroll
    for (int v = 0; v < 4; ++v) bc[sto(Lc, k0 + v, J, K)] = acc[v] * 0.125f;
}

// ---- vectorised red-only prolongation + correction (split fine level, hx % 4 == 0) -------
// one thread adds P ec to 4 consecutive red cells of one fine row
__global__ void k_prolong_red_vec(Lay L, Lay Lc, const float *__restrict__ ec, float *xv, int kind) {
    grid_wait();
    const int hx = L.hx, kv = hx >> 2;
    const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    const i64 rows = (i64)L.ny * L.nz;
    if (t >= rows * kv) return;
    // thread and row indices stay below 2^31 (at most 2e9 cells): 32-bit divisions, several
    // times cheaper than 64-bit ones
    const unsigned tu = (unsigned)t, rowu = tu / L.by4;
    const i64 row = rowu;
    const int k0 = (int)(tu - rowu * (unsigned)kv) << 2;
    const int z = (int)(rowu / L.by_ny), y = (int)(rowu - (unsigned)z * L.ny);
    const int p = (y + z) & 1;  // red x = 2k + p, coarse I = k
    const int J = y >> 1, K = z >> 1;
    float out[4];
    float4 x4 = *reinterpret_cast<const float4 *>(xv + row * hx + k0);
    out[0] = x4.x; out[1] = x4.y; out[2] = x4.z; out[3] = x4.w;
    if (kind == MG_PROLONG_CONSTANT) {
#pragma unroll
        for (int v = 0; v < 4; ++v) out[v] += __ldg(ec + sto(Lc, k0 + v, J, K));
    } else {
        int J2 = (y & 1) ? J + 1 : J - 1;
        int K2 = (z & 1) ? K + 1 : K - 1;
        if (J2 < 0 || J2 >= Lc.ny) J2 = J;
        if (K2 < 0 || K2 >= Lc.nz) K2 = K;
        // coarse values at I = k0 - 1 .. k0 + 4 of the four coarse rows
        float c[4][6];
        const int Js[2] = {J, J2}, Ks[2] = {K, K2};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int JJ = Js[r & 1], KK = Ks[r >> 1];
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                int I = k0 - 1 + u;
                if (I < 0) I = 0;
                if (I >= Lc.nx) I = Lc.nx - 1;
                c[r][u] = __ldg(ec + sto(Lc, I, JJ, KK));
            }
        }
        const float w0 = 0.75f, w1 = 0.25f;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int I = k0 + v;
            int I2 = p ? I + 1 : I - 1;
            if (I2 < 0 || I2 >= Lc.nx) I2 = I;
            const int u1 = I + 1 - k0, u2 = I2 + 1 - k0;  // positions in c[][]
            float a = w0 * w0 * w0 * c[0][u1];
            a += w1 * w0 * w0 * c[0][u2];
            a += w0 * w1 * w0 * c[1][u1];
            a += w1 * w1 * w0 * c[1][u2];
            a += w0 * w0 * w1 * c[2][u1];
            a += w1 * w0 * w1 * c[2][u2];
            a += w0 * w1 * w1 * c[3][u1];
            a += w1 * w1 * w1 * c[3][u2];
            out[v] += a;
        }
    }
    *reinterpret_cast<float4 *>(xv + row * hx + k0) = make_float4(out[0], out[1], out[2], out[3]);
}

// ---- separable red-only trilinear prolongation (split fine level, coarse nx % 8 == 0) -----
// One thread takes coarse row (J, K) and I0 = k0 .. k0+7: the 8 red cells k0 .. k0+7 of each of
// the 4 fine rows y = 2J + d, z = 2K + e.  Fine row (d, e) interpolates in y and z first,
//   R_de(I) = 9/16 c(J, K) + 3/16 c(J_d, K) + 3/16 c(J, K_e) + 1/16 c(J_d, K_e)
// with J_d = J - 1 + 2d and K_e = K - 1 + 2e clamped into the grid (the wall mirror), then in x:
// the red cell at k (x = 2k + p, coarse I = k) gains 3/4 R(I) + 1/4 R(I + 2p - 1), clamped.
// Each coarse row supplies I = k0 - 1 .. k0 + 8: two float4 (even and odd I, one per colour
// half) and two scalars.
constexpr int kProlThreads = 64;

// GHOST: the fine level is a slab and Lc a view of the whole coarse level from the slab's first
// coarse plane (Lc.zlo / Lc.zhi: the coarse planes next to the view are the neighbours', read
// where the whole grid would read them instead of the wall's mirror)
template <bool GHOST = false>
__global__ void __launch_bounds__(kProlThreads, 10) k_prolong_red8(Lay L, Lay Lc, const float *__restrict__ ec, float *xv) {
    grid_wait();
    const int hx = L.hx, kv = hx >> 3;  // 8-cell groups per fine row
    const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    const i64 crows = (i64)Lc.ny * Lc.nz;
    if (t >= crows * kv) return;
    // thread and row indices stay below 2^31 (at most 2e9 cells): 32-bit divisions, several
    // times cheaper than 64-bit ones
    const unsigned tu = (unsigned)t, crowu = 2 * tu / L.by4;
    const int k0 = (int)(tu - crowu * (unsigned)kv) << 3;
    const int K = (int)(crowu / Lc.by_ny), J = (int)(crowu - (unsigned)K * Lc.ny);
    const int hxc = Lc.hx, ncx = Lc.nx;
    const int Js[3] = {max(J - 1, 0), J, min(J + 1, Lc.ny - 1)};
    const int Ks[3] = {(GHOST && Lc.zlo) ? K - 1 : max(K - 1, 0), K, (GHOST && Lc.zhi) ? K + 1 : min(K + 1, Lc.nz - 1)};
    float R[4][10];  // [2e + d][I - k0 + 1]
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int u = 0; u < 10; ++u) R[r][u] = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {      // coarse row J - 1 + a
#pragma unroll
        for (int c = 0; c < 3; ++c) {  // coarse row K - 1 + c
            const int JJ = Js[a], KK = Ks[c];
            const int q = (JJ + KK) & 1;  // colour of coarse I even
            const i64 rowc = (i64)KK * Lc.ny + JJ;
            const float *ev = ec + (i64)q * Lc.half + rowc * hxc;        // even I, position I / 2
            const float *od = ec + (i64)(1 - q) * Lc.half + rowc * hxc;  // odd I
            const float4 e4 = *reinterpret_cast<const float4 *>(ev + (k0 >> 1));
            const float4 o4 = *reinterpret_cast<const float4 *>(od + (k0 >> 1));
            float v[10];
            v[1] = e4.x; v[2] = o4.x; v[3] = e4.y; v[4] = o4.y;
            v[5] = e4.z; v[6] = o4.z; v[7] = e4.w; v[8] = o4.w;
            v[0] = k0 > 0 ? od[(k0 >> 1) - 1] : v[1];          // I = k0 - 1, mirrored at the wall
            v[9] = k0 + 8 < ncx ? ev[(k0 >> 1) + 4] : v[8];    // I = k0 + 8
            // weight of this coarse row in fine row (d, e): y factor (3/4 own, 1/4 neighbour)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    // fine row (d, e) uses coarse rows J and J_d = J - 1 + 2d, K and K_e = K - 1 + 2e
                    const bool ya = (a == 1) || (a == 2 * d);
                    const bool za = (c == 1) || (c == 2 * e);
                    if (!ya || !za) continue;
                    // when J_d was clamped onto J the two y weights land on the same row
                    float wy = (a == 1) ? 0.75f : 0.25f;
                    float wz = (c == 1) ? 0.75f : 0.25f;
                    const float w = wy * wz;
#pragma unroll
                    for (int u = 0; u < 10; ++u) R[2 * e + d][u] = fmaf(w, v[u], R[2 * e + d][u]);
                }
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const int y = 2 * J + d, z = 2 * K + e;
            if (y >= L.ny || z >= L.nz) continue;
            const int p = (d + e) & 1;  // red x = 2k + p
            float *xr = xv + ((i64)z * L.ny + y) * hx + k0;
            float4 a4 = *reinterpret_cast<const float4 *>(xr);
            float4 b4 = *reinterpret_cast<const float4 *>(xr + 4);
            float o[8] = {a4.x, a4.y, a4.z, a4.w, b4.x, b4.y, b4.z, b4.w};
            const float *Rr = R[2 * e + d];
#pragma unroll
            for (int v = 0; v < 8; ++v) o[v] += 0.75f * Rr[v + 1] + 0.25f * (p ? Rr[v + 2] : Rr[v]);
            *reinterpret_cast<float4 *>(xr) = make_float4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<float4 *>(xr + 4) = make_float4(o[4], o[5], o[6], o[7]);
        }
    }
}

// The same with one fine row per thread (four coarse rows each, the sums in the same order): four times the
// threads on levels of up to kProlRowCells cells, 64^3 2.6 -> 1.6 us, 96^3 3.4 -> 2.2, 192^3 7.9 -> 7.2; 256^3 12.2 against
// 14.3 us, where the coarse rows read again cost more.
constexpr i64 kProlRowCells = 8000000;
constexpr int kProlRowThreads = 128;
__global__ void __launch_bounds__(kProlRowThreads, 8) k_prolong_red_row(Lay L, Lay Lc, const float *__restrict__ ec, float *xv) {
    const int hx = L.hx, kv = hx >> 3;  // 8-cell groups per fine row
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, row = 2 * t / L.by4;
    const int k0 = (int)(t - row * (unsigned)kv) << 3;
    const int z = (int)(row / L.by_ny), y = (int)(row - (unsigned)z * L.ny);
    grid_wait();
    if (row >= (unsigned)L.ny * L.nz) return;
    const int d = y & 1, e = z & 1, J = y >> 1, K = z >> 1, hxc = Lc.hx;
    const int J2 = d ? min(J + 1, Lc.ny - 1) : max(J - 1, 0), K2 = e ? min(K + 1, Lc.nz - 1) : max(K - 1, 0);
    float *xr = xv + (i64)row * hx + k0;
    const float4 a4 = *reinterpret_cast<const float4 *>(xr), b4 = *reinterpret_cast<const float4 *>(xr + 4);
    float R[10];
#pragma unroll
    for (int u = 0; u < 10; ++u) R[u] = 0.f;
    // coarse rows in the order J - 1, J, J + 1 and, in each, K - 1, K, K + 1
#pragma unroll
    for (int ja = 0; ja < 2; ++ja) {
#pragma unroll
        for (int ka = 0; ka < 2; ++ka) {
            const bool jn = ja == d, kn = ka == e;  // the neighbour row comes first for d = 0, last for d = 1
            const int JJ = jn ? J2 : J, KK = kn ? K2 : K, q = (JJ + KK) & 1;
            const i64 rowc = (i64)KK * Lc.ny + JJ;
            const float *ev = ec + (i64)q * Lc.half + rowc * hxc;        // even I, position I / 2
            const float *od = ec + (i64)(1 - q) * Lc.half + rowc * hxc;  // odd I
            const float4 e4 = *reinterpret_cast<const float4 *>(ev + (k0 >> 1));
            const float4 o4 = *reinterpret_cast<const float4 *>(od + (k0 >> 1));
            float v[10];
            v[1] = e4.x; v[2] = o4.x; v[3] = e4.y; v[4] = o4.y;
            v[5] = e4.z; v[6] = o4.z; v[7] = e4.w; v[8] = o4.w;
            v[0] = k0 > 0 ? od[(k0 >> 1) - 1] : v[1];
            v[9] = k0 + 8 < Lc.nx ? ev[(k0 >> 1) + 4] : v[8];
            const float w = (jn ? 0.25f : 0.75f) * (kn ? 0.25f : 0.75f);
#pragma unroll
            for (int u = 0; u < 10; ++u) R[u] = fmaf(w, v[u], R[u]);
        }
    }
    const int p = (d + e) & 1;  // red x = 2k + p
    float o[8] = {a4.x, a4.y, a4.z, a4.w, b4.x, b4.y, b4.z, b4.w};
#pragma unroll
    for (int v = 0; v < 8; ++v) o[v] += fmaf(0.75f, R[v + 1], 0.25f * (p ? R[v + 2] : R[v]));
    *reinterpret_cast<float4 *>(xr) = make_float4(o[0], o[1], o[2], o[3]);
    *reinterpret_cast<float4 *>(xr + 4) = make_float4(o[4], o[5], o[6], o[7]);
}

// ---- residual (generic) ------------------------------------------------------------------
// r(x, y, z) = b - A x   (FP32, any layout)
__device__ __forceinline__ float resid_any(const Lay &L, float ih2, const Coef32 &cf, const float *__restrict__ b,
                                           const float *__restrict__ xv, int x, int y, int z) {
    float num, den;
    stencil_any(L, cf, xv, x, y, z, num, den);
    const i64 c = sto(L, x, y, z);
    const float ax = xv[c] * den - num;
    return b[c] - (cf.s ? 0.5f : 1.f) * ax * ih2;
}

__global__ void k_residual_any(Lay L, float ih2, Coef32 cf, const float *__restrict__ b,
                               const float *__restrict__ xv, float *r, int apply_only) {
    grid_wait();
    const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= L.n) return;
    const int x = (int)(t % L.nx);
    const i64 row = t / L.nx;
    const int y = (int)(row % L.ny), z = (int)(row / L.ny);
    const i64 c = sto(L, x, y, z);
    if (apply_only) {
        float num, den;
        stencil_any(L, cf, xv, x, y, z, num, den);
        r[c] = (cf.s ? 0.5f : 1.f) * (xv[c] * den - num) * ih2;
    } else {
        r[c] = resid_any(L, ih2, cf, b, xv, x, y, z);
    }
}

// coarse b = mean of the children's residuals; red_only: black children contribute 0
// (exact after a black half sweep, which solves every black row)
__global__ void k_resid_restrict_any(Lay L, Lay Lc, float ih2, Coef32 cf, const float *__restrict__ b,
                                     const float *__restrict__ xv, float *bc, int red_only) {
    const unsigned T = blockIdx.x * blockDim.x + threadIdx.x, row = T / Lc.by_nx;
    const int I = (int)(T - row * (unsigned)Lc.nx), K = (int)(row / Lc.by_ny), J = (int)(row - (unsigned)K * Lc.ny);
    grid_wait();
    if (T >= Lc.n) return;
    float s = 0.f;
#pragma unroll
    for (int cc = 0; cc < 2; ++cc)
#pragma unroll
        for (int bb = 0; bb < 2; ++bb)
#pragma unroll
            for (int aa = 0; aa < 2; ++aa) {
                const int x = 2 * I + aa, y = 2 * J + bb, z = 2 * K + cc;
                if (red_only && ((x + y + z) & 1)) continue;
                s += resid_any(L, ih2, cf, b, xv, x, y, z);
            }
    bc[sto(Lc, I, J, K)] = s * 0.125f;
}

// x += P ec on cells of colour `only_col` (0 red, 1 black) or on all cells (-1)
__global__ void k_prolong_any(Lay L, Lay Lc, const float *__restrict__ ec, float *xv, int kind, int only_col) {
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, row = t / L.by_nx;
    const int x = (int)(t - row * (unsigned)L.nx), z = (int)(row / L.by_ny), y = (int)(row - (unsigned)z * L.ny);
    grid_wait();
    if (t >= L.n) return;
    if (only_col >= 0 && ((x + y + z) & 1) != only_col) return;
    const int I = x >> 1, J = y >> 1, K = z >> 1;
    float v;
    if (kind == MG_PROLONG_CONSTANT) {
        v = ec[sto(Lc, I, J, K)];
    } else {
        int I2 = (x & 1) ? I + 1 : I - 1;
        int J2 = (y & 1) ? J + 1 : J - 1;
        int K2 = (z & 1) ? K + 1 : K - 1;
        if (I2 < 0 || I2 >= Lc.nx) I2 = I;
        if (J2 < 0 || J2 >= Lc.ny) J2 = J;
        if (K2 < 0 || K2 >= Lc.nz) K2 = K;
        const float w0 = 0.75f, w1 = 0.25f;
        v = w0 * w0 * w0 * ec[sto(Lc, I, J, K)];
        v += w1 * w0 * w0 * ec[sto(Lc, I2, J, K)];
        v += w0 * w1 * w0 * ec[sto(Lc, I, J2, K)];
        v += w1 * w1 * w0 * ec[sto(Lc, I2, J2, K)];
        v += w0 * w0 * w1 * ec[sto(Lc, I, J, K2)];
        v += w1 * w0 * w1 * ec[sto(Lc, I2, J, K2)];
        v += w0 * w1 * w1 * ec[sto(Lc, I, J2, K2)];
        v += w1 * w1 * w1 * ec[sto(Lc, I2, J2, K2)];
    }
    xv[sto(L, x, y, z)] += v;
}

// e = pinv r on the coarsest level (FP64 accumulation), pinv in natural cell order; a warp takes a row.  r is
// brought into cell order and FP64 once per block: converted and looked up per product, 990 cells took 18.7 us
// (two FP64 operations and two integer divisions each), now 9 us less, of which the FMAs of eight rows per SM take 2.
__global__ void __launch_bounds__(kThreads) k_coarse_matvec_lay(Lay L, const double *__restrict__ pinv, const float *__restrict__ r,
                                                               float *e) {
    grid_wait();
    __shared__ double rs[MG_MAX_COARSE];
    const int nc = (int)L.n;
    auto place = [&](int q) {
        const int row = q / L.nx, z = row / L.ny;
        return sto(L, q - row * L.nx, row - z * L.ny, z);
    };
    for (int q = threadIdx.x; q < nc; q += kThreads) rs[q] = (double)r[place(q)];
    __syncthreads();
    const int row = (int)(((i64)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= nc) return;
    const double *a = pinv + (i64)row * nc;
    double s = 0.0;
#pragma unroll 8
    for (int q = lane; q < nc; q += 32) s += a[q] * rs[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) e[place(row)] = (float)s;
}

// natural <-> level storage
__global__ void k_pack(Lay L, const float *__restrict__ nat, float *st) {
    grid_wait();
    const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= L.n) return;
    const int x = (int)(t % L.nx);
    const i64 row = t / L.nx;
    st[sto(L, x, (int)(row % L.ny), (int)(row / L.ny))] = nat[t];
}
__global__ void k_unpack(Lay L, const float *__restrict__ st, float *nat) {
    grid_wait();
    const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= L.n) return;
    const int x = (int)(t % L.nx);
    const i64 row = t / L.nx;
    nat[t] = st[sto(L, x, (int)(row % L.ny), (int)(row / L.ny))];
}
// FP64 natural -> FP32 level storage, rounded to nearest; blocks take rows (grid y, strided)
__global__ void k_pack64(Lay L, const double *__restrict__ nat, float *st) {
    grid_wait();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= L.nx) return;
    const i64 rows = (i64)L.ny * L.nz;
    for (i64 row = blockIdx.y; row < rows; row += gridDim.y) {
        const int y = (int)(row % L.ny), z = (int)(row / L.ny);
        st[sto(L, x, y, z)] = d2f_rn(nat[row * L.nx + x]);
    }
}
// s = 1/rho (FP64, natural): FP32 in the level's layout, and optionally as a pair (hi, lo) of
// FP32 numbers with hi + lo = s to about 2^-48 (natural layout) for the double-float residual
__global__ void k_pack_inv64(Lay L, const double *__restrict__ sinv, float *st, float2 *s2) {
    grid_wait();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= L.nx) return;
    const i64 rows = (i64)L.ny * L.nz;
    for (i64 row = blockIdx.y; row < rows; row += gridDim.y) {
        const int y = (int)(row % L.ny), z = (int)(row / L.ny);
        const i64 t = row * L.nx + x;
        const double v = sinv[t];
        const float hi = d2f_rn(v);
        st[sto(L, x, y, z)] = hi;
        if (s2) s2[t] = make_float2(hi, d2f_rn(v - f2d_exact(hi)));
    }
}

}  // namespace

Lay make_lay(Dims d) {
    Lay L;
    L.nx = d.nx;
    L.ny = d.ny;
    L.nz = d.nz;
    L.n = d.n;
    L.split = (d.nx % 2 == 0);
    L.hx = d.nx / 2;
    L.half = d.n / 2;
    L.zlo = L.zhi = 0;
    L.by4 = make_div((unsigned)(L.hx / 4));
    L.by_ny = make_div((unsigned)L.ny);
    L.by_nx = make_div((unsigned)L.nx);
    L.by_half = make_div((unsigned)(L.nx + 1) / 2);
    return L;
}

// one half sweep of a split level with hx % 4 == 0.  GHOST: a slab (L.zlo / L.zhi) of the decomposed
// mixed cycle, its ghost planes as z neighbours (the face arrays with their ghost plane above)
template <bool SFORM, bool GHOST>
void half32_vec(cudaStream_t s, const Lay &L, float h2, const Coef32 &cf, const float *b, float *x, int col, bool from_zero) {
    const i64 work = (i64)L.ny * L.nz * (L.hx / 4);
    if (from_zero) {
        run_kernel(k_half_vec<SFORM, true, 0, GHOST>, blocks_for(work), kThreads, 0, s, L, h2, cf, b, x, col, Upd{});
        return;
    }
    if (SFORM && run_half_zr<GHOST>(s, L, h2, cf.s, b, x, col)) return;
    run_kernel(k_half_vec<SFORM, false, 0, GHOST>, blocks_for(work), kThreads, 0, s, L, h2, cf, b, x, col, Upd{});
}

void launch_half32(cudaStream_t s, Lay L, double h2, const float *sinv, const float *fx, const float *fy,
                   const float *fz, const float *b, float *x, int col, bool from_zero) {
    Coef32 cf{sinv, fx, fy, fz};
    count_launch();
    if (L.zlo || L.zhi) {
        if (sinv) half32_vec<true, true>(s, L, (float)h2, cf, b, x, col, from_zero);
        else half32_vec<false, true>(s, L, (float)h2, cf, b, x, col, from_zero);
    } else if (L.split && L.hx % 4 == 0) {
        if (sinv) half32_vec<true, false>(s, L, (float)h2, cf, b, x, col, from_zero);
        else half32_vec<false, false>(s, L, (float)h2, cf, b, x, col, from_zero);
    } else {
        const i64 work = (i64)L.ny * L.nz * ((L.nx + 1) / 2);
        run_kernel(k_half_any, blocks_for(work), kThreads, 0, s, L, (float)h2, cf, b, x, col, from_zero ? 1 : 0);
    }
}

bool half32_update_ok(Lay L) { return L.split && L.hx % 4 == 0; }

// k_half_vec at every size: its update sweep moves 26 B per cell at 6.46 TB/s (512^3 540 us; a z-marching
// form took 567, at 256^3 79 against 71, at 288^3 163 against 102)
void launch_half32_update(cudaStream_t s, Lay L, double h2, const float *sinv, const float *fx, const float *fy,
                          const float *fz, const float *b, const float *x, double *p, float2 *p2, double alpha,
                          double shift) {
    Coef32 cf{sinv, fx, fy, fz};
    Upd up{p, p2, (float)alpha, (float)shift};
    count_launch();
    const unsigned nb = blocks_for((i64)L.ny * L.nz * (L.hx / 4));
    float *xv = const_cast<float *>(x);  // read only in the UPDATE variants
    if (L.zlo || L.zhi)  // a slab: s-form, FP64 solution (the decomposed mixed cycle)
        run_kernel(k_half_vec<true, false, 1, true>, nb, kThreads, 0, s, L, (float)h2, cf, b, xv, 0, up);
    else if (p2 && sinv) run_kernel(k_half_vec<true, false, 2>, nb, kThreads, 0, s, L, (float)h2, cf, b, xv, 0, up);
    else if (p2) run_kernel(k_half_vec<false, false, 2>, nb, kThreads, 0, s, L, (float)h2, cf, b, xv, 0, up);
    else if (sinv) run_kernel(k_half_vec<true, false, 1>, nb, kThreads, 0, s, L, (float)h2, cf, b, xv, 0, up);
    else run_kernel(k_half_vec<false, false, 1>, nb, kThreads, 0, s, L, (float)h2, cf, b, xv, 0, up);
}

void launch_residual32(cudaStream_t s, Lay L, double ih2, const float *sinv, const float *fx, const float *fy,
                       const float *fz, const float *b, const float *x, float *r, bool apply_only) {
    Coef32 cf{sinv, fx, fy, fz};
    count_launch();
    run_kernel(k_residual_any, blocks_for(L.n), kThreads, 0, s, L, (float)ih2, cf, b, x, r, apply_only ? 1 : 0);
}

void launch_resid_restrict32(cudaStream_t s, Lay L, Lay Lc, double ih2, const float *sinv, const float *fx,
                             const float *fy, const float *fz, const float *b, const float *x, float *bc,
                             bool red_only, bool tail) {
    Coef32 cf{sinv, fx, fy, fz};
    count_launch();
    if (red_only && L.split && L.hx % 4 == 0) {
        const i64 work = (i64)Lc.ny * Lc.nz * (L.hx / 4);
        if (!(L.zlo || L.zhi) && L.n <= kRrRowCells) {
            if (tail) {
                // the cluster's CTAs want most of an SM's shared memory, which has to be set aside already
                static std::atomic<unsigned long long> carved[2];
                if (!prefer_smem((const void *)k_rr_red_row<true, true>, carved[0]) ||
                    !prefer_smem((const void *)k_rr_red_row<false, true>, carved[1]))
                    (void)cudaGetLastError();  // a preference only
            }
            auto kernel = sinv ? (tail ? k_rr_red_row<true, true> : k_rr_red_row<true, false>)
                               : (tail ? k_rr_red_row<false, true> : k_rr_red_row<false, false>);
            run_kernel(kernel, (unsigned)((4 * ((work + 7) / 8 * 8) + kRrRowThreads - 1) / kRrRowThreads), kRrRowThreads, 0, s, L, Lc,
                       (float)ih2, cf, b, x, bc);
            return;
        }
        const unsigned nb = (unsigned)((work + kRrThreads - 1) / kRrThreads);
        if ((L.zlo || L.zhi) && sinv) run_kernel(k_rr_red_vec<true, true>, nb, kRrThreads, 0, s, L, Lc, (float)ih2, cf, b, x, bc);
        else if (L.zlo || L.zhi) run_kernel(k_rr_red_vec<false, true>, nb, kRrThreads, 0, s, L, Lc, (float)ih2, cf, b, x, bc);
        else if (sinv) run_kernel(k_rr_red_vec<true>, nb, kRrThreads, 0, s, L, Lc, (float)ih2, cf, b, x, bc);
        else run_kernel(k_rr_red_vec<false>, nb, kRrThreads, 0, s, L, Lc, (float)ih2, cf, b, x, bc);
        return;
    }
    run_kernel(k_resid_restrict_any, blocks_for(Lc.n), kThreads, 0, s, L, Lc, (float)ih2, cf, b, x, bc, red_only ? 1 : 0);
}

void launch_prolong32(cudaStream_t s, Lay L, Lay Lc, const float *ec, float *x, int kind, int only_col) {
    count_launch();
    if (only_col == 0 && kind == MG_PROLONG_TRILINEAR && L.split && Lc.split && Lc.nx % 8 == 0 &&
        2 * Lc.nx == L.nx && 2 * Lc.ny == L.ny && 2 * Lc.nz == L.nz) {
        const i64 work = (i64)Lc.ny * Lc.nz * (L.hx / 8);
        if (!(Lc.zlo || Lc.zhi) && L.n <= kProlRowCells) {
            run_kernel(k_prolong_red_row, (unsigned)((4 * work + kProlRowThreads - 1) / kProlRowThreads), kProlRowThreads, 0, s, L, Lc, ec, x);
            return;
        }
        const unsigned nb = (unsigned)((work + kProlThreads - 1) / kProlThreads);
        if (Lc.zlo || Lc.zhi) run_kernel(k_prolong_red8<true>, nb, kProlThreads, 0, s, L, Lc, ec, x);
        else run_kernel(k_prolong_red8<false>, nb, kProlThreads, 0, s, L, Lc, ec, x);
        return;
    }
    if (only_col == 0 && L.split && L.hx % 4 == 0) {
        const i64 work = (i64)L.ny * L.nz * (L.hx / 4);
        run_kernel(k_prolong_red_vec, blocks_for(work), kThreads, 0, s, L, Lc, ec, x, kind);
        return;
    }
    run_kernel(k_prolong_any, blocks_for(L.n), kThreads, 0, s, L, Lc, ec, x, kind, only_col);
}

void launch_coarse_matvec32(cudaStream_t s, Lay L, const double *pinv, const float *r, float *e) {
    count_launch();
    run_kernel(k_coarse_matvec_lay, blocks_for(L.n * 32), kThreads, 0, s, L, pinv, r, e);
}

void launch_pack32(cudaStream_t s, Lay L, const float *nat, float *st) {
    count_launch();
    run_kernel(k_pack, blocks_for(L.n), kThreads, 0, s, L, nat, st);
}
void launch_unpack32(cudaStream_t s, Lay L, const float *st, float *nat) {
    count_launch();
    run_kernel(k_unpack, blocks_for(L.n), kThreads, 0, s, L, st, nat);
}
void launch_pack64to32(cudaStream_t s, Lay L, const double *nat, float *st) {
    count_launch();
    const i64 rows = (i64)L.ny * L.nz;
    const dim3 grd((unsigned)((L.nx + 127) / 128), (unsigned)(rows < 65535 ? rows : 65535));
    run_kernel(k_pack64, grd, 128, 0, s, L, nat, st);
}
void launch_pack_inv_rho(cudaStream_t s, Lay L, const double *sinv, float *st, float2 *s2) {
    count_launch();
    const i64 rows = (i64)L.ny * L.nz;
    const dim3 grd((unsigned)((L.nx + 127) / 128), (unsigned)(rows < 65535 ? rows : 65535));
    run_kernel(k_pack_inv64, grd, 128, 0, s, L, sinv, st, s2);
}

}  // namespace mg
