// The coarse levels of a V-cycle in one launch: one thread-block cluster holds every level from
// a given one (TailArgs::lv[0]) down in its CTAs' shared memory and runs their smoothing sweeps, transfers and the
// dense coarse solve, CTAs waiting only for what they read.
//
// What bounds the levels below about 40^3 is the chain of dependent launches (ten per level and
// cycle, 1.5-2 us each with programmatic serialisation, for work of a fraction of a microsecond), so the
// chain is made of cheaper links: a half sweep here is one shared-memory round trip and a wait for
// the neighbours' ghosts, 0.5 us at 32^3 and 0.4 us at 16^3.  The levels 32^3, 16^3 and 8^3 of a cycle take about 25 us:
// 2 us to copy the contexts in beside the kernel before, 5.5 us for the dense product of
// 512 cells (4 us of it the FP64 FMAs on 16 SMs), 5 us for the transfers, 16 half sweeps.  A whole cycle and its share
// of a residual, launch by launch and with the cluster: 64^3 mixed 56.7 and 43.5 us, down to 4^3 73.5 and 44.2; 64^3 in
// FP64 124 and 102, 32^3 82.9 and 58.3; 128^3 94.7 and 85.8; 72 x 80 x 88 with 990 coarse cells (two launches) 67.5 and 64.6.
//
// Layout.  The rows (y, z) of a level are dealt out in quads, the four rows of one coarse row
// (J, K), so that the eight children of a coarse cell sit in one CTA; CTA r holds the quads
// [r q4, (r + 1) q4) of the order K * (ny / 2) + J.  A row of x keeps its red cells, then its
// black ones (cell x at k = x >> 1), rows padded to 8 or 24 banks past a multiple of 32 so that
// the four rows of a quad fall on different banks.  Of a row's four neighbours two are in its
// quad; the outer ones in y and z, where another CTA holds them, are kept as ghost rows that
// their owner writes (a remote store) whenever it updates the row: a remote load takes 330
// clocks and a CTA's remote loads return about 17 B per clock, against 72 clocks and 114 B for its
// own shared memory.
//
// Threads.  Item e of a colour is the cell k = (e / 4) % hx of row e % 4 of quad e / (4 hx); a
// thread owns up to kCells items of each colour and keeps their faces, right-hand side and the
// six neighbours' addresses in registers while a level is smoothed, so that a half sweep is six
// shared loads, the arithmetic and the stores.
//
// Waits.  A CTA sends its ghosts, restricted residuals and coarse results by st.async, which counts their bytes at
// an mbarrier of the receiver; the receiver knows how many will come.  Stores and a barrier of the
// cluster instead cost 830 clocks per exchange between 16 CTAs of 512 threads, this 465, and all CTAs then wait for the
// slowest (64^3 step 1561 -> 1500 us with the shared-memory copies of the parameters and addresses below).  Before a
// level reads other CTAs' x on the way up the barrier stays, and one at the end, behind a CTA's last remote store.
//
// These contexts are laid out in memory once per
// operator (k_tail_prepare), one image per CTA and level in the order of its shared memory, and
// copied in at the start of a launch.
//
// Arithmetic.  Per cell as in the level kernels (kernels_split.cu: k_half_vec, k_rr_red_vec or, where nx / 2
// is no multiple of 4, k_resid_restrict_any, k_prolong_red8 where the coarse nx is a multiple of 8, else
// k_prolong_red_vec; FP64:
// k_rbgs_half, k_rr_red_diag64, k_prolong_red64; the coarse product as k_coarse_matvec), in the same order, so that a
// cycle is bitwise the one launched level by level.
#include <cooperative_groups.h>

#include <type_traits>

#include "mg_internal.cuh"

namespace cg = cooperative_groups;

namespace mg {

namespace {

constexpr int kTailThreads = 512;

__device__ __forceinline__ void ld_cluster_wide(unsigned a, float (&v)[1]) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v[0]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ld_cluster_wide(unsigned a, float (&v)[4]) {
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ld_cluster_wide(unsigned a, double (&v)[1]) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[0]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ld_cluster_wide(unsigned a, double (&v)[2]) {
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// a remote store that reports its bytes to the mbarrier m of the CTA it goes to
__device__ __forceinline__ void st_async(unsigned a, float v, unsigned m) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a), "r"(__float_as_uint(v)), "r"(m)
                 : "memory");
}
__device__ __forceinline__ void st_async(unsigned a, double v, unsigned m) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a), "l"(__double_as_longlong(v)), "r"(m)
                 : "memory");
}
__device__ __forceinline__ unsigned map_cluster(unsigned a, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// one cell of a thread: face coefficients in the order x-, x+, y-, y+, z-, z+, the divisor (FP32:
// their sum; FP64: the reciprocal of it, and the sum for the residual), the right-hand side, and
// element offsets from the level's x: the cell, its six neighbours, two per word; ghost copies of
// the cell in other CTAs (cluster addresses, 0: none) and the mbarriers there
template <typename T>
struct Cell {
    T w[6], d, dg, b;
    unsigned ax, ay, az, own;
    unsigned g0, g1, m0, m1;
};

// bound on one wait for other CTAs' cells, about a second at the top clock, and how long a CTA that gave up stays
// after its cluster's last remote store has been issued, far more than one takes to arrive (330 clocks)
constexpr long long kTailWaitCycles = 1ll << 31, kTailLingerCycles = 1ll << 17;

template <typename T>
struct Tail {
    static constexpr bool f64 = std::is_same<T, double>::value;
    static constexpr int kCells = f64 ? kTailCells64 : kTailCells32;
    static constexpr int kReal = f64 ? 8 : 7, kWords = 6;  // context fields: T and unsigned
    static constexpr unsigned kNone = 0xffffffffu;         // Cell::own of a missing cell
    const TailArgs &a;
    const TailLevel *lv;  // a.lv in shared memory: parameters of a launch come from far away when first read
    const unsigned *cb;   // where the CTAs' shared memory begins in the cluster's: a mapa per address costs a sweep's worth
    char *sm;
    unsigned sm0, mbar;   // shared addresses of sm and of the mbarriers
    int rank, ncta, tid;

    __device__ T *x(const TailLevel &L) const { return reinterpret_cast<T *>(sm + L.off_x); }
    // right-hand side [colour][item], contexts [field][colour][item]
    __device__ T *b(const TailLevel &L) const { return reinterpret_cast<T *>(sm + L.off_b); }
    __device__ T *ctx(const TailLevel &L) const { return reinterpret_cast<T *>(sm + L.off_c); }
    __device__ unsigned *ctxw(const TailLevel &L) const { return reinterpret_cast<unsigned *>(sm + L.off_w); }
    // (J, K) of a quad (-1: none), and the cluster addresses of the 3 x 3 coarse rows around it
    // (their x) and of its own coarse row's b at k = 0, red
    __device__ int *jk(const TailLevel &L) const { return reinterpret_cast<int *>(sm + L.off_q); }
    __device__ unsigned *crow(const TailLevel &L) const { return reinterpret_cast<unsigned *>(jk(L) + L.q4); }
    // bytes of one colour that other CTAs write into this one's ghosts, and of the right-hand side
    __device__ unsigned ghost_bytes(const TailLevel &L) const { return (unsigned)jk(L)[L.q4 * 11]; }
    __device__ unsigned cell_bytes(const TailLevel &L) const { return (unsigned)jk(L)[L.q4 * 11 + 1]; }
    // the mbarriers: ghosts of colour c and the right-hand side of level l, the coarsest level's r and e.  Each level has
    // its own because a CTA may be a level ahead of another.
    __device__ unsigned bar_x(int l, int c) const { return mbar + 8 * (3 * l + c); }
    __device__ unsigned bar_b(int l) const { return mbar + 8 * (3 * l + 2); }
    __device__ unsigned bar_r() const { return mbar + 8 * (3 * kTailLevels); }
    __device__ unsigned bar_e() const { return bar_r() + 8; }
    __device__ double *rc() const { return reinterpret_cast<double *>(sm + a.off_rc); }
    __device__ T *ec() const { return reinterpret_cast<T *>(sm + a.off_ec); }
    __device__ T *cw() const { return reinterpret_cast<T *>(sm + a.off_cw); }
    // e / d of a small e for the divisor whose ceil(2^32 / d) is m (0 for d = 1)
    __device__ static int div_by(int e, unsigned m) { return m ? (int)__umulhi((unsigned)e, m) : e; }
    // global index of the cell at (colour c, k) of row (y, z)
    __device__ static i64 gidx(const TailLevel &L, int c, int k, int y, int z) {
        const i64 row = (i64)z * L.ny + y;
        return f64 ? row * L.nx + 2 * k + ((c + y + z) & 1) : c * L.half + row * L.hx + k;
    }
    __device__ static unsigned saddr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

    // a remote place: CTA and byte offset from the start of shared memory; bit 0 is free
    __device__ static unsigned place(int owner, i64 bytes) { return (unsigned)owner << 24 | (unsigned)bytes; }
    __device__ unsigned at(unsigned pl) const { return cb[pl >> 24] + (pl & 0xfffffeu); }
    // the address in CTA `owner` of what lies at a in this one
    __device__ unsigned there(unsigned a, int owner) const { return cb[owner] + (a - sm0); }

    // right-hand side (and, in the ascent alone, x with its ghosts) of this CTA's cells from memory
    __device__ void load_b(const TailLevel &L) const {
        T v[2 * kCells];  // all of a thread's loads together
        bool in[2 * kCells];
#pragma unroll
        for (int u = 0; u < 2 * kCells; ++u) {
            const int e = tid + (u % kCells) * kTailThreads, i = (u / kCells) * L.nit + e;
            int col, k, y, z;
            in[u] = e < L.nit && cell_of(L, i, col, k, y, z);
            if (in[u]) v[u] = reinterpret_cast<const T *>(L.b)[gidx(L, col, k, y, z)];
        }
#pragma unroll
        for (int u = 0; u < 2 * kCells; ++u)
            if (in[u]) b(L)[(u / kCells) * L.nit + tid + (u % kCells) * kTailThreads] = v[u];
    }
    __device__ void load_x(int l) const {
        const TailLevel &L = lv[l];
        for (int col = 0; col < 2; ++col) {
            Cell<T> q[kCells];
            restore(l, col, q);
#pragma unroll
            for (int c = 0; c < kCells; ++c) {
                int cc, k, y, z;
                if (q[c].own == kNone || !cell_of(L, col * L.nit + tid + c * kTailThreads, cc, k, y, z)) continue;
                put_plain(x(L), q[c], reinterpret_cast<const T *>(L.x)[gidx(L, col, k, y, z)]);
            }
        }
    }
    // colour, k and row of item i = col * nit + e; false past the grid
    __device__ bool cell_of(const TailLevel &L, int i, int &col, int &k, int &y, int &z) const {
        col = i >= L.nit;
        const int e = i - col * L.nit, lq = div_by(e >> 2, L.magic_hx), q = jk(L)[lq];
        k = (e >> 2) - lq * L.hx;
        y = 2 * (q & 0xffff) + (e & 1);
        z = 2 * (q >> 16) + ((e >> 1) & 1);
        return q >= 0;
    }
    // this thread's cells of one colour, without b
    __device__ __forceinline__ void restore(int l, int col, Cell<T> (&q)[kCells]) const {
        const TailLevel &L = lv[l];
#pragma unroll
        for (int c = 0; c < kCells; ++c) {
            const int e = tid + c * kTailThreads;
            q[c].own = kNone;
            if (e >= L.nit) continue;
            const int i = col * L.nit + e, n2 = 2 * L.nit;
            const T *f = ctx(L) + i;
            const unsigned *w = ctxw(L) + i;
#pragma unroll
            for (int u = 0; u < 6; ++u) q[c].w[u] = f[u * n2];
            q[c].d = f[6 * n2];
            q[c].dg = f64 ? f[(kReal - 1) * n2] : T(0);
            q[c].ax = w[0];
            q[c].ay = w[n2];
            q[c].az = w[2 * n2];
            q[c].own = w[3 * n2];
            q[c].g0 = w[4 * n2] == kNone ? 0u : at(w[4 * n2]);
            q[c].g1 = w[5 * n2] == kNone ? 0u : at(w[5 * n2]);
            q[c].m0 = q[c].g0 ? there(bar_x(l, col), (int)(w[4 * n2] >> 24)) : 0u;
            q[c].m1 = q[c].g1 ? there(bar_x(l, col), (int)(w[5 * n2] >> 24)) : 0u;
        }
    }
    __device__ __forceinline__ void restore_b(const TailLevel &L, int col, Cell<T> (&q)[kCells]) const {
#pragma unroll
        for (int c = 0; c < kCells; ++c)
            if (q[c].own != kNone) q[c].b = b(L)[col * L.nit + tid + c * kTailThreads];
    }
    // x of this CTA's cells into memory, and b
    __device__ void store(const TailLevel &L, bool with_b) const {
#pragma unroll
        for (int u = 0; u < 2 * kCells; ++u) {
            const int e = tid + (u % kCells) * kTailThreads, i = (u / kCells) * L.nit + e;
            int col, k, y, z;
            if (e >= L.nit || !cell_of(L, i, col, k, y, z)) continue;
            const i64 g = gidx(L, col, k, y, z);
            reinterpret_cast<T *>(L.x)[g] = x(L)[ctxw(L)[3 * 2 * L.nit + i]];
            if (with_b) reinterpret_cast<T *>(L.b)[g] = b(L)[i];
        }
    }

    // a0 b0 + a1 b1 as the level kernels' sums of products begin: FP32 fma(a0, b0, a1 b1), FP64
    // fma(a1, b1, a0 b0)
    __device__ static T first_two(T a0, T b0, T a1, T b1) {
        return f64 ? fma(a1, b1, a0 * b0) : fma(a0, b0, a1 * b1);
    }
    __device__ __forceinline__ static void neighbours(const T *X, const Cell<T> &q, T (&v)[6]) {
        v[0] = X[q.ax & 0xffffu];
        v[1] = X[q.ax >> 16];
        v[2] = X[q.ay & 0xffffu];
        v[3] = X[q.ay >> 16];
        v[4] = X[q.az & 0xffffu];
        v[5] = X[q.az >> 16];
    }
    __device__ __forceinline__ static void put_plain(T *X, const Cell<T> &q, T v) {
        X[q.own] = v;
        if (q.g0) st_cluster(q.g0, v);
        if (q.g1) st_cluster(q.g1, v);
    }
    __device__ __forceinline__ static void put(T *X, const Cell<T> &q, T v, bool send) {
        X[q.own] = v;
        if (send && q.g0) st_async(q.g0, v, q.m0);
        if (send && q.g1) st_async(q.g1, v, q.m1);
    }

    // until `bytes` have come in for the mbarrier m; its bytes may come before this.  The wait is bounded: a thread
    // whose wait runs out is lost.  It then neither waits nor stores into other CTAs any more, so that no mbarrier
    // gets bytes of a later phase or a second arrival in one phase, and its neighbours' waits run out in turn;
    // it takes part in every barrier up to the end, and its CTA leaves NaN and an error flag.
    __device__ __forceinline__ void expect(unsigned m, unsigned bytes, bool lost) const {
        if (tid == 0 && !lost)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(m), "r"(bytes) : "memory");
    }
    __device__ __forceinline__ static bool arrived(unsigned m, unsigned parity) {
        unsigned done;
        asm volatile(
            "{.reg .pred P; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], %2; selp.u32 %0, 1, 0, P;}"
            : "=r"(done)
            : "r"(m), "r"(parity)
            : "memory");
        return done != 0;
    }
    __device__ __forceinline__ void wait(unsigned m, unsigned parity, bool &lost) const {
        if (lost || arrived(m, parity)) return;
        const long long t0 = clock64();
        while (!arrived(m, parity))
            if (clock64() - t0 > kTailWaitCycles) {
                lost = true;
                return;
            }
    }
    // after the cells of colour col have been put: until this CTA's are visible to its threads and the ghosts'
    // have arrived.  A neighbour sends the next values of a ghost only once it has had every cell of
    // this CTA that reads the present ones, so nothing is overwritten early.
    __device__ __forceinline__ void exchange(int l, int col, unsigned &parity, bool &lost) const {
        expect(bar_x(l, col), ghost_bytes(lv[l]), lost);
        __syncthreads();
        wait(bar_x(l, col), parity >> (2 * l + col) & 1u, lost);
        parity ^= 1u << (2 * l + col);
    }

    __device__ __forceinline__ void half(T *X, T h2, const Cell<T> (&q)[kCells], bool send) const {
#pragma unroll
        for (int c = 0; c < kCells; ++c) {
            if (q[c].own == kNone) continue;
            T v[6];
            neighbours(X, q[c], v);
            T num = first_two(q[c].w[0], v[0], q[c].w[1], v[1]);
#pragma unroll
            for (int u = 2; u < 6; ++u) num = fma(q[c].w[u], v[u], num);
            if constexpr (f64) put(X, q[c], fma(h2, q[c].b, num) * q[c].d, send);
            else put(X, q[c], __fdividef(fmaf(h2, q[c].b, num), q[c].d), send);
        }
    }

    // index of cell (I, J, K) of the coarsest level in memory
    __device__ i64 coarse_idx(int I, int J, int K, int cnx, int cny) const {
        const i64 row = (i64)K * cny + J;
        if (f64 || (cnx & 1)) return row * cnx + I;
        return ((I + J + K) & 1) * a.half_c + row * (cnx >> 1) + (I >> 1);
    }
    // mean of the children's residuals (black ones 0 after a black half sweep) into the next
    // level's b: its owner's shared memory, every CTA's copy for the coarse solve, or memory.  The four
    // red children of a coarse cell are four neighbouring lanes.
    __device__ void restrict_red(int l, const TailLevel *C, bool coarse_mem, const Cell<T> (&q)[kCells], bool lost) const {
        const TailLevel &L = lv[l];
        const T *X = x(L);
        const int cnx = L.nx >> 1, cny = L.ny >> 1;
#pragma unroll
        for (int c = 0; c < kCells; ++c) {
            const int e = tid + c * kTailThreads;
            T r = T(0);
            if (q[c].own != kNone) {
                T v[6];
                neighbours(X, q[c], v);
                const T xc = X[q[c].own];
                if constexpr (f64) {
                    r = (T)L.h2 * q[c].b;
#pragma unroll
                    for (int u = 0; u < 6; ++u) r = fma(q[c].w[u], v[u], r);
                    r = fma(-q[c].dg, xc, r);
                } else if (L.hx % 4 != 0) {  // as k_resid_restrict_any
                    float num = first_two(q[c].w[0], v[0], q[c].w[1], v[1]);
#pragma unroll
                    for (int u = 2; u < 6; ++u) num = fmaf(q[c].w[u], v[u], num);
                    r = fmaf(-fmaf(xc, q[c].d, -num), (float)L.ih2, q[c].b);
                } else {
                    float ax = first_two(q[c].w[0], xc - v[0], q[c].w[1], xc - v[1]);
#pragma unroll
                    for (int u = 2; u < 6; ++u) ax = fmaf(q[c].w[u], xc - v[u], ax);
                    r = fmaf(-ax, (float)L.ih2, q[c].b);
                }
            }
            const T r1 = __shfl_down_sync(0xffffffffu, r, 1), r2 = __shfl_down_sync(0xffffffffu, r, 2);
            const T r3 = __shfl_down_sync(0xffffffffu, r, 3);
            T bc = (((r + r1) + r2) + r3) * (T)(f64 ? L.ih2 * 0.125 : 0.125);
            bc = __shfl_sync(0xffffffffu, bc, (tid & 31) & ~3);
            const int ch = e & 3;
            if (q[c].own == kNone || (ch && (C || coarse_mem))) continue;
            const int lq = div_by(e >> 2, L.magic_hx), k = (e >> 2) - lq * L.hx;
            const int J = jk(L)[lq] & 0xffff, K = jk(L)[lq] >> 16;
            if (C) {
                const unsigned pl = crow(L)[lq * 10 + 9];
                if (!lost) st_async(at(pl) + (unsigned)((((k + J + K) & 1) * C->nit + (k >> 1) * 4) * sizeof(T)), bc,
                         there(bar_b(l + 1), (int)(pl >> 24)));
            } else if (coarse_mem) {
                reinterpret_cast<T *>(a.bc)[coarse_idx(k, J, K, cnx, cny)] = bc;
            } else if (!lost) {
                const unsigned r0 = saddr(rc() + (K * cny + J) * cnx + k);
                for (int t = ch; t < ncta; t += 4) st_async(there(r0, t), (double)bc, there(bar_r(), t));
            }
        }
    }

    // e = A^+ r on the coarsest level, every CTA receiving the whole e
    __device__ void coarse_solve(bool lost) const {
        const int lane = tid & 31, warp = tid >> 5, n = a.nc;
        const double *r = rc();
        // two rows per warp: lanes 0-15 end up with the first row's sum, 16-31 with the second's, each
        // in the order of the xor shuffle over 32 lanes (half the FP64 additions of two such sums)
        const int stride = ncta * (kTailThreads / 32);
        for (int row = warp * ncta + rank; row < n; row += 2 * stride) {
            const bool two = row + stride < n;
            const double *m0 = a.pinv + (i64)row * n, *m1 = two ? m0 + (i64)stride * n : m0;
            double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
            for (int q = lane; q < n; q += 32) {
                const double rq = r[q];
                s0 = fma(m0[q], rq, s0);
                if (two) s1 = fma(m1[q], rq, s1);
            }
            const bool hi = lane >= 16;
            double s = (hi ? s1 : s0) + __shfl_xor_sync(0xffffffffu, hi ? s0 : s1, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            const double t0 = __shfl_sync(0xffffffffu, s, 0), t1 = __shfl_sync(0xffffffffu, s, 16);
            if (lane < ncta && !lost) {
                const unsigned e0 = there(saddr(ec() + row), lane), m = there(bar_e(), lane);
                st_async(e0, (T)t0, m);
                if (two) st_async(e0 + (unsigned)(stride * sizeof(T)), (T)t1, m);
            }
        }
    }

    // the 3 x 3 coarse rows around each quad into this CTA's scratch, in the order of I with its end
    // values repeated beyond the walls: cw[(9 quad + 3 (K' - K + 1) + J' - J + 1) (cnx + 2) + I + 1]
    __device__ void gather(const TailLevel &L, const TailLevel &C) const {
        constexpr int kV = 16 / (int)sizeof(T);
        if (C.hx % kV == 0) gather_wide<kV>(L, C);
        else gather_wide<1>(L, C);
    }
    // kV cells of one colour per load, all of a thread's loads in flight (32^3 from 16^3: 576 loads of 16 bytes)
    template <int kV>
    __device__ void gather_wide(const TailLevel &L, const TailLevel &C) const {
        constexpr int kU = kV > 1 ? 2 : 4;
        const int per = C.nx / kV, n = L.q4 * 9 * per, st = C.nx + 2;
        for (int e0 = tid; e0 < n; e0 += kU * kTailThreads) {
            T v[kU][kV];
            int d[kU], Ic[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int e = min(e0 + u * kTailThreads, n - 1), r = div_by(e * kV, C.magic_nx), i = (e - r * per) * kV;
                const unsigned pl = crow(L)[r + r / 9];  // ten words per quad
                const int col = i >= C.hx;
                Ic[u] = 2 * (i - col * C.hx) + ((col + (int)pl) & 1);  // bit 0: parity of J' + K'
                d[u] = r * st + Ic[u] + 1;
#pragma unroll
                for (int w = 0; w < kV; ++w) v[u][w] = T(0);
                if (pl != kNone) ld_cluster_wide(at(pl) + (unsigned)(i * sizeof(T)), v[u]);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (e0 + u * kTailThreads >= n) continue;
#pragma unroll
                for (int w = 0; w < kV; ++w) cw()[d[u] + 2 * w] = v[u][w];
                if (Ic[u] == 0) cw()[d[u] - 1] = v[u][0];
                if (Ic[u] + 2 * (kV - 1) == C.nx - 1) cw()[d[u] + 2 * kV - 1] = v[u][kV - 1];
            }
        }
    }
    // x += P e on the red cells q, e the next level's x
    __device__ void prolong_red(const TailLevel &L, const TailLevel *C, const Cell<T> (&q)[kCells], bool lost) const {
        const int cnx = L.nx >> 1, cny = L.ny >> 1, cnz = L.nz >> 1;
        if (C) {
            gather(L, *C);
            __syncthreads();
        }
        T *X = x(L);
#pragma unroll
        for (int m = 0; m < kCells; ++m) {
            if (q[m].own == kNone) continue;
            const int e = tid + m * kTailThreads, lq = div_by(e >> 2, L.magic_hx), I = (e >> 2) - lq * L.hx;
            const int dy = e & 1, dz = (e >> 1) & 1;
            const T *o;        // own coarse value, and the steps to its neighbours
            int si, sj, sk;
            if (C) {
                si = (dy ^ dz) ? 1 : -1;
                sj = (dy ? 1 : -1) * (cnx + 2);
                sk = (dz ? 3 : -3) * (cnx + 2);
                o = cw() + (lq * 9 + 4) * (cnx + 2) + I + 1;
            } else {
                const int J = jk(L)[lq] & 0xffff, K = jk(L)[lq] >> 16;
                const int I2 = (dy ^ dz) ? min(I + 1, cnx - 1) : max(I - 1, 0);
                si = I2 - I;
                sj = ((dy ? min(J + 1, cny - 1) : max(J - 1, 0)) - J) * cnx;
                sk = ((dz ? min(K + 1, cnz - 1) : max(K - 1, 0)) - K) * cnx * cny;
                o = ec() + (K * cny + J) * cnx + I;
            }
            // c[4 kk + 2 jj + ii]: own (0) or neighbour (1) along z, y, x
            const T c[8] = {o[0], o[si], o[sj], o[sj + si], o[sk], o[sk + si], o[sk + sj], o[sk + sj + si]};
            T v = X[q[m].own];
            if constexpr (f64) {
                // as k_prolong_red64: y, then z, then x, weights 3 and 1, 1/64 at the end
                T R[2];
#pragma unroll
                for (int ii = 0; ii < 2; ++ii)
                    R[ii] = fma(T(3), fma(T(3), c[ii], c[2 + ii]), fma(T(3), c[4 + ii], c[6 + ii]));
                v = fma(fma(T(3), R[0], R[1]), T(0.015625), v);
            } else if (cnx % 8 == 0) {
                // separable: y and z first, rows in the order J - 1, J, J + 1 and then K - 1, K, K + 1
                T R[2];
#pragma unroll
                for (int ii = 0; ii < 2; ++ii) {
                    T r = T(0);
#pragma unroll
                    for (int ja = 0; ja < 2; ++ja)
#pragma unroll
                        for (int ka = 0; ka < 2; ++ka) {
                            const int jj = dy ? ja : 1 - ja, kk = dz ? ka : 1 - ka;  // 0 own, 1 neighbour
                            const T val = kk ? (jj ? c[6 + ii] : c[4 + ii]) : (jj ? c[2 + ii] : c[ii]);
                            r = fma((jj ? T(0.25) : T(0.75)) * (kk ? T(0.25) : T(0.75)), val, r);
                        }
                    R[ii] = r;
                }
                v += fma(T(0.75), R[0], T(0.25) * R[1]);
            } else {
                const T w[2] = {T(0.75), T(0.25)};
                T r = first_two(w[0] * w[0] * w[0], c[0], w[1] * w[0] * w[0], c[1]);
#pragma unroll
                for (int u = 2; u < 8; ++u) r = fma(w[u & 1] * w[(u >> 1) & 1] * w[u >> 2], c[u], r);
                v += r;
            }
            put(X, q[m], v, !lost);
        }
    }
};

// the image of one level and CTA (blockIdx.y, blockIdx.x) from the level's arrays: contexts and tables
template <typename T>
__global__ void __launch_bounds__(256) k_tail_prepare(const __grid_constant__ TailArgs a) {
    grid_wait();
    using U = Tail<T>;
    const TailLevel &L = a.lv[blockIdx.y];
    const TailLevel *C = (int)blockIdx.y + 1 < a.nl ? &a.lv[blockIdx.y + 1] : nullptr;
    const int rank = blockIdx.x, cny = L.ny >> 1, cnz = L.nz >> 1;
    char *img = reinterpret_cast<char *>(a.img) + L.img + (size_t)rank * L.img_bytes;
    T *ctx = reinterpret_cast<T *>(img);
    unsigned *ctxw = reinterpret_cast<unsigned *>(img + (L.off_w - L.off_c));
    int *jk = reinterpret_cast<int *>(img + (L.off_q - L.off_c));
    unsigned *crow = reinterpret_cast<unsigned *>(jk + L.q4);
    __shared__ int ghosts, quads;
    if (threadIdx.x == 0) ghosts = quads = 0;
    __syncthreads();
    for (int lq = threadIdx.x; lq < L.q4; lq += 256) {
        const int qd = rank * L.q4 + lq, K = qd / cny, J = qd - K * cny;
        jk[lq] = K < cnz ? J | K << 16 : -1;
        if (K < cnz) atomicAdd(&quads, 1);
        // the coarse rows around the quad (their x) and the place of its own coarse row's b
        for (int r = 0; r < 10 && C; ++r) {
            unsigned pl = U::kNone;
            if (K < cnz) {
                const int Jn = r < 9 ? min(max(J + r % 3 - 1, 0), cny - 1) : J;
                const int Kn = r < 9 ? min(max(K + r / 3 - 1, 0), cnz - 1) : K;
                const int qc = (Kn >> 1) * (C->ny >> 1) + (Jn >> 1), owner = qc / C->q4;
                const int lc = qc - owner * C->q4, ch = (Kn & 1) * 2 + (Jn & 1);
                pl = r < 9 ? U::place(owner, C->off_x + (i64)(lc * 4 + ch) * C->rs * sizeof(T)) | ((Jn + Kn) & 1)
                           : U::place(owner, C->off_b + (i64)(lc * 4 * C->hx + ch) * sizeof(T));
            }
            crow[lq * 10 + r] = pl;
        }
    }
    const T *fx = reinterpret_cast<const T *>(L.fx), *fy = reinterpret_cast<const T *>(L.fy);
    const T *fz = reinterpret_cast<const T *>(L.fz);
    for (int i = threadIdx.x; i < 2 * L.nit; i += 256) {
        const int col = i >= L.nit, e = i - col * L.nit, lq = (e >> 2) / L.hx, k = (e >> 2) - lq * L.hx, s = lq * 4 + (e & 3);
        const int qd = rank * L.q4 + lq, K = qd / cny, J = qd - K * cny;
        const int y = 2 * J + (e & 1), z = 2 * K + ((e >> 1) & 1), p = (col + y + z) & 1;
        const int o = (1 - col) * L.hx, cell = col * L.hx + k;
        T f[8] = {};
        unsigned w[U::kWords] = {0, 0, 0, U::kNone, U::kNone, U::kNone};
        if (K < cnz) {
            const i64 g = U::gidx(L, col, k, y, z);
            f[0] = fx[g];
            if (k + p < L.hx) f[1] = fx[U::gidx(L, 1 - col, k + p, y, z)];
            f[2] = fy[g];
            if (y < L.ny - 1) f[3] = fy[U::gidx(L, 1 - col, k, y + 1, z)];
            f[4] = fz[g];
            if (z < L.nz - 1) f[5] = fz[U::gidx(L, 1 - col, k, y, z + 1)];
            if constexpr (U::f64) {
                f[6] = reinterpret_cast<const T *>(L.invd)[col * L.half + ((i64)z * L.ny + y) * L.hx + k];
                f[7] = reinterpret_cast<const T *>(L.diag)[g];
            } else {
                f[6] = ((f[0] + f[1]) + (f[2] + f[3])) + (f[4] + f[5]);
            }
            // the rows of the outer neighbours: here, a ghost of a row elsewhere (then that CTA
            // keeps a ghost of this row at the same place of its own slot), or at a wall the row itself
            int out[2];
            for (int d = 0; d < 2; ++d) {
                const int yn = d ? y : y + ((y & 1) ? 1 : -1), zn = d ? z + ((z & 1) ? 1 : -1) : z;
                out[d] = s * L.rs;
                if (yn < 0 || yn >= L.ny || zn < 0 || zn >= L.nz) continue;
                const int qn = (zn >> 1) * cny + (yn >> 1), owner = qn / L.q4;
                const int sn = (qn - owner * L.q4) * 4 + (zn & 1) * 2 + (yn & 1);
                if (owner == rank) {
                    out[d] = sn * L.rs;
                } else {
                    if (k == 0 && col == 0) atomicAdd(&ghosts, 1);
                    out[d] = (L.q4 * 4 + s * 2 + d) * L.rs;
                    w[4 + d] = U::place(owner, L.off_x + (i64)((L.q4 * 4 + sn * 2 + d) * L.rs + cell) * sizeof(T));
                }
            }
            const unsigned row = s * L.rs + o, km = k + p - 1, kp = k + p;
            const unsigned yi = (s ^ 1) * L.rs + o + k, yo = out[0] + o + k, zi = (s ^ 2) * L.rs + o + k, zo = out[1] + o + k;
            w[0] = (row + (k + p >= 1 ? km : 0)) | (row + ((int)kp < L.hx ? kp : k)) << 16;
            w[1] = (s & 1) ? yi | yo << 16 : yo | yi << 16;
            w[2] = (s & 2) ? zi | zo << 16 : zo | zi << 16;
            w[3] = s * L.rs + cell;
        }
        for (int u = 0; u < U::kReal; ++u) ctx[u * 2 * L.nit + i] = f[u];
        for (int u = 0; u < U::kWords; ++u) ctxw[u * 2 * L.nit + i] = w[u];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        jk[L.q4 * 11] = ghosts * L.hx * (int)sizeof(T);  // one colour's
        jk[L.q4 * 11 + 1] = quads * 4 * L.nx * (int)sizeof(T);
    }
}

// mode: kTailAll the whole descent and ascent; kTailDown / kTailUp one of them, with the
// coarse solve launched between the two on the whole device and the levels kept in memory
template <typename T>
__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const __grid_constant__ TailArgs a, int mode) {
    extern __shared__ __align__(16) char tail_smem[];
    cg::cluster_group cl = cg::this_cluster();
    __shared__ __align__(8) unsigned long long mbar[3 * kTailLevels + 2];
    __shared__ TailLevel lv[kTailLevels];
    static_assert(sizeof(TailLevel) % 4 == 0 && std::is_trivially_copyable<TailLevel>::value, "copied by words");
    for (int e = threadIdx.x; e < a.nl * (int)(sizeof(TailLevel) / 4); e += kTailThreads)
        reinterpret_cast<unsigned *>(lv)[e] = reinterpret_cast<const unsigned *>(a.lv)[e];
    __shared__ unsigned cb[16];
    const unsigned sm0 = Tail<T>::saddr(tail_smem);
    if (threadIdx.x < cl.num_blocks()) cb[threadIdx.x] = map_cluster(sm0, (int)threadIdx.x);
    const Tail<T> t{a, lv, cb, tail_smem, sm0, Tail<T>::saddr(mbar), (int)cl.block_rank(), (int)cl.num_blocks(), (int)threadIdx.x};
    if (t.tid == 0) {
        for (int c = 0; c < 3 * kTailLevels + 2; ++c) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(t.mbar + 8 * c) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    unsigned parity = 0;  // of bar_x, bit 2 l + c
    bool lost = false;
    __syncthreads();
    const bool from_mem = mode == kTailUp;
#pragma unroll 1
    for (int l = 0; l < a.nl; ++l) {
        const TailLevel &L = lv[l];
        const char *img = reinterpret_cast<const char *>(a.img) + L.img + (size_t)t.rank * L.img_bytes;
        const float4 *src = reinterpret_cast<const float4 *>(img);
        float4 *dst = reinterpret_cast<float4 *>(tail_smem + L.off_c);
        const int n4 = L.img_bytes / 16;
        // eight loads in flight per thread (cp.async would be shorter, but every cluster barrier of a
        // block that has used it takes 700 clocks more)
        for (int o0 = t.tid; o0 < n4; o0 += 8 * kTailThreads) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (o0 + u * kTailThreads < n4) v[u] = __ldg(src + o0 + u * kTailThreads);
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (o0 + u * kTailThreads < n4) dst[o0 + u * kTailThreads] = v[u];
        }
        float4 *x4 = reinterpret_cast<float4 *>(t.x(L));  // rows and ghosts from zero
        for (int e = t.tid; e < (L.off_b - L.off_x) / 16; e += kTailThreads) x4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    grid_wait();  // the contexts were written long before (set-up ends with a synchronisation); b was not
    __syncthreads();
    t.load_b(lv[0]);
    if (from_mem) {
        cl.sync();  // every CTA's ghosts are zeroed before others write them
        for (int l = 0; l < a.nl; ++l) {
            t.load_x(l);
            if (l > 0) t.load_b(lv[l]);
        }
        for (int q = t.tid; q < a.nc; q += kTailThreads) {
            const int cnx = lv[a.nl - 1].nx >> 1, cny = lv[a.nl - 1].ny >> 1, row = q / cnx;
            t.ec()[q] = reinterpret_cast<const T *>(a.xc)[t.coarse_idx(q - row * cnx, row % cny, row / cny, cnx, cny)];
        }
    }
    cl.barrier_arrive();
    // visits nl levels down and nl up; `first` is the colour a sweep begins with
    const int v0 = from_mem ? a.nl : 0, v1 = mode == kTailDown ? a.nl : 2 * a.nl;
    Cell<T> first[Tail<T>::kCells], second[Tail<T>::kCells];
    auto restore = [&](int v) {  // everything but b, which may still be on its way
        const bool up = v >= a.nl;
        const int l = up ? 2 * a.nl - 1 - v : v;
        t.restore(l, up ? 1 : 0, first);
        t.restore(l, up ? 0 : 1, second);
    };
    // the last of this thread's remote accesses is over: no CTA leaves the kernel before all threads of the cluster have
    // come this far, whether or not their waits ran out (what was sent before may still be under way)
    auto leave = [] { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); };
    restore(v0);
    cl.barrier_wait();
#pragma unroll 1
    for (int v = v0; v < v1; ++v) {
        const bool up = v >= a.nl;
        const int l = up ? 2 * a.nl - 1 - v : v;
        const TailLevel &L = lv[l];
        const TailLevel *C = l + 1 < a.nl ? &lv[l + 1] : nullptr;
        t.restore_b(L, up ? 1 : 0, first);
        t.restore_b(L, up ? 0 : 1, second);
        const int c0 = up ? 1 : 0;
        if (up) {
            t.prolong_red(L, C, second, lost);
            t.exchange(l, 0, parity, lost);
        }
        T *X = t.x(L);
        const T h2 = (T)L.h2;
#pragma unroll 1
        for (int sw = up ? a.post : a.pre;;) {
            t.half(X, h2, first, !lost);
            t.exchange(l, c0, parity, lost);
            --sw;
            if (up && sw == 0 && v + 1 == v1) leave();
            t.half(X, h2, second, !lost && (!up || sw > 0));  // nothing reads the ghosts of an ascent's last half sweep
            if (sw == 0) break;
            t.exchange(l, 1 - c0, parity, lost);
        }
        if (!up) {
            t.exchange(l, 1 - c0, parity, lost);
            if (mode == kTailDown && v + 1 == v1) leave();
            t.restrict_red(l, C, mode == kTailDown, first, lost);
        }
        if (v + 1 == v1) break;
        // the next level's contexts come in meanwhile.  On the way down a CTA waits for what it
        // reads; on the way up the next level reads other CTAs' x
        if (up) cl.barrier_arrive();
        restore(v + 1);
        if (up) {
            cl.barrier_wait();
        } else if (C) {
            t.expect(t.bar_b(l + 1), t.cell_bytes(*C), lost);
            t.wait(t.bar_b(l + 1), 0, lost);
        } else {
            t.expect(t.bar_r(), (unsigned)(a.nc * sizeof(double)), lost);
            t.wait(t.bar_r(), 0, lost);
            t.coarse_solve(lost);
            t.expect(t.bar_e(), (unsigned)(a.nc * sizeof(T)), lost);
            t.wait(t.bar_e(), 0, lost);
        }
    }
    const bool gave_up = __syncthreads_or(lost);
    if (gave_up) {  // the level's x without a number fails the solve
        if (t.tid == 0) atomicOr(a.err, 8u);
        for (int i = t.tid; i < (lv[0].off_b - lv[0].off_x) / (int)sizeof(T); i += kTailThreads) t.x(lv[0])[i] = (T)NAN;
        __syncthreads();
    }
    for (int l = 0; l < (mode == kTailDown ? a.nl : 1); ++l) t.store(lv[l], l > 0);
    cl.barrier_wait();  // that of leave(), over by now where no wait ran out
    // what other CTAs had sent this one, which a CTA that did not give up has waited for, arrives before it goes
    if (gave_up)
        for (const long long t0 = clock64(); clock64() - t0 < kTailLingerCycles;) {}
}

template <typename T>
cudaError_t launch_mode(cudaStream_t s, const TailArgs &a, int mode) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.ncta);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = (size_t)a.smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)a.ncta;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = stream_capturing(s) ? 1 : 2;
    return cudaLaunchKernelEx(&cfg, k_tail<T>, a, mode);
}

// whether one cluster of a.ncta CTAs with a.smem bytes fits the device; opts the kernel in
template <typename T>
bool cluster_fits(const TailArgs &a) {
    if (cudaFuncSetAttribute(k_tail<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTailMaxSmem) != cudaSuccess ||
        cudaFuncSetAttribute(k_tail<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.ncta);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = (size_t)a.smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)a.ncta;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_tail<T>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return n >= 1;
}

}  // namespace

bool tail_layout(TailArgs &a, bool fp64, int ncta) {
    const int es = fp64 ? 8 : 4, cells = fp64 ? kTailCells64 : kTailCells32;
    const int real = fp64 ? Tail<double>::kReal : Tail<float>::kReal;
    a.ncta = ncta;
    i64 off = 0, cw = 0, img = 0;  // cw: coarse rows gathered for a prolongation
    auto take = [&](i64 bytes) {
        const i64 o = off;
        off += (bytes + 15) & ~(i64)15;
        return (int)o;
    };
    auto magic = [](int d) { return d > 1 ? (unsigned)((0x100000000ull + d - 1) / d) : 0u; };
    for (int l = 0; l < a.nl; ++l) {
        TailLevel &L = a.lv[l];
        const i64 quads = (i64)(L.ny / 2) * (L.nz / 2), q4 = (quads + ncta - 1) / ncta;
        if (q4 * 2 * L.nx > (i64)cells * kTailThreads) return false;  // items per colour
        // (J, K) are packed in 16 bits
        if (L.ny >= 32768 || L.nz >= 32768) return false;
        L.hx = L.nx / 2;
        L.q4 = (int)q4;
        L.nit = L.q4 * 4 * L.hx;
        L.rs = L.nx;
        while (L.rs % 32 != 8 && L.rs % 32 != 24) ++L.rs;
        // element offsets (rows and ghosts) are packed in 16 bits, and the magic divisions are
        // exact below 2^16
        if ((i64)L.q4 * 12 * L.rs >= 65536 || (i64)L.q4 * 9 * L.nx >= 65536) return false;
        L.magic_nx = magic(L.nx);
        L.magic_hx = magic(L.hx);
        L.off_x = take((i64)L.q4 * 12 * L.rs * es);
        L.off_b = take((i64)2 * L.nit * es);
        L.off_c = take((i64)real * 2 * L.nit * es);
        L.off_w = take((i64)Tail<float>::kWords * 2 * L.nit * 4);
        L.off_q = take(4 * ((i64)L.q4 * 11 + 2));
        L.img_bytes = (int)(off - L.off_c);
        L.img = img;
        img += (i64)ncta * L.img_bytes;
        if (l + 1 < a.nl && (i64)L.q4 * 9 * (L.hx + 2) > cw) cw = (i64)L.q4 * 9 * (L.hx + 2);
        if (off > kTailMaxSmem) return false;
    }
    a.off_rc = take(8 * (i64)a.nc);
    a.off_ec = take((i64)es * a.nc);
    a.off_cw = take(es * cw);
    a.img_total = img;
    if (off > kTailMaxSmem) return false;
    // more than half of an SM's shared memory: two CTAs of the cluster on one SM would share its
    // FP64 pipe and issue slots while another SM idles
    a.smem = (int)(off > kTailMinSmem ? off : kTailMinSmem);
    return fp64 ? cluster_fits<double>(a) : cluster_fits<float>(a);
}

void launch_tail_prepare(cudaStream_t s, const TailArgs &a, bool fp64) {
    count_launch();
    const dim3 grd(a.ncta, a.nl);
    if (fp64) run_kernel(k_tail_prepare<double>, grd, 256, 0, s, a);
    else run_kernel(k_tail_prepare<float>, grd, 256, 0, s, a);
}

unsigned *tail_ghost_bytes(const TailArgs &a) {
    const TailLevel &L = a.lv[0];
    return reinterpret_cast<unsigned *>(reinterpret_cast<char *>(a.img) + L.img + (L.off_q - L.off_c) + 4 * (i64)L.q4 * 11);
}

void launch_tail(cudaStream_t s, const TailArgs &a, bool fp64, int mode) {
    count_launch();
    // a refused launch stays in the runtime's last error, which the caller checks
    (void)(fp64 ? launch_mode<double>(s, a, mode) : launch_mode<float>(s, a, mode));
}

}  // namespace mg
