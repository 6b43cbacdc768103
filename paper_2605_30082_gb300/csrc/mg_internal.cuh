// Internal declarations of the GB300 multigrid Poisson library (not part of the ABI).
//
// Storage inside the library.  Every per-level array is a cell array of the
// level's shape (nz, ny, nx), x fastest.  Face coefficients are kept as three
// cell arrays of LOW faces: fx[c] is the coefficient of the face between cell
// c and its x-1 neighbour (0 for i = 0, the wall); the high face of c is the
// low face of its x+1 neighbour, or the wall (0) when i = nx-1.  The ABI's
// (n+1)-long face layouts are converted on entry and exit.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/mg.h"

namespace mg {

typedef long long i64;

struct Dims {
    int nx, ny, nz;
    i64 nxy, n;
    // z slab of a domain-decomposed level (mg_dd.cu): a ghost plane below (zlo) or above (zhi)
    // the nz own planes holds the neighbouring slab's values, so the faces between slabs count
    // as interior; 0 on every whole-grid level (the walls)
    int zlo, zhi;
};

inline Dims make_dims(int nx, int ny, int nz) {
    Dims d;
    d.nx = nx;
    d.ny = ny;
    d.nz = nz;
    d.nxy = (i64)nx * ny;
    d.n = d.nxy * nz;
    d.zlo = d.zhi = 0;
    return d;
}

// Division of n < 2^31 by a fixed d >= 1 with one multiplication (m = floor(2^32 (2^s - d) / d) + 1, s = ceil(log2 d)):
// n / d = (umulhi(n, m) + n) >> s.  A 32-bit division by a variable takes some 20 dependent
// instructions, and the small half sweeps, where a thread has three before its first load, feel them.
struct FastDiv {
    unsigned m, s;
};
inline FastDiv make_div(unsigned d) {
    if (d < 1) d = 1;
    unsigned s = 0;
    while ((1ull << s) < d) ++s;
    return FastDiv{(unsigned)(((1ull << 32) * ((1ull << s) - d)) / d + 1), s};
}
#ifdef __CUDACC__
__device__ __forceinline__ unsigned operator/(unsigned n, const FastDiv &f) { return (__umulhi(n, f.m) + n) >> f.s; }
#endif

// Storage layout of an FP32 level: colour-split (all red cells, then all black, each
// colour row by row, cell x of a row at k = x >> 1) when nx is even, else natural.
// A z slab of a decomposed level (mg_dd.cu, split layout only) keeps a ghost plane below and
// above its nz own planes in each colour half: `half` is then the stride between the two
// halves (nz + 2 planes each), the arrays point at the red half's first own plane, and zlo /
// zhi say whether the ghost below / above holds a neighbour's values (the planes between
// slabs count as interior) or is a wall; the slab starts at an even whole-grid plane, so the
// colour of a cell is the same as on the whole grid.
struct Lay {
    int nx, ny, nz;
    i64 n;
    bool split;
    int hx;     // nx / 2
    i64 half;   // n / 2 (a slab: the colour stride)
    int zlo, zhi;
    FastDiv by4, by_ny, by_nx, by_half;  // by hx / 4, ny, nx, (nx + 1) / 2
};
Lay make_lay(Dims d);

template <typename T>
struct Coef {
    const T *fx, *fy, *fz;  // low-face coefficients
    const T *invd;          // 1 / sum of the cell's interior face coefficients (FP64 only)
};

#ifdef __CUDACC__
// ---- IEEE-754 conversions and the FP64 reciprocal, with few FP64-pipe instructions --------
// GB300 runs FP64 arithmetic and FP64<->FP32 conversions at a small fraction of its FP32
// rate, so the hot kernels convert by integer operations on the IEEE-754 fields
// (binary64: 1 sign, 11 exponent (bias 1023), 52 fraction bits; binary32: 1, 8 (bias 127), 23).

// FP64 -> FP32 by truncating the IEEE-754 fields with integer operations (the
// binary64 layout: 1 sign, 11 exponent (bias 1023), 52 fraction bits; binary32:
// 1, 8 (bias 127), 23).  Rounds toward zero; results below the FP32 normal range
// become zero, above it infinity; NaN stays NaN.  Keeps the conversion off the
// FP64 pipe, which GB300 runs at a small fraction of the FP32 rate.
__device__ __forceinline__ float d2f_trunc(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(u >> 32);
    const unsigned sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned frac = (unsigned)((u >> 29) & 0x7fffffu);
    if (e == 0x7ff) return __uint_as_float(sign | 0x7f800000u | (frac ? 0x400000u : 0u));
    const int e32 = e - 1023 + 127;
    if (e32 <= 0) return __uint_as_float(sign);
    if (e32 >= 255) return __uint_as_float(sign | 0x7f800000u);
    return __uint_as_float(sign | ((unsigned)e32 << 23) | frac);
}

// FP32 -> FP64 exactly with integer operations (FP32 subnormals become zero)
__device__ __forceinline__ double f2d_exact(float f) {
    const unsigned u = __float_as_uint(f);
    const unsigned sign = u & 0x80000000u;
    const unsigned e = (u >> 23) & 0xffu;
    const unsigned m = u & 0x7fffffu;
    if (e == 0) return __hiloint2double((int)sign, 0);
    const unsigned ed = (e == 0xffu) ? 0x7ffu : (e - 127u + 1023u);
    return __hiloint2double((int)(sign | (ed << 20) | (m >> 3)), (int)(m << 29));
}

// FP64 -> FP32 rounded to nearest, ties to even, with integer operations on the IEEE-754
// fields: the 29 dropped fraction bits decide the rounding; a carry out of the fraction
// increments the exponent (up to infinity).  Results below the FP32 normal range become
// (signed) zero; NaN stays NaN.
__device__ __forceinline__ float d2f_rn(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(u >> 32);
    const unsigned sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned frac = (unsigned)((u >> 29) & 0x7fffffu);
    if (e == 0x7ff) return __uint_as_float(sign | 0x7f800000u | (((u << 12) != 0ull) ? 0x400000u : 0u));
    const int e32 = e - 1023 + 127;
    if (e32 <= 0) return __uint_as_float(sign);
    if (e32 >= 255) return __uint_as_float(sign | 0x7f800000u);
    const unsigned rest = (unsigned)(u & 0x1fffffffull);  // the 29 dropped bits
    const unsigned up = (rest > 0x10000000u || (rest == 0x10000000u && (frac & 1u))) ? 1u : 0u;
    const unsigned mag = ((unsigned)e32 << 23) + frac + up;  // a carry moves into the exponent
    return __uint_as_float(sign | (mag >= 0x7f800000u ? 0x7f800000u : mag));
}

// 1 / x for positive x.  Seed: the FP32 reciprocal (round to nearest) of x rounded to FP32,
// relative error <= 2^-23; then two Newton-Raphson steps y <- y + y (1 - x y) in FP64, each
// squaring the relative error (2^-46, then below FP64 rounding), so the result is within one
// unit in the last place of 1/x.  Outside [2^-100, 2^100] (where the FP32 seed could leave
// the FP32 range) it divides.
__device__ __forceinline__ double recip64(double x) {
    // the range test on the bit pattern (positive doubles order like their bits): no FP64
    // comparison on the FP64 pipe
    const long long xb = __double_as_longlong(x);
    if (!(xb >= 0x39b0000000000000ll && xb <= 0x4630000000000000ll)) return 1.0 / x;
    double y = f2d_exact(__frcp_rn(d2f_rn(x)));
    double e = fma(-x, y, 1.0);
    y = fma(y, e, y);
    e = fma(-x, y, 1.0);
    return fma(y, e, y);
}
#endif

#ifdef __CUDACC__
// Launches.  Between two dependent kernels of a stream GB300 takes 1 to 2.5 us when they are
// launched plainly (the second starts on a 2.05 us tick: 2.07, 4.10, 4.11, 6.15, 8.20 us per
// launch for kernels that run 0.1, 1.1, 2.1, 3.2, 5.3 us), and 0.4-0.5 us with programmatic stream
// serialisation (1.4, 1.6, 2.6, 3.6, 5.6 us) or inside a graph.  So every kernel here is launched with
// that attribute and begins with grid_wait(), before any access to memory: it waits until the
// kernel before it in the stream has completed and its writes are visible.  No kernel but the
// restriction into the coarse levels' cluster triggers its successor early, so two kernels do not
// run side by side (blocks of a successor that only wait would take the place of the predecessor's).  Under a stream capture the launch is plain: the
// graph's own edges cost the same, and forks and joins keep full dependencies.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// lets the next kernel's blocks come in beside this one's, up to their grid_wait(); only where that kernel
// has work to do before it (k_tail)
__device__ __forceinline__ void trigger_next() { asm volatile("griddepcontrol.launch_dependents;"); }

inline bool stream_capturing(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return st != cudaStreamCaptureStatusNone;
}

// a refused launch stays in the runtime's last error, which the entry points check
template <typename... P, typename... A>
inline void run_kernel(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = stream_capturing(s) ? 0 : 1;
    (void)cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}
#endif

// Opts `kernel` into `bytes` of dynamic shared memory (and the largest carveout) on the current
// device, once per device: `done` is the kernel's own mask.  False: refused, and the reason stays
// in the runtime's last error.
bool opt_in_smem(const void *kernel, int bytes, std::atomic<unsigned long long> &done);
// the largest shared-memory carveout as a preference, once per device
bool prefer_smem(const void *kernel, std::atomic<unsigned long long> &done);

// process-wide count of kernel launches (read through mg_kernel_launches)
void count_launch(int k = 1);
unsigned long long launches_total();

// the stream a handle queues its work on, replaced by `s`; returns the previous one (the
// decomposed solver records its cycle, the whole-grid handle's launches included, on a
// private stream)
cudaStream_t swap_handle_stream(mg_handle *h, cudaStream_t s);

// A mixed-precision handle's FP32 level l, for the decomposed mixed cycle (mg_dd.cu), which
// runs the levels from its switch level down on a whole-grid handle: the level's storage layout,
// its right-hand side and iterate arrays, and one FP32 V-cycle of the handle from level l down
// (from x = 0, on that level's b32, into its x32; the handle's options)
Lay handle_lay32(mg_handle *h, int l);
float *handle_b32(mg_handle *h, int l);
float *handle_x32(mg_handle *h, int l);
void handle_vcycle32(mg_handle *h, int l);
// MG_ERR_CUDA, with the handle's message, if a bounded wait of its kernels ran out
int handle_check_waits(mg_handle *h);
// the adaptive inner-cycle count of the mixed outer loop: the first, and the next from the
// contraction of the last outer iteration (k cycles from relres rr_prev to rr)
int handle_first_inner();
int handle_next_inner(double rr_prev, double rr, int k, double rtol);

// NVTX range for the lifetime of the object: a profiler attached to the process (Nsight
// Systems, ncu --nvtx) sees each entry point as one named range; without one the calls do
// nothing (header-only NVTX3, which looks up a tool only when one is injected)
struct NvtxRange {
    explicit NvtxRange(const char *name);
    ~NvtxRange();
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// the most blocks a deterministic reduction over n elements uses (its partials buffer holds
// that many pairs); launchers take min(this, one wave of the kernel)
int reduce_blocks(i64 n);
// streaming multiprocessors of the current device (queried once per device; 152 on GB300)
int device_sms();
constexpr int kReduceThreads = 256;
// blocks of one full wave of `kernel` at `threads` threads per block on the current device
// (resident blocks per SM x SMs; 2^30 if the query fails).  Launchers cache it in a function-
// local static: every device a process uses is of the same model.
int wave_blocks(const void *kernel, int threads);
// min(nb, wave): the grid of a grid-stride reduction that needs nb <= reduce_blocks(n) blocks
int fill_blocks(int nb, int wave);

// Where a reduction's two sums go: device memory (out[0], out[1]), and with `host` also mapped
// pinned host memory, followed by the sequence number `want` in *seq, which the host polls
// (a stream synchronisation after a read-back launch takes about 10 us longer).  `count` (zero at
// rest) lets the reduction's last block add up the partials; without it k_final does.
struct ReduceOut {
    double *out;
    unsigned *count;
    double *host;
    unsigned long long *seq, want;
};
#ifdef __CUDACC__
// the two sums into mapped host memory, then the sequence number the host polls
__device__ __forceinline__ void to_host(const ReduceOut &o) {
    if (!o.host) return;
    volatile double *h = o.host;
    h[0] = o.out[0];
    h[1] = o.out[1];
    __threadfence_system();
    *(volatile unsigned long long *)o.seq = o.want;
}
#endif
// sums into device memory only, by a launch of k_final
inline ReduceOut sums_to(double *out) { return ReduceOut{out, nullptr, nullptr, nullptr, 0}; }

// ---- setup kernels (FP64) -------------------------------------------------------
void launch_density(cudaStream_t s, i64 n, int nfrac, const double *const *frac,
                    const double *rho_phase, double *rho);
// s = 1/rho per cell into `sinv` (validated: err |= 1 on a bad density), then the FP64 low faces
void launch_faces_from_rho(cudaStream_t s, Dims d, const double *rho, double *sinv, double *fx, double *fy,
                           double *fz, unsigned *err, Lay L = Lay{}, float *s32 = nullptr, float2 *s2 = nullptr);
void launch_faces_from_api(cudaStream_t s, Dims d, const double *bx, const double *by,
                           const double *bz, double *fx, double *fy, double *fz, unsigned *err);
void launch_faces_to_api(cudaStream_t s, Dims d, const double *fx, const double *fy,
                         const double *fz, double *bx, double *by, double *bz);
// 1 / sum of the interior face coefficients of each cell, and (diag non-null) the sum itself
void launch_invdiag(cudaStream_t s, Dims d, const double *fx, const double *fy, const double *fz,
                    double *invd64, i64 invd_half, double *diag);
void launch_coarsen(cudaStream_t s, Dims fine, const double *ffx, const double *ffy,
                    const double *ffz, double *cfx, double *cfy, double *cfz, Lay L = Lay{}, float *c32x = nullptr, float *c32y = nullptr,
                    float *c32z = nullptr);
void launch_to_f32(cudaStream_t s, i64 n, const double *src, float *dst);

void launch_csf_faces(cudaStream_t s, Dims d, double h, const double *f, const double *kappa,
                      double *cx, double *cy, double *cz);
void launch_rhs(cudaStream_t s, Dims d, double h, const double *b0, const double *ux, const double *uy,
                const double *uz, const double *fx, const double *fy, const double *fz,
                const double *csfx, const double *csfy, const double *csfz, double sigma,
                double *b);
// ---- dense coarse solve (kernels_coarse.cu) -----------------------------------------
// M (n x n, row-major) = pseudo-inverse of the operator of a grid of n <= MG_MAX_COARSE cells,
// n >= 2 (low faces fx, fy, fz); scratch: coarse_scratch_doubles(d) doubles
size_t coarse_scratch_doubles(Dims d);
void launch_coarse_pinv(cudaStream_t s, Dims d, double ih2, const double *fx, const double *fy, const double *fz,
                        double *M, double *scratch);

// ---- V-cycle kernels --------------------------------------------------------------
// ---- FP32 colour-split level kernels (kernels_split.cu) ----
// half sweep of colour col in place; sinv = 1/rho per cell (beta = (s_L + s_R)/2) when
// non-null, else the low-face arrays; from_zero: the other colour is taken as zero.
// On a slab (L.zlo / L.zhi; see Lay) the V-cycle kernels take its ghost planes as z
// neighbours: split layout with hx % 4 == 0, s-form or face form (fz with its ghost plane
// above: the face to the neighbour above), restriction of red residuals only, trilinear
// prolongation of the red cells from a coarse slab or view (Lc.zlo / Lc.zhi) whose nx is a
// multiple of 8; other cases are not supported on slabs
void launch_half32(cudaStream_t s, Lay L, double h2, const float *sinv, const float *fx, const float *fy,
                   const float *fz, const float *b, float *x, int col, bool from_zero);
// the last red half sweep of the finest level with the outer update fused in: the new red
// values and the black values of the same row positions (x, split, level 0) go straight
// into p = (p - shift) + alpha * x (p natural FP64); x itself is not written.
// Needs a split layout with hx % 4 == 0 (half32_update_ok).
bool half32_update_ok(Lay L);
// p2 non-null: the double-float solution is updated instead of p
void launch_half32_update(cudaStream_t s, Lay L, double h2, const float *sinv, const float *fx, const float *fy,
                          const float *fz, const float *b, const float *x, double *p, float2 *p2, double alpha,
                          double shift);

// ---- fused red-black sweep of the finest level (kernels_fused.cu) ----
// s-form split level with hx % 64 == 0: one sweep, colour c1 first, reading x from X and
// writing both colours to Y (X != Y); from_zero: X is not read (x = 0).  With p non-null the
// second colour's new values and the first colour's go into p = (p - shift) + alpha x (natural
// FP64) instead of Y.  A bounded wait that runs out sets bit 4 of *err.  inject_wait (tests
// only): one block issues no copies for one plane, so that its wait runs out.
bool sweep_fused_ok(Lay L);
void launch_sweep_fused(cudaStream_t s, Lay L, double h2, const float *sinv, const float *b, const float *X,
                        float *Y, int c1, bool from_zero, double *p, double alpha, double shift, unsigned *err,
                        bool inject_wait = false);

// ---- MG_MIXED_DF outer loop (kernels_df.cu): double-float (hi, lo) FP32 pairs ----
void launch_split(cudaStream_t s, i64 n, const double *src, float2 *dst);   // hi = fl32(v), lo = fl32(v - hi)
void launch_join(cudaStream_t s, i64 n, const float2 *src, double *dst);    // v = hi + lo in FP64
// h^2 r = b + sum_f beta_f p_nb - d p_c (b scaled by h^2); out[0] = sum (h^2 r)^2, out[1] = sum p;
// optional r32 = s32 * h^2 r in the split level-0 layout.  Needs even nx.
void launch_resid_df(cudaStream_t s, Dims d, Lay L, const float2 *fx, const float2 *fy, const float2 *fz,
                     const float2 *diag, const float2 *b, const float2 *p, float *r32, float s32,
                     double *partials, ReduceOut ro);
// s-form double-float residual: s2 = 1/rho as FP32 pairs (natural layout), otherwise as launch_resid_df
void launch_resid_dfs(cudaStream_t s, Dims d, Lay L, const float2 *s2, const float2 *b, const float2 *p,
                      float *r32, float s32, double *partials, ReduceOut ro);
// ---- flexible CG (kernels_cg.cu) --------------------------------------------------------
// slots of the device scalar array: r . z of the current and of the previous iteration
// alternate between CG_RZ0 and CG_RZ1
enum { CG_RZ0 = 0, CG_PQ = 1, CG_ALPHA = 2, CG_ZQ = 3, CG_RZ1 = 4, CG_RR = 5, CG_SX = 6, CG_NSLOT = 8 };
void launch_cg_apply32(cudaStream_t s, Lay L, double ih2, const float *sinv, const float *fx, const float *fy,
                       const float *fz, const float *d, float *q, double *partials, double *sc);
void launch_cg_dots32(cudaStream_t s, i64 n, const float *r, const float *z, const float *q, double *partials,
                      double *sc, int rz_slot);
void launch_cg_dir32(cudaStream_t s, i64 n, const float *z, float *d, const double *sc, bool first, int rz_prev);
void launch_cg_update32(cudaStream_t s, i64 n, float *x, float *r, const float *d, const float *q, double *sc,
                        int rz_cur);
void launch_cg_apply64(cudaStream_t s, Dims d, double ih2, const double *fx, const double *fy, const double *fz,
                       const double *dg, const double *dv, double *q, double *partials, double *sc);
void launch_cg_dots64(cudaStream_t s, i64 n, const double *r, const double *z, const double *q, double *partials,
                      double *sc, int rz_slot);
void launch_cg_dir64(cudaStream_t s, i64 n, const double *z, double *d, const double *sc, bool first, int rz_prev);
void launch_cg_update64(cudaStream_t s, i64 n, double *x, double *r, const double *d, const double *q, double *sc,
                        int rz_cur, double *partials);

void launch_update_df(cudaStream_t s, Dims d, Lay L, float2 *p, const float *e32, double alpha, double shift);
// r = b - A x (or r = A x when apply_only)
void launch_residual32(cudaStream_t s, Lay L, double ih2, const float *sinv, const float *fx, const float *fy,
                       const float *fz, const float *b, const float *x, float *r, bool apply_only);
// bc = mean of the 8 children's residuals (red_only: black children count as 0); tail: launch_tail
// follows on the stream
void launch_resid_restrict32(cudaStream_t s, Lay L, Lay Lc, double ih2, const float *sinv, const float *fx,
                             const float *fy, const float *fz, const float *b, const float *x, float *bc,
                             bool red_only, bool tail = false);
// x += P ec on the cells of colour only_col (0 red, 1 black) or all cells (-1)
void launch_prolong32(cudaStream_t s, Lay L, Lay Lc, const float *ec, float *x, int kind, int only_col);
void launch_coarse_matvec32(cudaStream_t s, Lay L, const double *pinv, const float *r, float *e);
void launch_pack32(cudaStream_t s, Lay L, const float *nat, float *st);
void launch_unpack32(cudaStream_t s, Lay L, const float *st, float *nat);
void launch_pack64to32(cudaStream_t s, Lay L, const double *nat, float *st);
// s (FP64, natural) -> FP32 in the level layout, and optionally FP32 pairs (natural)
void launch_pack_inv_rho(cudaStream_t s, Lay L, const double *sinv, float *st, float2 *s2);
// FP64 red-black half sweep of one colour, in place
// FP64 red-only residual + restriction in diagonal form (dg = sum of the cell's face betas)
void launch_rr_red_diag64(cudaStream_t s, Dims fine, double h2, Coef<double> c, const double *dg,
                          const double *b, const double *x, double *bc, bool b_split = false);
// b_split: h2 b colour by colour as in Lay (only with invd_split, the reciprocal diagonal likewise); from_zero: the red
// half sweep of x = 0, which need not have been written (b not split)
void launch_rbgs_half64(cudaStream_t s, Dims d, double h2, Coef<double> c, const double *b, double *p, int colour,
                        bool b_split = false, bool invd_split = false, bool from_zero = false);
template <typename T>
void launch_apply(cudaStream_t s, Dims d, double ih2, Coef<T> c, const T *x, T *y);
template <typename T>
void launch_residual(cudaStream_t s, Dims d, double ih2, Coef<T> c, const T *b, const T *x, T *r);
// bc = mean of the 8 children's residuals (red_only: black children count as 0)
template <typename T>
void launch_resid_restrict(cudaStream_t s, Dims fine, double ih2, Coef<T> c, const T *b,
                           const T *x, T *bc, bool red_only);
// e += P ec on the cells of colour only_col (0 red, 1 black) or all cells (-1)
template <typename T>
void launch_prolong(cudaStream_t s, Dims coarse, const T *ec, T *e, int kind, int only_col);
template <typename T>
void launch_coarse_matvec(cudaStream_t s, int nc, const double *pinv, const T *r, T *e);

// ---- the coarse levels of a V-cycle in one cluster launch (kernels_tail.cu) -------------
constexpr int kTailLevels = 6;
constexpr int kTailCells32 = 2, kTailCells64 = 1;  // cells of a colour per thread
constexpr int kTailMaxSmem = 225 * 1024, kTailMinSmem = 118 * 1024;  // per CTA, dynamic
enum { kTailAll = 0, kTailDown = 1, kTailUp = 2 };
struct TailLevel {
    int nx, ny, nz;
    i64 half;              // colour stride of the FP32 arrays in memory (Lay.half)
    double h2, ih2;
    const void *fx, *fy, *fz, *invd, *diag;  // the level's arrays (FP32 in its Lay; FP64 natural, invd colour by colour)
    void *x, *b;
    // set by tail_layout
    int hx, q4, nit, rs;   // nx / 2, row quads and cells of a colour per CTA, row stride of x
    unsigned magic_nx, magic_hx;
    int off_x, off_b, off_c, off_w, off_q;
    int img_bytes;         // one CTA's contexts and tables, from off_c
    i64 img;               // offset of the level's images in TailArgs::img
};
// nl smoothed levels and the dense coarse solve of nc cells below them
struct TailArgs {
    int nl, nc, pre, post;
    TailLevel lv[kTailLevels];
    const double *pinv;
    void *bc, *xc;         // the coarsest level's b and x in memory (split runs), colour stride half_c
    i64 half_c;
    void *img;             // img_total bytes, written by launch_tail_prepare
    i64 img_total;
    unsigned *err;         // |= 8 when a wait for ghosts ran out
    int ncta, smem, off_rc, off_ec, off_cw;
};
// lays the levels (nx, ny, nz, nc set) out over ncta CTAs; false if they do not fit
bool tail_layout(TailArgs &a, bool fp64, int ncta);
// the cells' coefficients and addresses as the launches below read them, from the levels' arrays
void launch_tail_prepare(cudaStream_t s, const TailArgs &a, bool fp64);
// one V-cycle of those levels from x = 0 on lv[0].b into lv[0].x (mode kTailAll), or its descent
// or ascent alone.  pre, post >= 1, trilinear prolongation, every level's nx, ny, nz even.
void launch_tail(cudaStream_t s, const TailArgs &a, bool fp64, int mode);
// where the first CTA's image keeps the bytes it expects of its neighbours per colour of the first level
unsigned *tail_ghost_bytes(const TailArgs &a);

// ---- reductions, fine-level FP64 passes, adjoint -----------------------------------
// partials: reduce_blocks(n) x 2 doubles; out: 2 doubles (deterministic order)
// scalars for the host: a one-thread-per-value kernel stores n (<= 32) doubles, or one
// unsigned, into mapped pinned host memory (device-side address of a cudaHostAllocMapped
// buffer), so that the host's wait for them never queues behind bulk copies that other
// streams run on the copy engines
void launch_readback(cudaStream_t s, const double *src, double *dst_mapped, int n);
void launch_readback_u32(cudaStream_t s, const unsigned *src, unsigned *dst_mapped);
// *p += v, one thread (test faults)
void launch_add_u32(cudaStream_t s, unsigned *p, int v);
// out[0] = sum x, out[1] = sum x^2 (0 unless `squares`)
template <typename T>
void launch_sum_sumsq(cudaStream_t s, i64 n, const T *x, double *partials, ReduceOut ro, bool squares);
// b64 = (b - sum[0]/n) * scale, with the sum of squares of b64 into out[0]
void launch_sub_mean(cudaStream_t s, i64 n, const double *b, const double *sum, double scale, double *b64,
                     double *partials, ReduceOut ro, const Dims *split = nullptr);
// fine FP64 residual in diagonal form, h^2 r = h^2 b - (diag p_c - sum_f beta_f p_nb):
// out[0] = sum (h^2 r)^2, out[1] = sum p; optional r32 = s32 * h^2 r in the level-0 layout L.
// On a slab of a decomposed grid (d.zlo or d.zhi, even nx; p with its ghost planes beside the
// own ones, fz with the face to the ghost above) the ghost planes count as interior neighbours,
// and r32 is stored in the slab's layout L (L.half the colour stride)
void launch_fine_resid2(cudaStream_t s, Dims d, Lay L, double h2, const double *fx, const double *fy,
                        const double *fz, const double *diag, const double *b, bool b_scaled, const double *p,
                        float *r32, float s32, double *partials, ReduceOut ro, bool b_split = false);
// r32 = (float)(ih2 scale) * trunc_fp32(b): the scaled FP32 residual of p = 0, as the outer
// residual kernels would write it (b = h^2 b~ in the mixed modes)
void launch_zero_resid32(cudaStream_t s, Dims d, Lay L, const double *b, double scale32, float *r32);
// p = p - shift + alpha * e32 (e32 in the level-0 FP32 layout L; shift a host scalar)
void launch_update(cudaStream_t s, Dims d, Lay L, double *p, const float *e32, double alpha, double shift);
void launch_add_const(cudaStream_t s, i64 n, double *p, double c);
// p -= sum[0] / n (sum on the device)
void launch_sub_sum(cudaStream_t s, i64 n, double *p, const double *sum);
// zeroes `bytes` bytes (a multiple of 4) at p (4-byte aligned): a kernel, because a memset between two
// kernels costs both of them the 2 us gap that run_kernel avoids
void launch_zero(cudaStream_t s, void *p, size_t bytes);
void launch_adjoint_grad(cudaStream_t s, Dims d, double h, const double *lam, const double *p,
                         const double *fx, const double *fy, const double *fz, const double *csfx,
                         const double *csfy, const double *csfz, double sigma, float *gx,
                         float *gy, float *gz, double *partials, double *out);

// ---- either side of the solve (kernels_project.cu) --------------------------------------
// o = u + beta (G p + sigma csf) on the interior faces, o = u on the walls (csfx NULL: no
// surface term); o may be u (in place; the walls are then not rewritten)
void launch_project(cudaStream_t s, Dims d, double h, const double *p, const double *fx, const double *fy,
                    const double *fz, const double *csfx, const double *csfy, const double *csfz, double sigma,
                    const double *ux, const double *uy, const double *uz, double *ox, double *oy, double *oz);
// dL/drho from FP32 face gradients, and dL/df_q = dL/drho (rho_q - rho_last) into dfrac[q]
void launch_density_grads(cudaStream_t s, Dims d, const double *rho, const float *gx, const float *gy,
                          const float *gz, double *drho, int nfrac, const double *rho_phase,
                          double *const *dfrac);

}  // namespace mg
