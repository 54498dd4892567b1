// hom_internal.h -- shared declarations of the library's kernels.
//
// Data layout in device memory
//   real field     : 6 x V, component-major (Mandel components), C order voxels
//   half spectrum  : n1 x n2 x h x 6 complex, h = n3/2 + 1, component fastest
//                    (the six components of one frequency are adjacent, which
//                    the projector and the n1 pass read together)
// The MINRES vectors live in the half-spectrum space: MINRES runs on
//   A^(v) = G F C F^-1 G v,
// the operator of eq. (linearOp) conjugated by the DFT, with the projector
// applied on the input as well as on the output, under the Parseval inner
// product <a,b> = sum_k w(k3) Re(conj(a_k) b_k) with w = 1 on the self-
// conjugate planes k3 = 0 and k3 = n3/2 (even n3) and 2 elsewhere.  On
// compatible fields this is the same iteration as MINRES on A(e) in real space.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "hom_fft.cuh"
#include "hom_tma.cuh"

namespace hom {

// Scalars of one MINRES solve, resident in device memory.  Written only by
// the single-CTA scalar kernels; read by the field kernels.  FP64 always.
struct MinresState {
    int done;          // no further operator / Krylov work (first field: the
                       // pass kernels read it through any solver's state)
    int done_update;   // set with done on a NaN: keep the last finite iterate (no flush)
    int k;             // iterations done
    int max_it;
    int status;        // 0 ok, 1 max_it, -5 NaN
    int pad;
    double beta1;      // ||b||
    double beta;       // beta_k = ||u_k||: the stored Lanczos vector u_k = beta_k v_k
    double beta_prev;  // beta_{k-1} (0 before the second step: no v_0 term)
    double alpha;      // alpha_k
    double c, s;       // previous Givens rotation
    double dbar;       // delta-bar_{k+1}
    double eps;        // epsilon_{k+1}
    double phibar;     // phi-bar_k
    double tol;
    // coefficients of the w / x update of the last finished iteration k,
    // applied one iteration later: w_k = (u_k u_inv_beta - u_delta w_{k-1}
    // - u_eps w_{k-2}) u_inv_gamma, x += u_tau w_k
    double u_delta, u_eps, u_inv_gamma, u_tau, u_inv_beta;
    // tau_{k-1}, tau_{k-2}: the fused MINRES step adds tau_j w_j to x for
    // three j at once, every third iteration (x is read and written a third
    // as often)
    double u_tau1, u_tau2;
    double est;        // phibar_k / beta_1
    int bodies;        // captured bodies run by the device-side loop
    int max_bodies;    // hard cap of that loop
    // FP32 fields under stress control (dc != 0): the vectors' values at xi = 0,
    // the macroscopic strain the load drives, carried in FP64 beside their FP32
    // entries, with A u at xi = 0 from the n3 pass's FP64 stress sums.  One FP32
    // rounding of them is a uniform strain, which no average over voxels takes
    // out: without this the stresses of an uniaxial solve after 50 steps are
    // 1.4 to 2.7e-6 off an FP64 solve's, with it 1.3 to 1.5e-6 (a numpy
    // restatement, 48^3 octet).  Six real components each (Mandel).
    int dc;
    double dc_tau[6], dc_u[6], dc_um[6], dc_un[6], dc_w1[6], dc_w2[6], dc_x[6];
    double dc_keep[6];   // x there as of the FP32 vectors' last update of x
};

// the fused step updates x when the iterations done (the state's k) are a multiple of 3
__host__ __device__ constexpr bool minres_xstep(int k) { return k > 0 && k % 3 == 0; }

// the step's w and x at xi = 0, and u_{k+1} in u_k's place (one thread; ib =
// 1 / beta_k, ig = 1 / gamma; the values are loaded together, one memory
// latency and not six)
__device__ __forceinline__ void dc_step(MinresState *st, double ib, double delta, double eps, double ig, double tau) {
    double u[6], un[6], w1[6], w2[6], x[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        u[c] = st->dc_u[c];
        un[c] = st->dc_un[c];
        w1[c] = st->dc_w1[c];
        w2[c] = st->dc_w2[c];
        x[c] = st->dc_x[c];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const double w = (u[c] * ib - delta * w1[c] - eps * w2[c]) * ig;
        st->dc_w2[c] = w1[c];
        st->dc_w1[c] = w;
        st->dc_x[c] = x[c] + tau * w;
        st->dc_um[c] = u[c];
        st->dc_u[c] = un[c];
    }
}
// u_{k+1} at xi = 0 (one thread of the fused n1 pass); q: its three values
template <typename R> __device__ __forceinline__ void dc_lanczos(MinresState *st, int mask, cpx<R> *q) {
    const double ib = 1.0 / st->beta, cu = -st->alpha * ib;
    const double cv = st->beta_prev > 0.0 ? -st->beta / st->beta_prev : 0.0;
    double v[6];
#pragma unroll
    for (int c = 0; c < 6; ++c)
        v[c] = (mask >> c) & 1 ? st->dc_tau[c] * ib + cu * st->dc_u[c] + cv * st->dc_um[c] : 0.0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        st->dc_un[c] = v[c];
        if (c & 1) q[c / 2].y = (R)v[c];
        else q[c / 2].x = (R)v[c];
    }
}

// alpha_k = <v_k, A v_k> = <u_k, A u_k> / beta_k^2 from sum = <u_k, A u_k> / scale
__device__ __forceinline__ void alpha_step(MinresState *st, double sum, double scale) {
    if (st->done) return;
    st->alpha = scale * sum / (st->beta * st->beta);
}

// MINRES step k (one thread): apply the previous Givens rotation to the new
// column of the Lanczos tridiagonal, form the next rotation and the
// coefficients of the w_k / x_k update (applied by the next step's kernel,
// or by the flush after the loop); stop when phibar_k / beta_1 <= tol,
// beta_{k+1} = 0, or k reaches max_it.  bn2 = ||u_{k+1}||^2.
__device__ __forceinline__ void givens_step(MinresState *st, double bn2) {
    if (st->done) return;
    // everything the step reads, before it writes: one memory latency and not one
    // after each group of stores
    const double alpha = st->alpha, c = st->c, s = st->s, dbar = st->dbar, eps = st->eps, beta = st->beta;
    const double phibar0 = st->phibar, beta1 = st->beta1, tol = st->tol, u_tau = st->u_tau, u_tau1 = st->u_tau1;
    const int k = st->k, max_it = st->max_it, dc = st->dc;
    const double beta_next = sqrt(bn2 > 0 ? bn2 : 0.0);
    const double delta = c * dbar + s * alpha;
    const double gbar = s * dbar - c * alpha;
    const double eps_next = s * beta_next;
    const double dbar_next = -c * beta_next;
    double gamma = hypot(gbar, beta_next);
    if (gamma == 0.0) gamma = 1e-300;
    const double cn = gbar / gamma, sn = beta_next / gamma;
    const double tau = cn * phibar0;
    const double phibar = sn * phibar0;
    const double inv_gamma = 1.0 / gamma, inv_beta = 1.0 / beta, est = phibar / beta1;
    const bool finite = isfinite(alpha) && isfinite(beta_next) && isfinite(phibar);
    if (dc) {
        // this step's n1 pass took x to the iterations done so far; a breakdown
        // keeps the iterate of the last such pass, at xi = 0 as everywhere else
        if (minres_xstep(k))
            for (int i = 0; i < 6; ++i) st->dc_keep[i] = st->dc_x[i];
        if (finite) dc_step(st, inv_beta, delta, eps, inv_gamma, tau);
        else
            for (int i = 0; i < 6; ++i) st->dc_x[i] = st->dc_keep[i];
    }
    st->u_delta = delta;
    st->u_eps = eps;            // epsilon_k multiplies w_{k-2}
    st->u_inv_gamma = inv_gamma;
    st->u_tau2 = u_tau1;
    st->u_tau1 = u_tau;
    st->u_tau = tau;
    st->u_inv_beta = inv_beta;   // v_k = u_k / beta_k in the lagged update
    st->c = cn;
    st->s = sn;
    st->dbar = dbar_next;
    st->eps = eps_next;
    st->phibar = phibar;
    st->beta_prev = beta;
    st->beta = beta_next;
    st->k = k + 1;
    st->est = est;
    if (!finite) {
        st->status = -5;
        st->done = 1;
        st->done_update = 1;        // keep the last finite iterate
        return;
    }
    if (est <= tol || beta_next == 0.0) {
        st->done = 1;               // the flush still applies this step's update
    } else if (k + 1 >= max_it) {
        st->status = 1;
        st->done = 1;
    }
}

// Scalars of one preconditioned CG solve (MoDBFFT, section 2.2); same
// leading flags as MinresState.
struct CgState {
    int done, done_update, k, max_it, status, pad;
    double rho;        // <r, M r>
    double rr0;        // ||r_0||^2
    double rr;         // ||r_k||^2
    double a, b;       // step length and direction update of this iteration
    double tol;
    double est;        // ||r_k|| / ||r_0||
    double sc;         // about 1 / rms(r_0), a power of two (MoDBFFT)
};

// Kernel-side description of one cell for one precision.
struct Geometry {
    int n1, n2, n3, h;      // h = n3/2 + 1
    long long V, S;         // voxels, half-spectrum points per component
    AxisPlan ax[3];
    int line[3];            // FP64: length of the axis if the line engine runs it, else 0
    int ord[3];             // FP64: the same for ordered_fft
    const double2 *Dc[3], *Mc[3];   // FP64: difference symbol and averaging factor, complex (gamma_at_c)
    const double2 *etab = nullptr;  // unit vectors of every frequency, or null: formed in the pass
    const void *D[3];       // per axis: difference symbol without its phase (real, length n_p; see gamma_e)
    const void *M[3];       // per axis: averaging factor without its phase (real, length n_p)
    // launch shapes: rows per CTA of the n3 pass, columns per CTA of the n2
    // and n1 passes, threads per CTA, dynamic shared memory, and whether the
    // axis uses the compile-time register FFT (its length, or 0)
    int rows3, tile2, tile1;
    int threads3, threads2, threads1;
    size_t smem3, smem2, smem1;
    int fast[3];
    int nc;                 // complex components per frequency in the spectrum (6, or 10 for MoDBFFT)
    // load cases stacked along k1 in one launch of the MINRES kernels (work
    // spectrum nb x n1 x n2 x h x nc, Krylov vectors nb blocks of kvec, one
    // MinresState per case); 1 everywhere else
    int nb = 1;
    // nonzero: the MINRES passes launch with programmatic stream serialization
    // (set for the stacked graph's body; the kernels wait on their
    // predecessor with griddepcontrol before touching memory)
    int pdl = 0;
    int mask0;              // stress-controlled Mandel components (bit c): the projector keeps them at xi = 0
    // persistent TMA-staged passes (FP32): tma enables the unfused n1 pass
    // (register-FFT n1 and n2 in [64, 512]); persistent grid sizes, shared
    // memory, host-side cache of tensor maps (never dereferenced on the
    // device) and the device word a pass sets when a bounded wait gives up
    int tma;
    // fused MINRES chain: complex elements of one Krylov vector, three
    // components a frequency (gamma_to_q) in n1-tile order: tiles of tile1l
    // (k2,k3) columns, each krylov_tile(n1, tile1l) values, one plane n1 x
    // tile1l per component
    long long kvec;
    // register-resident n3 pass (k_x3r: FP32, n3 = 256) for
    // spectrum-to-spectrum applications
    int x3r;
    int x3l = 0;            // the persistent n3 pass of X3Plan instead (see x3_line_kernel)
    int grid2_tma, grid1_tma, grid1d_tma;
    int grid1l_tma = 0;     // persistent grid of the fused MINRES n1 pass (0: plain-load form)
    size_t smem2_tma, smem1_tma, smem1d_tma;
    // TMA-staged n2 pass and fused n1 pass, the line engine's lengths (the n2 pass
    // but 375 and 405, the fused pass but 270, 300, 324, 375, 405, 450, 486 and 500:
    // beyond 256 a tile moves in boxes, and those lengths have no division whose
    // boxes start on 128-byte boundaries): x2t enables the n2 pass (threads2t
    // threads); the fused n1 pass has grp1l transform threads (0: plain-load form),
    // tiles of tile1l columns and stage1l bytes per shared-memory stage; rows per
    // TMA box
    int x2t = 0, threads2t = 0, grp1l = 0;
    int tile1l;             // columns of a Krylov-vector tile (tile1 where the plain-load form runs)
    size_t stage1l = 0;
    int box2 = 0, box1 = 0, box1l = 0;
    int grid3r = 0;         // persistent grid of the register n3 pass
    int x2_stages = 2;      // TMA ring stages of the persistent n2 pass
    int x1_l2pf = 1;        // fused n1 pass: L2 prefetch of each tile's u_k, u_{k-1} blocks
    size_t smem1l_tma = 0;  // fused MINRES n1 pass: work-tile stages + lagged-update ring
    int x1_lag_stages = 0;  // stages of that ring (kX1LagChunk bytes of each of 4 operands)
    void *tma_cache;
    int *err;
};

// register-resident n3 pass (k_x3r, n3 = 256: the length at which it is faster
// than the persistent pass of X3Plan): lanes of a row, rows per warp (32 /
// lanes), and per warp the prefetch buffer of a row group (its rows' half
// spectra, then phi) and one transpose slab (Q x (P + 1) complex values,
// N = P Q) per row; four warps per CTA
__host__ __device__ constexpr bool x3r_length(int n) { return n == 256; }
__host__ __device__ constexpr int x3r_row_lanes(int) { return 16; }
__host__ __device__ constexpr int x3r_rows_per_warp(int n) { return 32 / x3r_row_lanes(n); }
__host__ __device__ constexpr size_t x3r_in_bytes(int n) {
    return (size_t)x3r_rows_per_warp(n) * (n / 2 + 1) * 6 * sizeof(float2);
}
__host__ __device__ constexpr size_t x3r_phi_bytes(int n) { return (size_t)x3r_rows_per_warp(n) * n * sizeof(float); }
__host__ __device__ constexpr size_t x3r_slab_elems(int n) {
    return (size_t)(n / x3r_row_lanes(n)) * (x3r_row_lanes(n) + 1);
}
__host__ __device__ constexpr size_t x3r_warp_bytes(int n) {
    return x3r_in_bytes(n) + x3r_phi_bytes(n) + (size_t)x3r_rows_per_warp(n) * x3r_slab_elems(n) * sizeof(float2);
}
constexpr int kX3rWarps = 4;
__host__ __device__ constexpr size_t x3r_smem(int n) { return kX3rWarps * x3r_warp_bytes(n); }

// A kernel launch, with programmatic stream serialization when pdl != 0.
template <typename... KArgs, typename... Args>
inline void launch_k(int pdl, void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     Args... args) {
    if (!pdl) {
        k<<<grid, block, smem, st>>>(args...);
        return;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k, args...);
}

// tensor-map kinds of the TMA passes
enum TmaKind { TMA_X2 = 0, TMA_X1 = 1, TMA_X1L = 2 };
// Host: the cached tensor map of `ptr` (a half spectrum of this geometry) for
// the given pass; nullptr if the driver entry point is unavailable.
const CUtensorMap *tma_map(const Geometry &g, const void *ptr, int kind, int elem_units);
void *tma_cache_new();
bool tma_available();
void tma_cache_free(void *cache);

// n3 pass (x3): input, middle and output stages
enum X3In { X3_IN_SPEC = 0, X3_IN_REAL = 1, X3_IN_MACRO = 2 };
enum X3Mid { X3_MID_NONE = 0, X3_MID_MATERIAL = 1,
             X3_MID_MODB = 2 };   // 10 components: tau = phi C_m eps (0-5), chi_v g (6-8), 0 (9)
enum X3Out { X3_OUT_SPEC = 0, X3_OUT_REAL = 1 };
// n1 pass (x1) flags
// (X1_BACK: the inverse transform after the projection, FP32 plain-load form)
enum X1Flags { X1_FWD = 1, X1_GAMMA_IN = 2, X1_GAMMA_OUT = 4, X1_DOT = 8, X1_BACK = 16 };

constexpr int kEwBlocks = 152 * 8;   // grid of the element-wise Krylov kernels
constexpr int kNbMax = 8;            // load cases of one stacked MINRES batch
// persistent fused n1 pass: the most threads its transform group may have, and
// its lagged-update ring
constexpr int kX1Group = 192;
constexpr int kX1LagChunk = 2048;      // bytes of one operand per ring stage
constexpr int kX1LagMaxStages = 3;
constexpr int kX2MaxStages = 4;        // TMA ring of the persistent n2 pass
constexpr int kEwThreads = 256;

struct Mac6 { double v[6]; };

// complex values of a Krylov tile of t columns: three planes, padded to 16 bytes
// for the bulk copies
__host__ __device__ constexpr int krylov_tile(int n1, int t) { return (3 * n1 * t + 1) / 2 * 2; }

// The MINRES scalar steps folded into the pass that produces their partial
// sums: every CTA of a group counts itself on a counter after writing its
// partial, and the last one reduces the group's partials (fixed order) and
// applies the step to the FP64 state, then resets the counter for the next
// launch.  cnt == nullptr: no folding (a separate scalar kernel does the step).
// Counters: cnt[c] the n3 pass's CTAs of case c, cnt[kNbMax + c] the plain
// n1 pass's CTAs of case c, cnt[2 kNbMax] the persistent n1 pass's CTAs.
struct Fold {
    int *cnt;
    MinresState *st;     // the states (one per case)
    double scale;        // alpha: the partials sum to <u, A^ u> / scale
};
constexpr int kFoldCounters = 2 * kNbMax + 1;

// Kernels of the line engine (FP32) for one length; nullptr where it has none.
using X2LineFn = void (*)(Geometry, CUtensorMap, int, const MinresState *);
using X1lLineFn = void (*)(Geometry, CUtensorMap, const float2 *, const float2 *, float2 *, const float2 *, float2 *,
                           float2 *, const MinresState *, double *, Fold);
X2LineFn x2_line_kernel(int n, int inverse);
X1lLineFn x1l_line_kernel(int n);
// FP64 passes at one line length (hom_f64_*.cu; null members: no such length)
using F64X1Fn = void (*)(Geometry, int, const double2 *, double2 *, const double2 *, double *, const MinresState *);
using F64X1lFn = void (*)(Geometry, double2 *, const double2 *, const double2 *, double2 *, const double2 *, double2 *,
                          double2 *, const MinresState *, double *, Fold);
using F64X2Fn = void (*)(Geometry, double2 *, const MinresState *);
using F64X3Fn = void (*)(Geometry, int, const void *, int, double, double, Mac6, double, int, void *, const double *,
                         const MinresState *, double *, Fold, double *);
int f64_line_tpl(int n);   // threads of a line (0: the runtime engine)
F64X1Fn f64_x1_kernel(int n);
F64X1lFn f64_x1l_kernel(int n);
F64X2Fn f64_x2_kernel(int n, int inverse);
F64X3Fn f64_x3_kernel(int n, int pairs);   // pairs of components: 3 or 5
// the same on ordered_fft (6 components)
F64X1Fn f64_ord_x1_kernel(int n);
F64X2Fn f64_ord_x2_kernel(int n, int inverse);
F64X3Fn f64_ord_x3_kernel(int n);

// persistent n3 pass of a length (fn_sums: with the stress sums), with its threads,
// rows per tile and shared memory (fn null: none)
struct X3Line {
    using Fn = void (*)(Geometry, const float2 *, float2 *, int, float, float, const float *, const MinresState *,
                        double *, Fold, double *);
    Fn fn = nullptr, fn_sums = nullptr;
    int threads = 0, rows = 0;
    size_t smem = 0;
};
X3Line x3_line_kernel(int n);
// shared-memory limit and carve-out of one of them
void line_kernel_attr(const void *kernel, int optin);
// rows of a TMA box for tiles of n rows of rowb bytes: the most that divide n,
// fit a box dimension (256) and keep every box on a 128-byte boundary of
// shared memory (0: none)
constexpr int tma_box_rows(int n, int rowb) {
    for (int k = (n + 255) / 256; k <= n; ++k)
        if (n % k == 0 && (k == 1 || (n / k) * rowb % 128 == 0)) return n / k;
    return 0;
}
// columns of a tile of the TMA-staged fused n1 pass (FP32, six components): as
// many as its transform group has threads for and its boxes allow (0: none)
constexpr int x1l_cols(int n, int tpl) {
    int t = kX1Group / (6 * tpl);
    for (t = t > 16 ? 16 : t; t > 0; --t)
        if (tma_box_rows(n, 48 * t)) break;
    return t;
}
// its transform threads, lagged-update threads and both.  One lagged warp
// beside small groups, so that four CTAs fit at 80 registers (40 against 44 us
// at 108^3), two beside full ones, which three CTAs leave the registers for
// (398 against 423 us at 256^3).
constexpr int x1l_group(int n, int tpl) { return (6 * x1l_cols(n, tpl) * tpl + 31) / 32 * 32; }
constexpr int x1l_lag_threads(int grp) { return grp > 160 ? 64 : 32; }
constexpr int x1l_threads(int n, int tpl) { return x1l_group(n, tpl) + x1l_lag_threads(x1l_group(n, tpl)); }

template <typename R> struct Launch {
    // n3 pass: C2R (SPEC in) or real / macro input, optional material law
    // tau = phi C_m e, R2C (SPEC out) or real output; scale applied to the
    // real-space values (1/V for SPEC in is included automatically).
    // epart (6-component spectra only): per-CTA sums of the strain energy
    // e : C : e of the scaled real-space input (x3_grid(g) values).
    // fold: the alpha step folded into the pass (see Fold in hom_passes.cuh)
    // tsum (with the material law): per-CTA partial sums over the voxels of
    // the six stress components it forms, tsum[(c * nb + case) * blocks + block],
    // blocks a case's partials (x3_epart_grid(g) from spectrum to spectrum)
    static void x3(const Geometry &g, cudaStream_t st, int in_mode, const void *in, int mid, double lam, double mu,
                   const double *macro_mandel, double scale, int out_mode, void *out, const R *phi,
                   const MinresState *state, double *epart = nullptr, Fold fold = Fold{}, double *tsum = nullptr);
    // n2 pass, in place on the half spectrum
    static void x2(const Geometry &g, cudaStream_t st, int inverse, cpx<R> *spec, const MinresState *state);
    // n1 pass: in -> out (may alias), optional projector before / after, and
    // the weighted partial sum <dotv, out> per CTA
    static void x1(const Geometry &g, cudaStream_t st, int flags, const cpx<R> *in, cpx<R> *out,
                   const cpx<R> *dotv, double *partials, const MinresState *state);
    // the elastoplastic increments' (FP64): the unit frequency vectors (Geometry::
    // etab), and x1's weighted partial sum <dotv, z> alone
    static void gamma_table(const Geometry &g, cudaStream_t st, double2 *out);
    static void x1_dot(const Geometry &g, cudaStream_t st, const cpx<R> *z, const cpx<R> *dotv, double *partials,
                       const MinresState *state);
    // MoDBFFT: forward n1 pass of the 10-component spectrum in10 with the
    // contraction to 3 components fused (out3 = tau xi + g, eq. modbfftfop;
    // with dot3, the weighted <dot3, out3> partials).  Returns the number of
    // partials written, or 0 without launching where the fused form does not
    // apply (not the TMA-staged FP32 pass, or more partials than max_partials).
    static int x1_modb_contract(const Geometry &g, cudaStream_t st, const cpx<R> *in10, cpx<R> *out3,
                                const cpx<R> *dot3, double *partials, int max_partials, const MinresState *state);
    // MoDBFFT: the expansion of u3 to 10 components with the penalty alpha
    // (modb_expand) and the inverse n1 pass as one TMA-staged FP32 pass into
    // out10.  Returns false without launching where the fused form does not
    // apply (not the TMA-staged FP32 pass).
    static bool x1_modb_expand(const Geometry &g, cudaStream_t st, double alpha, const cpx<R> *u3, cpx<R> *out10,
                               const MinresState *state);
    // MINRES step k on unnormalised Lanczos vectors u_j = beta_j v_j, p = A u_k:
    //   um <- (p - alpha u_k - beta_k^2/beta_{k-1} um) / beta_k   (= u_{k+1}),
    //   weighted partial ||u_{k+1}||^2, and the lagged update of step k-1
    //   (k > 1): wb <- (um_old/beta_{k-1} - delta wa - eps wb) / gamma,
    //   x += tau wb.  wa = w_{k-2}, wb = w_{k-3} on entry.
    static void lanczos_update(const Geometry &g, cudaStream_t st, const cpx<R> *p, const cpx<R> *uk, cpx<R> *um,
                               const cpx<R> *wa, cpx<R> *wb, cpx<R> *x, const MinresState *state, double *partials);
    // fused n1 pass of a MINRES step (see k_x1_lanczos): spec holds the
    // forward n3 / n2 transforms of C e_k on entry and the inverse n1
    // transform of G u_{k+1} on exit; u_{k+1} is written to un (a third
    // buffer, neither uk nor um); wb, x as for lanczos_update;
    // x1_lanczos_grid(g) partials of ||u_{k+1}||^2
    // (fold: the Givens step folded into the pass)
    static void x1_lanczos(const Geometry &g, cudaStream_t st, cpx<R> *spec, const cpx<R> *uk, const cpx<R> *um,
                           cpx<R> *un, const cpx<R> *wa, cpx<R> *wb, cpx<R> *x, const MinresState *state,
                           double *partials, Fold fold = Fold{});
    static int x1_lanczos_grid(const Geometry &g);
    // half spectrum in standard order <-> Krylov vector (its padding is left
    // untouched); to_krylov returns the number of partials of ||q||^2
    static int to_krylov(const Geometry &g, cudaStream_t st, const cpx<R> *in, cpx<R> *out, double *partials);
    // (state: its FP64 values at xi = 0 are taken where it has them)
    static void from_krylov(const Geometry &g, cudaStream_t st, const cpx<R> *in, cpx<R> *out, const MinresState *state);
    // the lagged update of the last step K after the loop; u_K sits in
    // buffer K mod 3 of (ua, ub, uc), or without uc (two Lanczos buffers) in
    // ub for odd K, in ua for even K; w_{K-1} in wd for even K, wc for odd K
    static void minres_flush(const Geometry &g, cudaStream_t st, const cpx<R> *ua, const cpx<R> *ub,
                             const cpx<R> *uc, cpx<R> *wc, cpx<R> *wd, cpx<R> *x, MinresState *state, long long n);
    // Parseval partials of <phi, (G x^)_c>, c = 0..5 (see k_phi_dot); returns
    // the number of blocks (partials[c * nb + block])
    static int phi_dot(const Geometry &g, cudaStream_t st, const cpx<R> *x, const cpx<R> *phihat, double *partials);
    // b^ = -G (phi^ tau) for the constant tensor tau = C_m : E_bar (Mandel)
    // sbar_v: V times the prescribed mean stress of the stress-controlled
    // components (Mandel, units of E), added at xi = 0; nullptr for none
    static void rhs_phihat(const Geometry &g, cudaStream_t st, const cpx<R> *phihat, const double *tau,
                           const double *sbar_v, cpx<R> *out);
    // out10 = (-phi^ tau, 0, 0, 0, 0): the MoDBFFT stress input of C : E_bar
    static void phihat_tau10(const Geometry &g, cudaStream_t st, const cpx<R> *phihat, const double *tau,
                             cpx<R> *out10);
    // y = a x + b y over n reals
    static void axpby(long long n, cudaStream_t st, double a, const R *x, double b, R *y);
    // weighted partial ||x||^2 of a spectral vector with nc components per frequency
    static void norm2w(const Geometry &g, cudaStream_t st, const cpx<R> *x, double *partials, int nc = 6);
    // MoDBFFT point-wise kernels (hom_modb.cuh); 3-component half spectra
    static void modb_expand(const Geometry &g, cudaStream_t st, double alpha, int with_penalty, const cpx<R> *u,
                            cpx<R> *out, int nc_out, const MinresState *state);
    static void modb_contract(const Geometry &g, cudaStream_t st, const cpx<R> *in10, cpx<R> *out3,
                              const cpx<R> *dotv, double *partials, const MinresState *state);
    static void modb_precond(const Geometry &g, cudaStream_t st, double lam_b, double mu_b, const cpx<R> *in,
                             cpx<R> *out);
    static void cg_xr(const Geometry &g, cudaStream_t st, double lam_b, double mu_b, cpx<R> *x, cpx<R> *r,
                      const cpx<R> *p, const cpx<R> *q, cpx<R> *z, const CgState *state, double *partials);
    static void cg_p(const Geometry &g, cudaStream_t st, cpx<R> *p, const cpx<R> *z, const CgState *state);
    static int ew_grid(long long n);
    static void table_init(const Geometry &g);
    static int x3_grid(const Geometry &g);
    static int x3_epart_grid(const Geometry &g);
    // resident CTAs x SMs of the persistent register n3 pass (0: it cannot run)
    static int x3r_grid(const Geometry &g);
    static int x1_grid(const Geometry &g);
    static void tma_grids(Geometry &g);
};

// FP64 helpers on spectral vectors (double2) and real fields
void spec_residual64(const Geometry &g, cudaStream_t st, const double2 *b, const double2 *ax, double2 *r,
                     double *partials, int nc = 6);             // r = b - ax, weighted ||r||^2
void spec_residual_mixed(const Geometry &g, cudaStream_t st, const double2 *b, const float2 *ax, double2 *r,
                         double *partials);                     // r = b - ax (ax FP32), weighted ||r||^2
void spec_d2f(long long ncplx, cudaStream_t st, const double2 *in, float2 *out);
void spec_f2d_acc(long long ncplx, cudaStream_t st, const float2 *in, double2 *out,
                  double a = 1.0);   // out += a in
void mean_stress64(long long V, cudaStream_t st, const double *x, const double *phi, double lam, double mu,
                   const double *macro_mandel, double *partials);   // partials[6][ew_grid(V)]
template <typename Ro>
void fields_from64(long long V, cudaStream_t st, const double *x, const double *phi, double lam, double mu,
                   double Escale, const double *macro_mandel, Ro *strain, Ro *stress);
void real_convert_f2d(long long n, cudaStream_t st, const float *in, double *out);
void real_convert_d2f(long long n, cudaStream_t st, const double *in, float *out);
void mandel_scale64(long long V, cudaStream_t st, double *f, double s);
template <typename R>
void phi_convert(long long V, cudaStream_t st, const void *in, int kind, R *out, int *bad);
int ew_blocks(long long n);
// sets the message hom_last_error(NULL) returns
void hom_set_error(const char *msg);

// single-CTA scalar kernels
void scalar_start(cudaStream_t st, MinresState *s, const double *partials, int np, double tol, int max_it,
                  int max_bodies = 0);
// end of a captured MINRES body inside a WHILE graph node: count the body and
// keep looping while one of the nb states is not done and the cap (of the
// first state) is not reached
void loop_cond(cudaStream_t st, cudaGraphConditionalHandle h, MinresState *s, int nb = 1);
// alpha_k from partials summing to <u_k, A^ u_k> / scale.  The scalar
// kernels of a stacked batch run one CTA per case c, on s[c] and the
// partials at c * np.
// tsum: the stress sums of the n3 pass (see x3), for states with dc set.
void scalar_alpha(cudaStream_t st, MinresState *s, const double *partials, int np, double scale = 1.0, int nb = 1,
                  int pdl = 0, const double *tsum = nullptr);
// the FP64 values at xi = 0 of a stress-controlled FP32 solve start from the
// right-hand side's
void dc_start(cudaStream_t st, MinresState *s, const float2 *rhs, int mask);
void scalar_givens(cudaStream_t st, MinresState *s, const double *partials, int np, int nb = 1);
// PCG scalars (MoDBFFT): start from <r0,z0>, ||r0||^2; step length; direction
void scalar_cg_start(cudaStream_t st, CgState *s, const double *partials, int np, double tol, int max_it);
void scalar_cg_alpha(cudaStream_t st, CgState *s, const double *partials, int np);
void scalar_cg_beta(cudaStream_t st, CgState *s, const double *partials, int np);
void reduce_to(cudaStream_t st, const double *partials, int np, double *out);

}  // namespace hom
