// hom_fft.cuh -- shared-memory mixed-radix FFT engine for the batched 3-D
// real FFTs of the Galerkin operator (section 2.1: the transforms of
// eq. (gal) are discrete Fourier transforms evaluated with an FFT).
//
// A CTA holds a batch of L lines of one axis in shared memory, element e of
// line l at buf[e*ES + l] with ES >= L (lines interleaved, so that the threads
// of a warp touch consecutive words whatever the stage's index pattern), and runs
// Stockham auto-sort stages between two buffers.  Each stage applies radix-R
// butterflies (R in {2,3,4,5,8,16}) held in registers; twiddles come from a
// per-axis table w[t] = exp(-2 pi i t / N) computed on the host in double.
#pragma once
#include <initializer_list>
#include <type_traits>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hom {

template <typename R> struct cpx_t;
template <> struct cpx_t<float> { using type = float2; };
template <> struct cpx_t<double> { using type = double2; };
template <typename R> using cpx = typename cpx_t<R>::type;

template <typename R> __device__ __forceinline__ cpx<R> mk(R x, R y) { cpx<R> c; c.x = x; c.y = y; return c; }
template <typename R> __device__ __forceinline__ cpx<R> add(cpx<R> a, cpx<R> b) { return mk<R>(a.x + b.x, a.y + b.y); }
template <typename R> __device__ __forceinline__ cpx<R> sub(cpx<R> a, cpx<R> b) { return mk<R>(a.x - b.x, a.y - b.y); }
template <typename R> __device__ __forceinline__ cpx<R> mul(cpx<R> a, cpx<R> b) {
    return mk<R>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename R> __device__ __forceinline__ cpx<R> conjc(cpx<R> a) { return mk<R>(a.x, -a.y); }
template <typename R> __device__ __forceinline__ cpx<R> scale(cpx<R> a, R s) { return mk<R>(a.x * s, a.y * s); }
// multiply by s*i (s = +1 or -1)
template <typename R> __device__ __forceinline__ cpx<R> mul_si(cpx<R> a, int s) {
    return s > 0 ? mk<R>(-a.y, a.x) : mk<R>(a.y, -a.x);
}

constexpr int kMaxStages = 8;

struct AxisPlan {
    int n;                    // transform length
    int nstages;
    int radix[kMaxStages];
    const void *tw;           // n complex values exp(-2 pi i t / n) (float2 or double2)
};

// ---------------------------------------------------------------------------
// In-register DFT codelets, kernel exp(S * 2 pi i j k / R), S = -1 forward.
// Constants are closed-form values: cos(2pi/5) = (sqrt5-1)/4, etc.
// ---------------------------------------------------------------------------
template <typename R, int S> __device__ __forceinline__ void dft2(cpx<R> &a, cpx<R> &b) {
    cpx<R> t = a;
    a = add<R>(t, b);
    b = sub<R>(t, b);
}

template <typename R, int S> __device__ __forceinline__ void dft3(cpx<R> *v) {
    const R h = (R)0.86602540378443864676;  // sqrt(3)/2
    cpx<R> t = add<R>(v[1], v[2]), u = sub<R>(v[1], v[2]);
    cpx<R> m = sub<R>(v[0], scale<R>(t, (R)0.5));
    cpx<R> r = mul_si<R>(scale<R>(u, h), S);
    v[0] = add<R>(v[0], t);
    v[1] = add<R>(m, r);
    v[2] = sub<R>(m, r);
}

template <typename R, int S> __device__ __forceinline__ void dft4(cpx<R> *v) {
    cpx<R> a = add<R>(v[0], v[2]), b = sub<R>(v[0], v[2]);
    cpx<R> c = add<R>(v[1], v[3]), d = mul_si<R>(sub<R>(v[1], v[3]), S);
    v[0] = add<R>(a, c);
    v[2] = sub<R>(a, c);
    v[1] = add<R>(b, d);
    v[3] = sub<R>(b, d);
}

template <typename R, int S> __device__ __forceinline__ void dft5(cpx<R> *v) {
    const R c1 = (R)0.30901699437494742410;   // cos(2pi/5)
    const R c2 = (R)-0.80901699437494742410;  // cos(4pi/5)
    const R s1 = (R)0.95105651629515357212;   // sin(2pi/5)
    const R s2 = (R)0.58778525229247312917;   // sin(4pi/5)
    cpx<R> t1 = add<R>(v[1], v[4]), t2 = add<R>(v[2], v[3]);
    cpx<R> u1 = sub<R>(v[1], v[4]), u2 = sub<R>(v[2], v[3]);
    cpx<R> a = v[0];
    cpx<R> m1 = mk<R>(a.x + c1 * t1.x + c2 * t2.x, a.y + c1 * t1.y + c2 * t2.y);
    cpx<R> m2 = mk<R>(a.x + c2 * t1.x + c1 * t2.x, a.y + c2 * t1.y + c1 * t2.y);
    cpx<R> n1 = mul_si<R>(mk<R>(s1 * u1.x + s2 * u2.x, s1 * u1.y + s2 * u2.y), S);
    cpx<R> n2 = mul_si<R>(mk<R>(s2 * u1.x - s1 * u2.x, s2 * u1.y - s1 * u2.y), S);
    v[0] = add<R>(a, add<R>(t1, t2));
    v[1] = add<R>(m1, n1);
    v[4] = sub<R>(m1, n1);
    v[2] = add<R>(m2, n2);
    v[3] = sub<R>(m2, n2);
}

// exp(S * 2 pi i k / 16) for k = 0..7
template <typename R, int S> __device__ __forceinline__ cpx<R> w16(int k) {
    const R c = (R)0.92387953251128675613;   // cos(pi/8)
    const R s = (R)0.38268343236508977173;   // sin(pi/8)
    const R h = (R)0.70710678118654752440;   // sqrt(1/2)
    R re, im;
    switch (k) {
        case 0: re = 1; im = 0; break;
        case 1: re = c; im = s; break;
        case 2: re = h; im = h; break;
        case 3: re = s; im = c; break;
        case 4: re = 0; im = 1; break;
        case 5: re = -s; im = c; break;
        case 6: re = -h; im = h; break;
        default: re = -c; im = s; break;
    }
    return mk<R>(re, S * im);
}

// a * exp(S 2 pi i k / 16) with the trivial factors spelled out: k = 4 is a
// multiplication by S i, k = 2 and 6 by sqrt(1/2) (+-1 + S i).  (IEEE rules
// keep a compiler from dropping the products with 0 and 1 by itself.)
template <typename R, int S> __device__ __forceinline__ cpx<R> mul_w16(cpx<R> a, int k) {
    const R h = (R)0.70710678118654752440;
    if (k == 0) return a;
    if (k == 4) return mul_si<R>(a, S);
    if (k == 2) return mk<R>(h * (a.x - (R)S * a.y), h * (a.y + (R)S * a.x));
    if (k == 6) return mk<R>(-h * (a.x + (R)S * a.y), h * ((R)S * a.x - a.y));
    return mul<R>(a, w16<R, S>(k));
}

template <typename R, int S> __device__ __forceinline__ void dft8(cpx<R> *v) {
    cpx<R> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft4<R, S>(e);
    dft4<R, S>(o);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const cpx<R> t = mul_w16<R, S>(o[k], 2 * k);
        v[k] = add<R>(e[k], t);
        v[k + 4] = sub<R>(e[k], t);
    }
}

template <typename R, int S> __device__ __forceinline__ void dft16(cpx<R> *v) {
    cpx<R> e[8], o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { e[k] = v[2 * k]; o[k] = v[2 * k + 1]; }
    dft8<R, S>(e);
    dft8<R, S>(o);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const cpx<R> t = mul_w16<R, S>(o[k], k);
        v[k] = add<R>(e[k], t);
        v[k + 8] = sub<R>(e[k], t);
    }
}

// exp(S 2 pi i e / 9) for e = 1, 2, 4, the twiddles of the radix-9 butterfly:
// cosines and sines of 40, 80 and 160 degrees
template <typename R, int S> __device__ __forceinline__ cpx<R> w9(int e) {
    const R c1 = (R)0.76604444311897803520, s1 = (R)0.64278760968653932632;
    const R c2 = (R)0.17364817766693034885, s2 = (R)0.98480775301220805937;
    const R c4 = (R)-0.93969262078590838405, s4 = (R)0.34202014332566873304;
    return e == 1 ? mk<R>(c1, (R)S * s1) : (e == 2 ? mk<R>(c2, (R)S * s2) : mk<R>(c4, (R)S * s4));
}

template <typename R, int S, int RAD> __device__ __forceinline__ void dft(cpx<R> *v);

template <typename R, int S> __device__ __forceinline__ void dft9(cpx<R> *v) {
    cpx<R> y[3][3];   // y[k1][n2]: DFT-3 over n1 of x[3 n1 + n2], times w9^(n2 k1)
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
        cpx<R> a[3] = {v[n2], v[3 + n2], v[6 + n2]};
        dft3<R, S>(a);
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) y[k1][n2] = n2 * k1 == 0 ? a[k1] : mul<R>(a[k1], w9<R, S>(n2 * k1));
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
        dft3<R, S>(y[k1]);
#pragma unroll
        for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = y[k1][k2];
    }
}

// DFT of length N1 N2, N1 and N2 coprime, in registers without twiddles
// (Good's prime-factor mapping): inputs x[(N2 n1 + N1 n2) mod N], output
// X[k] from the DFT-N1 index k mod N1 and the DFT-N2 index k mod N2.
template <typename R, int S, int N1, int N2> __device__ __forceinline__ void dft_pfa(cpx<R> *v) {
    constexpr int N = N1 * N2;
    cpx<R> y[N1][N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
        cpx<R> a[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) a[n1] = v[(N2 * n1 + N1 * n2) % N];
        dft<R, S, N1>(a);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) y[k1][n2] = a[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) dft<R, S, N2>(y[k1]);
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = y[k % N1][k % N2];
}

template <typename R, int S, int RAD> __device__ __forceinline__ void dft(cpx<R> *v) {
    if constexpr (RAD == 2) dft2<R, S>(v[0], v[1]);
    else if constexpr (RAD == 3) dft3<R, S>(v);
    else if constexpr (RAD == 4) dft4<R, S>(v);
    else if constexpr (RAD == 5) dft5<R, S>(v);
    else if constexpr (RAD == 6) dft_pfa<R, S, 2, 3>(v);
    else if constexpr (RAD == 8) dft8<R, S>(v);
    else if constexpr (RAD == 9) dft9<R, S>(v);
    else if constexpr (RAD == 10) dft_pfa<R, S, 2, 5>(v);
    else if constexpr (RAD == 12) dft_pfa<R, S, 4, 3>(v);
    else if constexpr (RAD == 15) dft_pfa<R, S, 3, 5>(v);
    else if constexpr (RAD == 18) dft_pfa<R, S, 2, 9>(v);
    else if constexpr (RAD == 20) dft_pfa<R, S, 4, 5>(v);
    else {
        static_assert(RAD == 16, "no butterfly of this radix");
        dft16<R, S>(v);
    }
}

// ---------------------------------------------------------------------------
// One Stockham stage over L interleaved lines: src -> dst.
// Butterfly j (0 <= j < N/RAD) reads src[j + r N/RAD], multiplies input r by
// w_{Ns RAD}^{(j mod Ns) r}, and writes dst[(j/Ns) Ns RAD + (j mod Ns) + r Ns].
// ---------------------------------------------------------------------------
template <typename R, int S, int RAD>
__device__ __forceinline__ void stockham_stage(const cpx<R> *__restrict__ src, cpx<R> *__restrict__ dst,
                                               int N, int Ns, int L, int ES, const cpx<R> *__restrict__ tw) {
    const int nb = N / RAD;
    const int total = nb * L;
    const int twstep = N / (Ns * RAD);
    for (int b = threadIdx.x; b < total; b += blockDim.x) {
        const int j = b / L;
        const int l = b - j * L;
        cpx<R> v[RAD];
#pragma unroll
        for (int r = 0; r < RAD; ++r) v[r] = src[(j + r * nb) * ES + l];
        const int jm = j % Ns;
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < RAD; ++r) {
                cpx<R> w = __ldg(&tw[jm * r * twstep]);
                if (S > 0) w.y = -w.y;
                v[r] = mul<R>(v[r], w);
            }
        }
        dft<R, S, RAD>(v);
        const int o = (j - jm) * RAD + jm;
#pragma unroll
        for (int r = 0; r < RAD; ++r) dst[(o + r * Ns) * ES + l] = v[r];
    }
}

// Full transform of L interleaved lines held in bufA.  Returns the buffer
// holding the result (bufA or bufB).  All threads of the block must call it.
template <typename R, int S>
__device__ cpx<R> *fft_lines(cpx<R> *bufA, cpx<R> *bufB, int L, int ES, const AxisPlan &p) {
    cpx<R> *src = bufA, *dst = bufB;
    const cpx<R> *tw = reinterpret_cast<const cpx<R> *>(p.tw);
    int Ns = 1;
    for (int s = 0; s < p.nstages; ++s) {
        const int rad = p.radix[s];
        switch (rad) {
            case 2: stockham_stage<R, S, 2>(src, dst, p.n, Ns, L, ES, tw); break;
            case 3: stockham_stage<R, S, 3>(src, dst, p.n, Ns, L, ES, tw); break;
            case 4: stockham_stage<R, S, 4>(src, dst, p.n, Ns, L, ES, tw); break;
            case 5: stockham_stage<R, S, 5>(src, dst, p.n, Ns, L, ES, tw); break;
            case 8: stockham_stage<R, S, 8>(src, dst, p.n, Ns, L, ES, tw); break;
            default: stockham_stage<R, S, 16>(src, dst, p.n, Ns, L, ES, tw); break;
        }
        __syncthreads();
        Ns *= rad;
        cpx<R> *t = src; src = dst; dst = t;
    }
    return src;
}

// ---------------------------------------------------------------------------
// Register-resident engine for lengths known at compile time (powers of two,
// and 96 and 160, the mixed lengths of the batched cell studies).
// Every thread owns E elements of one line for the whole transform (BPT =
// E/RAD butterflies per stage), so a stage is: load the thread's butterfly
// inputs from the single shared buffer into registers, barrier, compute,
// store the outputs in place, barrier.  One buffer instead of two, all index
// arithmetic on compile-time powers of two.  The CTA must have exactly
// L * N / E threads; thread t works on line t % L.
// ---------------------------------------------------------------------------
// Stages in order R0, R1, R2, R3 (NS of them); E is a multiple of every
// stage's radix.  The mixed lengths 96 = 4 4 2 3 and 160 = 4 4 2 5 put the
// odd radix last, so that the sub-transform length before every stage is a
// power of two.
template <int N> struct FastPlan;
template <> struct FastPlan<8>   { static constexpr int E = 8,  NS = 1, R0 = 8,  R1 = 1,  R2 = 1, R3 = 1; };
template <> struct FastPlan<16>  { static constexpr int E = 16, NS = 1, R0 = 16, R1 = 1,  R2 = 1, R3 = 1; };
template <> struct FastPlan<32>  { static constexpr int E = 8,  NS = 2, R0 = 8,  R1 = 4,  R2 = 1, R3 = 1; };
template <> struct FastPlan<64>  { static constexpr int E = 8,  NS = 2, R0 = 8,  R1 = 8,  R2 = 1, R3 = 1; };
template <> struct FastPlan<96>  { static constexpr int E = 12, NS = 4, R0 = 4,  R1 = 4,  R2 = 2, R3 = 3; };
template <> struct FastPlan<128> { static constexpr int E = 16, NS = 2, R0 = 16, R1 = 8,  R2 = 1, R3 = 1; };
template <> struct FastPlan<160> { static constexpr int E = 20, NS = 4, R0 = 4,  R1 = 4,  R2 = 2, R3 = 5; };
template <> struct FastPlan<256> { static constexpr int E = 16, NS = 2, R0 = 16, R1 = 16, R2 = 1, R3 = 1; };
template <> struct FastPlan<512> { static constexpr int E = 16, NS = 3, R0 = 16, R1 = 16, R2 = 2, R3 = 1; };

// The n3 pass (shared-memory form) takes 96 and 160 in two stages instead
// of four, with radix-12 and radix-20 butterflies in registers (24 and 40
// elements per thread): 96 = 8 12, 160 = 8 20.  Other lengths as FastPlan.
template <int N> struct FastPlanN3 : FastPlan<N> {};
template <> struct FastPlanN3<96>  { static constexpr int E = 24, NS = 2, R0 = 8, R1 = 12, R2 = 1, R3 = 1; };
template <> struct FastPlanN3<160> { static constexpr int E = 40, NS = 2, R0 = 8, R1 = 20, R2 = 1, R3 = 1; };

__host__ __device__ constexpr bool is_fast_length(int n) {
    return n == 8 || n == 16 || n == 32 || n == 64 || n == 96 || n == 128 || n == 160 || n == 256 || n == 512;
}
__host__ __device__ constexpr int fast_elems(int n) {
    return (n == 8 || n == 32 || n == 64) ? 8 : (n == 96 ? 12 : (n == 160 ? 20 : 16));
}
__host__ __device__ constexpr int fast_elems_n3(int n) { return n == 96 ? 24 : (n == 160 ? 40 : fast_elems(n)); }
// Position of element e of a line in a tile with element stride ES; with
// PAD, one slot is skipped every 16 elements so that the stride-16 writes of
// a radix-16 stage spread over the shared-memory banks.
template <int PAD> __device__ __forceinline__ int epos(int e, int ES) { return e * ES + (PAD ? (e >> 4) : 0); }

// Barrier of the threads that run a transform: the whole CTA (n = 0), or
// the first n threads on named barrier 1 (n a multiple of 32).
__device__ __forceinline__ void group_sync(int n) {
    if (n == 0) __syncthreads();
    else asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory");
}

template <typename R, int S, int N, int RAD, int NS_BEFORE, int PAD, typename Plan = FastPlan<N>>
__device__ __forceinline__ void fast_stage(cpx<R> *buf, int ES, int l, int j0, const cpx<R> *__restrict__ tw) {
    constexpr int E = Plan::E;
    constexpr int BPT = E / RAD;
    constexpr int nb = N / RAD;
    constexpr int jstep = N / E;
    constexpr int twstep = N / (NS_BEFORE * RAD);
    cpx<R> v[BPT][RAD];
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int j = j0 + i * jstep;
#pragma unroll
        for (int r = 0; r < RAD; ++r) v[i][r] = buf[epos<PAD>(j + r * nb, ES) + l];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int j = j0 + i * jstep;
        const int jm = j & (NS_BEFORE - 1);
        if (NS_BEFORE > 1) {
#pragma unroll
            for (int r = 1; r < RAD; ++r) {
                cpx<R> w = __ldg(&tw[jm * r * twstep]);
                if (S > 0) w.y = -w.y;
                v[i][r] = mul<R>(v[i][r], w);
            }
        }
        dft<R, S, RAD>(v[i]);
        const int o = (j - jm) * RAD + jm;
#pragma unroll
        for (int r = 0; r < RAD; ++r) buf[epos<PAD>(o + r * NS_BEFORE, ES) + l] = v[i][r];
    }
    __syncthreads();
}

// Transform of L interleaved lines in buf (in place), element e of line l
// at buf[epos<PAD>(e, ES) + l] (ES >= L).  The CTA has exactly L * N / E threads:
// every thread takes part in every barrier.
template <typename R, int S, int N, int PAD = 0, typename P = FastPlan<N>>
__device__ __forceinline__ void fast_fft(cpx<R> *buf, int L, int ES, const cpx<R> *__restrict__ tw) {
    const int l = (int)threadIdx.x % L;
    const int j0 = (int)threadIdx.x / L;
    fast_stage<R, S, N, P::R0, 1, PAD, P>(buf, ES, l, j0, tw);
    if constexpr (P::NS > 1) fast_stage<R, S, N, P::R1, P::R0, PAD, P>(buf, ES, l, j0, tw);
    if constexpr (P::NS > 2) fast_stage<R, S, N, P::R2, P::R0 * P::R1, PAD, P>(buf, ES, l, j0, tw);
    if constexpr (P::NS > 3) fast_stage<R, S, N, P::R3, P::R0 * P::R1 * P::R2, PAD, P>(buf, ES, l, j0, tw);
}

// ---------------------------------------------------------------------------
// Line engine: the register engine above for every length 2^a 3^b 5^c in
// [16, 512], with two or three stages of any of the butterflies.  TPL threads
// share a line; a stage of radix RAD has N / RAD butterflies, which the TPL
// threads take in ceil(N / (RAD TPL)) rounds (idle where they do not divide:
// 108 = 12 9 with TPL = 12 idles 3 threads of 12 in its radix-12 stage).
// Measured against the runtime Stockham engine (whose index arithmetic
// divides at run time and which needs two shared buffers) in the comments of
// the passes that use it.
// ---------------------------------------------------------------------------
struct LinePlanV { int r0, r1, r2, tpl; };

constexpr bool line_radix(int r) {
    return r == 2 || r == 3 || r == 4 || r == 5 || r == 6 || r == 8 || r == 9 || r == 10 || r == 12 || r == 15 ||
           r == 16 || r == 18 || r == 20;
}
constexpr int kLineMaxElems = 20;

// (complex) elements a thread holds between the barriers of its widest stage
constexpr int line_elems(int N, int r0, int r1, int r2, int tpl) {
    const int rs[3] = {r0, r1, r2};
    int e = 0;
    for (int i = 0; i < 3; ++i) {
        const int v = (N / rs[i] + tpl - 1) / tpl * rs[i];
        if (rs[i] > 1 && v > e) e = v;
    }
    return e;
}

// radices (largest first: a stage's twiddles are N (1 - 1/r)) and threads of a
// line.  The score weighs the element slots a line passes through (its
// stages' rounds times TPL threads, idle ones included) against the elements
// a thread holds; more than 16 of them (32 registers) only where few plans
// divide N in two stages.  The power-of-two plans are 64 = 8 8, 128 = 16 8,
// 256 = 16 16 with 8, 8 and 16 threads.
constexpr LinePlanV line_plan(int N) {
    LinePlanV best{0, 0, 0, 0};
    int bc = 1 << 30;
    for (int r0 = 20; r0 >= 2; --r0) {
        if (!line_radix(r0) || N % r0) continue;
        for (int r1 = r0; r1 >= 1; --r1) {
            if ((r1 > 1 && !line_radix(r1)) || (N / r0) % r1) continue;
            const int r2 = N / r0 / r1;
            if (r2 > r1 || (r2 > 1 && !line_radix(r2))) continue;
            for (int tpl = 2; tpl <= 32; ++tpl) {
                const int e = line_elems(N, r0, r1, r2, tpl);
                if (e > kLineMaxElems) continue;
                int slots = 0;
                for (int r : {r0, r1, r2})
                    if (r > 1) slots += (N / r + tpl - 1) / tpl * r * tpl;
                const int score = slots * 1000 / N + e * 40 + tpl + (e > 16 ? 400 : 0);
                if (score < bc) {
                    bc = score;
                    best = LinePlanV{r0, r1, r2, tpl};
                }
            }
        }
    }
    return best;
}
// The lengths' kernels are instantiated from these lists (see the passes).
#define HOM_LINE_LENGTHS_A(X) \
    X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64) X(72) X(75) X(80)
#define HOM_LINE_LENGTHS_B(X) \
    X(81) X(90) X(96) X(100) X(108) X(120) X(125) X(128) X(135) X(144) X(150) X(160) X(162) X(180) X(192) X(200)
#define HOM_LINE_LENGTHS_C(X) \
    X(216) X(225) X(240) X(243) X(250) X(256) X(270) X(288) X(300) X(320) X(324) X(360) X(375) X(384) X(400) X(405) \
    X(432) X(450) X(480) X(486) X(500) X(512)

template <int N> struct LinePlan {
    static constexpr LinePlanV P = line_plan(N);
    static constexpr int R0 = P.r0, R1 = P.r1, R2 = P.r2, TPL = P.tpl;
    static constexpr int E = line_elems(N, P.r0, P.r1, P.r2, P.tpl);
    static_assert(R0 * R1 * R2 == N, "no plan for this length");
};
// (FP64 passes also run 8 on it)
#define HOM_F64_LENGTHS_A(X) X(8) HOM_LINE_LENGTHS_A(X)
// threads of a line at run time (0: not a length of the line engine)
int line_tpl(int n);

template <typename R, int S, int N, int RAD, int NSB, int TPL>
__device__ __forceinline__ void line_stage(cpx<R> *buf, int ES, int l, int j0, const cpx<R> *__restrict__ tw,
                                           int nsync) {
    constexpr int nb = N / RAD;
    constexpr int BPT = (nb + TPL - 1) / TPL;
    constexpr bool even = nb % TPL == 0;
    constexpr int twstep = N / (NSB * RAD);
    cpx<R> v[BPT][RAD];
    // idle slots load and transform butterfly 0 and store nothing, so that
    // only the stores are conditional
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int jj = j0 + i * TPL, j = j0 < TPL && (even || jj < nb) ? jj : 0;
#pragma unroll
        for (int r = 0; r < RAD; ++r) v[i][r] = buf[(j + r * nb) * ES + l];
    }
    group_sync(nsync);
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int jj = j0 + i * TPL;
        const bool live = j0 < TPL && (even || jj < nb);
        const int j = live ? jj : 0;
        const int jm = nb == NSB ? j : j % NSB;   // nb = NSB in the last stage
        if constexpr (NSB > 1) {
#pragma unroll
            for (int r = 1; r < RAD; ++r) {
                cpx<R> w = __ldg(&tw[jm * r * twstep]);
                if (S > 0) w.y = -w.y;
                v[i][r] = mul<R>(v[i][r], w);
            }
        }
        dft<R, S, RAD>(v[i]);
        const int o = (j - jm) * RAD + jm;
        if (live) {
#pragma unroll
            for (int r = 0; r < RAD; ++r) buf[(o + r * NSB) * ES + l] = v[i][r];
        }
    }
    group_sync(nsync);
}

// Transform of L interleaved lines in buf (in place), element e of line l at
// buf[e * ES + l].  The CTA's threads (nsync = 0), or its first nsync on named
// barrier 1, all call it; those beyond L * TPL only take part in the barriers.
template <typename R, int S, int N>
__device__ __forceinline__ void line_fft(cpx<R> *buf, int L, int ES, const cpx<R> *__restrict__ tw, int nsync = 0) {
    using P = LinePlan<N>;
    const int l = (int)threadIdx.x % L;
    const int j0 = (int)threadIdx.x / L;
    line_stage<R, S, N, P::R0, 1, P::TPL>(buf, ES, l, j0, tw, nsync);
    if constexpr (P::R1 > 1) line_stage<R, S, N, P::R1, P::R0, P::TPL>(buf, ES, l, j0, tw, nsync);
    if constexpr (P::R2 > 1) line_stage<R, S, N, P::R2, P::R0 * P::R1, P::TPL>(buf, ES, l, j0, tw, nsync);
}

// The runtime engine's transform (its radices in its order: powers of two from
// the largest, then threes, then fives) with everything but the data known at
// compile time and the line engine's in-place stages: the same operations on the
// same values, so the same bits, without the second buffer and the divisions by
// run-time values.
constexpr int ordered_radix(int n, int s) {
    int a = 0, b = 0, c = 0;
    while (n % 2 == 0) { n /= 2; ++a; }
    while (n % 3 == 0) { n /= 3; ++b; }
    while (n % 5 == 0) { n /= 5; ++c; }
    const int st2 = (a + 3) / 4;
    if (s < st2) return 1 << (a / st2 + (s < a % st2 ? 1 : 0));
    return s < st2 + b ? 3 : (s < st2 + b + c ? 5 : 1);
}
// threads of a line: 12 to 16 elements each
__host__ __device__ constexpr int ordered_tpl(int n) { return (n + 11) / 12; }

template <typename R, int S, int N, int STAGE = 0, int NSB = 1>
__device__ __forceinline__ void ordered_fft(cpx<R> *buf, int L, int ES, const cpx<R> *__restrict__ tw) {
    constexpr int RAD = ordered_radix(N, STAGE);
    if constexpr (RAD > 1) {
        line_stage<R, S, N, RAD, NSB, ordered_tpl(N)>(buf, ES, (int)threadIdx.x % L, (int)threadIdx.x / L, tw, 0);
        ordered_fft<R, S, N, STAGE + 1, NSB * RAD>(buf, L, ES, tw);
    }
}

}  // namespace hom
