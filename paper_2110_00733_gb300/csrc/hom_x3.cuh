// hom_x3.cuh -- persistent n3 pass (FP32, 6-component spectra, spectrum in and
// out) at every length of X3Plan: the C2R of a row, the material law with the
// strain-energy sums, and the R2C.
//
// A row is three packed lines Z_p = X_2p + i X_2p+1 of N = A B values.  A CTA
// takes tiles of ROWS consecutive rows (one contiguous block of the spectrum)
// and runs both transforms in two stages with the law between them in
// registers:
//   1. inverse radix-A butterflies straight from the staged half spectrum
//      (the upper half of a line is the conjugate mirror of the lower);
//   2. a thread takes one radix-B butterfly of all three lines, which leaves
//      it with all six components of B voxels: the law and the energy, then
//      the forward radix-B butterflies on the same voxels;
//   3. forward radix-A butterflies, two of a line per thread (u and B - u),
//      whose outputs hold every Z[k] together with the Z[N - k] that
//      unpacking needs, stored as 16-byte values that consecutive threads
//      place one after another.
// Between the stages the values cross the CTA through shared memory (each
// element written and read twice); the rows' spectra come by one bulk copy
// into a staging buffer that the next tile's copy fills while stages 2 and 3
// run.  Strides are odd, and the lines of a row 6 (mod 16) of them apart, so
// that the accesses of half a warp fall on different banks.
//
// Bound by instruction issue at 8 to 12 warps per SM (shared memory holds the
// rows in flight, registers the law's 6 B values), then by HBM.  Against the
// shared-memory pass k_x3, whose three lines of a row take separate threads
// and whose stages of the runtime engine divide by run-time values: 192^3 283
// to 126 us (52 at the copy rate), 108^3 67 to 26, 160^3 120 to 67, 240^3 557
// to 239.  At 128 it also beats the register pass k_x3r (32 against 35 us at
// 128^3, equal at 64); at 256, whose 16 x 16 plan leaves 8 warps per SM, k_x3r
// is the faster (234 against 254 us at 256^3) and keeps that length.
#pragma once
#include "hom_passes.cuh"

namespace hom {

constexpr bool x3_radix(int r) { return line_radix(r) && r <= 20; }

struct X3PlanV { int a, b; };
// N = A B: registers of the widest stage, 3 B values (the law) or 2 A (the
// unpacking pairs), as few as possible
constexpr X3PlanV x3_plan(int N) {
    X3PlanV best{0, 0};
    int bc = 1 << 30;
    for (int a = 2; a <= 20; ++a) {
        if (!x3_radix(a) || N % a || !x3_radix(N / a)) continue;
        const int b = N / a, c = 3 * b > 2 * a ? 3 * b : 2 * a;
        if (c < bc) {
            bc = c;
            best = X3PlanV{a, b};
        }
    }
    return best;
}

// the lengths that have a plan (two of the butterflies up to radix 20)
#define HOM_X3_LENGTHS_A(X) \
    X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64) \
    X(72) X(75) X(80)
#define HOM_X3_LENGTHS_B(X) \
    X(81) X(90) X(96) X(100) X(108) X(120) X(128) X(135) X(144) X(150) X(160) X(162) X(180)
#define HOM_X3_LENGTHS_C(X) \
    X(192) X(200) X(216) X(225) X(240) X(256) X(270) X(288) X(300) X(320) X(324) X(360) X(400)

template <int N> struct X3Plan {
    static constexpr int A = x3_plan(N).a, B = x3_plan(N).b, H = N / 2 + 1;
    static_assert(A * B == N, "no plan for this length");
    static constexpr int A1 = A | 1, B1 = B | 1;              // odd strides of the two exchanges
    static constexpr int LINE = A1 * B > B1 * A ? A1 * B : B1 * A;
    static constexpr int PS = LINE + ((6 * A1 - LINE) % 16 + 16) % 16;   // line stride = 6 A1 (mod 16)
    static constexpr int RS = 3 * PS;
    // rows per tile: as many as two warps take the law's butterflies of at once
    static constexpr int NT = 64, ROWS = NT / A;
    static constexpr size_t STAGE = ((size_t)ROWS * H * 48 + 127) / 128 * 128;
    static constexpr size_t SMEM = STAGE + (size_t)ROWS * RS * sizeof(float2);
    // resident CTAs asked for: what shared memory allows (227 KB, about 1 KB of
    // it the system's per CTA), with registers for 3 B or 2 A values and about
    // as many again for addresses, twiddles and butterfly temporaries (10, 8,
    // 6 and 4 CTAs of two warps leave 96, 128, 168 and 255 registers)
    static constexpr int WIDE = 3 * B > 2 * A ? 3 * B : 2 * A;
    static constexpr int BY_SMEM = (int)(227 * 1024 / (SMEM + 1536));
    static constexpr int BY_REGS = WIDE <= 18 ? 10 : (WIDE <= 24 ? 8 : (WIDE <= 36 ? 6 : 4));
    static constexpr int CTAS = BY_SMEM < BY_REGS ? BY_SMEM : BY_REGS;
};

// SUMS: the per-CTA stress sums (tsum of Launch::x3) too
template <int N, bool SUMS>
__global__ void __launch_bounds__(X3Plan<N>::NT, X3Plan<N>::CTAS)
    k_x3_line(Geometry g, const float2 *__restrict__ in, float2 *__restrict__ out, int material, float lam, float mu2,
              const float *__restrict__ phi, const MinresState *state, double *__restrict__ epart, Fold fold,
              double *__restrict__ tsum) {
    pdl_release();
    pdl_wait();   // predecessor complete (programmatic launch in the MINRES graph)
    using P = X3Plan<N>;
    constexpr int A = P::A, B = P::B, H = P::H, ROWS = P::ROWS, NT = P::NT, PS = P::PS, RS = P::RS;
    constexpr int A1 = P::A1, B1 = P::B1, UP = B / 2 + 1;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ double sacc[kNbMax * (NT / 32)];   // energy of each case, one running sum a warp
    const float4 *stg = reinterpret_cast<const float4 *>(smem_raw);     // [row][k][line]
    float2 *w = reinterpret_cast<float2 *>(smem_raw + P::STAGE);        // exchange buffer
    __shared__ double ssum[SUMS ? 6 * kNbMax * (NT / 32) : 1];   // the same for the stress components
    __shared__ Acc<float> sff[SUMS ? 6 * NT : 1];                // and each thread's sums of the running case
    const int tid = threadIdx.x;
    const bool leader = tid == 0;
    const int nrows = g.n1 * g.n2;
    const int tpc = (nrows + ROWS - 1) / ROWS;   // tiles per load case
    const int ntiles = tpc * g.nb;
    const float2 *tw = reinterpret_cast<const float2 *>(g.ax[2].tw);
    const float sV = 1.0f / (float)g.V;
    if (leader) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    for (int i = tid; i < kNbMax * (NT / 32); i += NT) sacc[i] = 0.0;
    if constexpr (SUMS)
    {
        for (int i = tid; i < 6 * kNbMax * (NT / 32); i += NT) ssum[i] = 0.0;
        for (int c = 0; c < 6; ++c) sff[c * NT + tid] = Acc<float>{};
    }
    __syncthreads();
    auto live_from = [&](int t) {
        while (t < ntiles && skip_case(state, t / tpc)) t += gridDim.x;
        return t;
    };
    auto issue = [&](int t) {
        const int cs = t / tpc, row0 = (t - cs * tpc) * ROWS;
        const uint32_t bytes = (uint32_t)min(ROWS, nrows - row0) * (uint32_t)(H * 48);
        mbar_expect_tx(&bar, bytes);
        bulk_load(smem_raw, in + ((size_t)cs * nrows + row0) * (H * 6), bytes, &bar);
    };
    double eacc = 0.0;   // this thread's energy of the running case
    int tile = live_from(blockIdx.x);
    if (leader && tile < ntiles) issue(tile);
    for (int it = 0; tile < ntiles; ++it) {
        const int next = live_from(tile + gridDim.x);
        const int cs = tile / tpc, row0 = (tile - cs * tpc) * ROWS;
        const int nr = min(ROWS, nrows - row0);
        const bool ok = mbar_wait_bounded(&bar, (uint32_t)it & 1u);
        if (__syncthreads_or(!ok)) {
            if (leader) {   // record, then wait (bounded) for this CTA's load in flight
                atomicExch(g.err, 1);
                mbar_wait_bounded(&bar, (uint32_t)it & 1u);
            }
            return;
        }
        // ---- 1: inverse radix-A butterflies j of line p, inputs k = j + B r
#pragma unroll 1
        for (int t = tid; t < ROWS * B * 3; t += NT) {
            const int row = t / (3 * B), q = t - row * (3 * B), j = q / 3, p = q - 3 * j;
            if (row >= nr) break;
            const float4 *x = stg + (size_t)row * (3 * H) + p;
            float2 z[A];
#pragma unroll
            for (int r = 0; r < A; ++r) {
                const int k = j + B * r;
                const bool up = 2 * k > N;
                float4 v = x[3 * (up ? N - k : k)];
                if (k == 0 || 2 * k == N) v.y = v.w = 0.f;   // self-conjugate bins: real parts
                // a = (v.x, v.y), b = (v.z, v.w): Z[k] = a + i b, Z[N - k] = conj a + i conj b
                z[r] = up ? make_float2(v.x + v.w, v.z - v.y) : make_float2(v.x - v.w, v.y + v.z);
            }
            dft<float, 1, A>(z);
            float2 *o = w + row * RS + p * PS + j * A1;
#pragma unroll
            for (int r = 0; r < A; ++r) o[r] = z[r];
        }
        __syncthreads();
        if (leader && next < ntiles) issue(next);   // the staging buffer is read
        // ---- 2: radix-B butterfly j of the three lines, the law, radix-B forward
        const int row2 = tid / A, j2 = tid - row2 * A;
        const bool live2 = row2 < nr && row2 < ROWS;
        float2 z[3][B];
        float ph[B];
        if (live2) {
            const float *prow = phi + (size_t)(row0 + row2) * N + j2;
            if (material) {
#pragma unroll
                for (int r = 0; r < B; ++r) ph[r] = __ldg(prow + A * r);
            }
            const float2 *o = w + row2 * RS + j2;
#pragma unroll
            for (int p = 0; p < 3; ++p)
#pragma unroll
                for (int r = 0; r < B; ++r) z[p][r] = o[p * PS + r * A1];
        }
        __syncthreads();
        float en = 0.f, ts[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // sums over B voxels
        if (live2) {
            const float2 *twj;
            asm volatile("mov.b64 %0, %1;" : "=l"(twj) : "l"(tw));
#pragma unroll
            for (int r = 1; r < B; ++r) {
                float2 c = tw_load(twj + j2 * r);
                c.y = -c.y;
#pragma unroll
                for (int p = 0; p < 3; ++p) z[p][r] = mul<float>(z[p][r], c);
            }
#pragma unroll
            for (int p = 0; p < 3; ++p) dft<float, 1, B>(z[p]);
            // voxels j2 + A r (scaled by 1/V)
            if (material) {
#pragma unroll
                for (int r = 0; r < B; ++r) {
                    float t[6];
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        t[2 * p] = z[p][r].x * sV;
                        t[2 * p + 1] = z[p][r].y * sV;
                    }
                    const float sum = t[0] + t[1] + t[2];
                    const float tr = lam * sum;
                    float ee = t[0] * t[0];
#pragma unroll
                    for (int c = 1; c < 6; ++c) ee += t[c] * t[c];
                    en += ph[r] * (tr * sum + mu2 * ee);
#pragma unroll
                    for (int c = 0; c < 6; ++c) {
                        t[c] = ph[r] * ((c < 3 ? tr : 0.f) + mu2 * t[c]);
                        if constexpr (SUMS) ts[c] += t[c];
                    }
#pragma unroll
                    for (int p = 0; p < 3; ++p) z[p][r] = make_float2(t[2 * p], t[2 * p + 1]);
                }
            } else {
#pragma unroll
                for (int p = 0; p < 3; ++p)
#pragma unroll
                    for (int r = 0; r < B; ++r) z[p][r] = make_float2(z[p][r].x * sV, z[p][r].y * sV);
            }
            float2 *o = w + row2 * RS + j2 * B1;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                dft<float, -1, B>(z[p]);
#pragma unroll
                for (int r = 0; r < B; ++r) o[p * PS + r] = z[p][r];
            }
        }
        // reduced over the warp once a case, not once a tile: FP64 adds run at
        // a small rate (six sums a tile took 17 of 50 us at 128^3)
        const bool last = next >= ntiles || next / tpc != cs;
        eacc += (double)en;
        if (epart && last) {
            const double ws = warp_sum(eacc);
            if ((tid & 31) == 0) sacc[cs * (NT / 32) + (tid >> 5)] += ws;
            eacc = 0.0;
        }
        if constexpr (SUMS) {
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                Acc<float> s = sff[c * NT + tid];
                s.add(ts[c]);
                if (last) {
                    const double ws = warp_sum(s.value());
                    if ((tid & 31) == 0) ssum[(c * kNbMax + cs) * (NT / 32) + (tid >> 5)] += ws;
                    s = Acc<float>{};
                }
                sff[c * NT + tid] = s;
            }
        }
        __syncthreads();
        // ---- 3: forward radix-A butterflies u and v = B - u (mod B) of line p:
        // frequencies u + B r and v + B r, the partner of u + B r being
        // v + B (A - 1 - r), or B (A - r) for u = 0
#pragma unroll 1
        for (int t = tid; t < ROWS * UP * 3; t += NT) {
            const int row = t / (3 * UP), q = t - row * (3 * UP), u = q / 3, p = q - 3 * u;
            if (row >= nr) break;
            const int v = u == 0 ? 0 : B - u;
            const float2 *o = w + row * RS + p * PS;
            const float2 *twj;
            asm volatile("mov.b64 %0, %1;" : "=l"(twj) : "l"(tw));
            float2 zu[A], zv[A];
#pragma unroll
            for (int r = 0; r < A; ++r) {
                zu[r] = o[r * B1 + u];
                zv[r] = o[r * B1 + v];
                if (r > 0) {
                    zu[r] = mul<float>(zu[r], tw_load(twj + u * r));
                    zv[r] = mul<float>(zv[r], tw_load(twj + v * r));
                }
            }
            dft<float, -1, A>(zu);
            dft<float, -1, A>(zv);
            float4 *dst = reinterpret_cast<float4 *>(out + ((size_t)cs * nrows + row0 + row) * (H * 6)) + p;
            // X_a[k] = (Z[k] + conj Z[N-k]) / 2,  X_b[k] = (Z[k] - conj Z[N-k]) / (2i)
            auto unpack = [](float2 z, float2 m) {
                return make_float4(0.5f * (z.x + m.x), 0.5f * (z.y - m.y), 0.5f * (z.y + m.y), -0.5f * (z.x - m.x));
            };
#pragma unroll
            for (int r = 0; r <= A / 2; ++r) {
                const int k = u + B * r;
                if (2 * k <= N) {
                    const float2 m = u == 0 ? zu[(A - r) % A] : zv[A - 1 - r];
                    dst[3 * k] = unpack(zu[r], m);
                }
            }
#pragma unroll
            for (int r = 0; r <= A / 2; ++r) {
                const int k = v + B * r;
                if (v != u && 2 * k <= N) dst[3 * k] = unpack(zv[r], zu[A - 1 - r]);
            }
        }
        tile = next;   // (the barrier after the next wait: the exchange buffer is read)
    }
    if constexpr (SUMS) {
        __syncthreads();
        if (tid < 6 * g.nb) {
            const int c = tid / g.nb, cc = tid - c * g.nb;
            double t = 0.0;
            for (int i = 0; i < NT / 32; ++i) t += ssum[(c * kNbMax + cc) * (NT / 32) + i];
            tsum[(size_t)tid * gridDim.x + blockIdx.x] = t;   // = tsum[(c * nb + case) * grid + block]
        }
    }
    if (epart) {
        __syncthreads();
        if (tid < g.nb) {
            double t = 0.0;
            for (int i = 0; i < NT / 32; ++i) t += sacc[tid * (NT / 32) + i];
            epart[(size_t)tid * gridDim.x + blockIdx.x] = t;   // = epart[case * grid + block]
            __threadfence();
        }
        if (fold.cnt && last_of(fold.cnt, gridDim.x)) {   // alpha of every case
            for (int cc = tid >> 5; cc < g.nb; cc += NT / 32) {
                double t = 0.0;
                for (int i = tid & 31; i < (int)gridDim.x; i += 32) t += __ldcg(epart + (size_t)cc * gridDim.x + i);
                t = warp_sum(t);
                if ((tid & 31) == 0) alpha_step(fold.st + cc, t, fold.scale);
            }
            if (tid == 0) fold.cnt[0] = 0;
        }
    }
}

}  // namespace hom
