// hom_lines.cuh -- the persistent TMA-staged n2 pass and fused MINRES n1 pass
// (FP32) at the lengths of the line engine (hom_fft.cuh) whose tiles TMA boxes can
// move: all but 375 and 405 in the n2 pass, all but 270, 300, 324, 375, 405, 450,
// 486 and 500 in the n1 pass, which run the plain-load kernels.  The kernels of a
// length are reached through x2_line_kernel / x1l_line_kernel, whose tables
// are built in the translation units that include this file.
//
// Why lengths between the powers of two: grids between the powers of two are as common as these
// (the paper's own are 90, 108 and 160).  The runtime Stockham engine with
// plain loads, which ran them, divides by run-time values for every butterfly,
// holds two buffers per tile and overlaps nothing with its loads: at 192^3 the
// n2 pass took 187 us (65 here; 50 is the copy rate) and the fused n1 pass
// 649 us (173 here), at 108^3 39 (14) and 147 us (38).
#pragma once
#include "hom_passes.cuh"

namespace hom {

// Steps 1-3 of the fused pass (see k_x1_lanczos) on the tile of columns [g0, g0
// + T) held in buf, element e of line l at buf[e * L + l], L = 6 T; the GRP
// threads of the transform group call it.  Everything but n2, n3 is known at
// compile time, and a thread keeps one column, so that its part of xi (axes 2
// and 3), the Parseval weight and the addresses are formed once per tile.
template <typename R, int N, int T, int GRP>
__device__ __forceinline__ void x1_lanczos_line(const Geometry &g, cpx<R> *buf, int g0, const LzCoef<R> &c,
                                                const cpx<R> *__restrict__ uk, const cpx<R> *__restrict__ um,
                                                cpx<R> *__restrict__ un, Acc<R> &acc, MinresState *dst) {
    constexpr int NC = 6, L = NC * T, NT = N * T, ES = GRP / T;   // ES frequencies at once
    const cpx<R> *tw = reinterpret_cast<const cpx<R> *>(g.ax[0].tw);
    line_fft<R, -1, N>(buf, L, L, tw, GRP);
    const int t = threadIdx.x % T, e0 = threadIdx.x / T;
    const int col = g0 + t, H = g.h;
    if (e0 < ES && col < g.n2 * H) {
        const int k2 = col / H, k3 = col - k2 * H;
        const R w = (R)pweight(k3, g.n3);
        // mode of the column: 0 a Nyquist index of axis 2 or 3, else 1
        const bool nyq = 2 * k2 == g.n2 || 2 * k3 == g.n3;
        const R m1 = __ldg(reinterpret_cast<const R *>(g.M[1]) + k2), m2 = __ldg(reinterpret_cast<const R *>(g.M[2]) + k3);
        const R m12 = m1 * m2;
        const R d1 = __ldg(reinterpret_cast<const R *>(g.D[1]) + k2) * m2;
        const R d2 = __ldg(reinterpret_cast<const R *>(g.D[2]) + k3) * m1;
        const R *D0 = reinterpret_cast<const R *>(g.D[0]), *M0 = reinterpret_cast<const R *>(g.M[0]);
        const size_t i0 = (size_t)(g0 / T) * krylov_tile(N, T) + t;
#pragma unroll 1
        for (int e = e0; e < N; e += ES) {
            const size_t i = i0 + e * T;
            cpx<R> *sp = buf + e * L + t * NC;
            cpx<R> v[NC], q[3], u[3], uo[3];
#pragma unroll
            for (int c3 = 0; c3 < 3; ++c3) {
                u[c3] = uk[i + c3 * NT];
                uo[c3] = um[i + c3 * NT];
            }
            const R m0 = __ldg(&M0[e]);
            GammaE<R> ge;
            ge.e0 = __ldg(&D0[e]) * m12;
            ge.e1 = d1 * m0;
            ge.e2 = d2 * m0;
            const R n2 = ge.e0 * ge.e0 + ge.e1 * ge.e1 + ge.e2 * ge.e2;
            ge.mode = (nyq || 2 * e == N || !(n2 > (R)0)) ? 0 : 1;
            if (col == 0 && e == 0) ge.mode = 2;
            const R inv = inv_norm(n2);
            ge.e0 *= inv;
            ge.e1 *= inv;
            ge.e2 *= inv;
#pragma unroll
            for (int p = 0; p < 3; ++p) Six<R>::load_pair(sp, p, v[2 * p], v[2 * p + 1]);
            gamma_to_q<R>(g, ge, v, q);
#pragma unroll
            for (int c3 = 0; c3 < 3; ++c3) {
                q[c3] = mk<R>(c.cp * q[c3].x + c.cu * u[c3].x + c.cv * uo[c3].x,
                              c.cp * q[c3].y + c.cu * u[c3].y + c.cv * uo[c3].y);
            }
            if (c.dc && ge.mode == 2) dc_lanczos<R>(dst, g.mask0, q);
#pragma unroll
            for (int c3 = 0; c3 < 3; ++c3) {
                acc.add_prod(w * q[c3].x, q[c3].x);
                acc.add_prod(w * q[c3].y, q[c3].y);
                un[i + c3 * NT] = q[c3];
            }
            gamma_from_q<R>(g, ge, q, v);
#pragma unroll
            for (int p = 0; p < 3; ++p) Six<R>::store_pair(sp, p, v[2 * p], v[2 * p + 1]);
        }
    }
    // (the columns beyond the last hold zeros: TMA fills them, and a DFT keeps them)
    group_sync(GRP);
    line_fft<R, 1, N>(buf, L, L, tw, GRP);
}

// Held to 64 registers (CTAs of 128 to 256 threads, as many as the ring's
// shared memory leaves room for) except where the plan needs more, and from 225
// up, where that room is two or three CTAs anyway: there the twiddles stay in
// registers across the loop (141 against 146 us at 256^3, 118 against 127 at
// 240^3; at 192^3 68 against 66).
// At 512 the register engine runs the same plan, at 64 registers: its stages have no
// idle threads to tell apart.  The tiles' rows are 64 bytes there, half of the lines
// they come from, and neighbouring tiles find the other half in L2 only as long as
// their CTAs stay together: on the line engine the pass read 0.96 to 0.99 GB of DRAM
// at 256 x 512 x 256 where the register engine reads the 0.81 it needs, and took 0.36
// against 0.275 ms, 1.9 against 1.06 at 512^3.  (At 256, whose rows are whole lines,
// the line engine is the faster, 141 against 148 us at 256^3.)
template <int N> constexpr bool x2_register_engine() { return N == 512; }

template <typename R, int S, int N>
__global__ void __launch_bounds__(512, LinePlan<N>::E <= 16 && (N < 225 || x2_register_engine<N>()) ? 2 : 1) k_x2_tma(Geometry g, const __grid_constant__ CUtensorMap tm, int qtiles,
                                            const MinresState *state) {
    pdl_release();
    pdl_wait();   // predecessor complete (programmatic launch in the MINRES graph)
    if constexpr (x2_register_engine<N>()) static_assert(LinePlan<N>::TPL == N / FastPlan<N>::E, "every thread in the transform");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar[kX2MaxStages];
    const int T = g.tile2, NS = g.x2_stages;
    const int ntiles = g.n1 * g.nb * qtiles;   // stacked cases along k1
    const int tpc = g.n1 * qtiles;             // tiles per case
    // next tile of this CTA's sequence whose case is still iterating
    auto live_from = [&](int t) {
        while (t < ntiles && skip_case(state, t / tpc)) t += gridDim.x;
        return t;
    };
    cpx<R> *const base = reinterpret_cast<cpx<R> *>(smem_raw);
    const int per = N * T;   // stage s starts at base + s * per
    const uint32_t bytes = (uint32_t)(per * sizeof(cpx<R>));
    const bool leader = threadIdx.x == 0;
    if (leader) {
        for (int q = 0; q < NS; ++q) mbar_init(&bar[q], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // NS-stage ring: the leader keeps NS - 1 tiles in flight ahead of the one
    // being transformed (tile j of the sequence in stage j mod NS)
    int tile = live_from(blockIdx.x);
    int ahead = tile, issued = 0;   // next tile to load, tiles loaded (leader)
    auto issue = [&]() {
        const int q = issued % NS;
        mbar_expect_tx(&bar[q], bytes);
        tma_load_rows_3d(base + q * per, &tm, (ahead % qtiles) * T, N, g.box2, ahead / qtiles, T * (int)sizeof(cpx<R>),
                         &bar[q]);
        ++issued;
        ahead = live_from(ahead + gridDim.x);
    };
    if (leader)
        for (int q = 0; q < NS - 1 && ahead < ntiles; ++q) issue();
    const cpx<R> *tw = reinterpret_cast<const cpx<R> *>(g.ax[1].tw);
    for (int i = 0; tile < ntiles; ++i) {
        const int q = i % NS;
        if (leader && ahead < ntiles) {
            bulk_wait_read_all();   // the store of the tile that used this stage has read it
            issue();
        }
        const bool ok = mbar_wait_bounded(&bar[q], (uint32_t)(i / NS) & 1u);
        if (__syncthreads_or(!ok)) {
            if (leader) {   // record, then wait (bounded) for this CTA's loads in flight
                atomicExch(g.err, 1);
                for (int m = i; m < issued; ++m) mbar_wait_bounded(&bar[m % NS], (uint32_t)(m / NS) & 1u);
                bulk_wait_all();
            }
            return;
        }
        cpx<R> *buf = base + q * per;
        if constexpr (x2_register_engine<N>()) fast_fft<R, S, N>(buf, T, T, tw);
        else line_fft<R, S, N>(buf, T, T, tw);
        fence_proxy_async_smem();
        __syncthreads();
        if (leader) {
            tma_store_rows_3d(&tm, (tile % qtiles) * T, N, g.box2, tile / qtiles, buf, T * (int)sizeof(cpx<R>));
            bulk_commit();
        }
        tile = live_from(tile + gridDim.x);
    }
    if (leader) bulk_wait_all();
}

// OR of a predicate over the n threads that use named barrier ID
template <int ID>
__device__ __forceinline__ bool group_or(bool v, int n) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, %2, %3, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(ID), "r"(n)
        : "memory");
    return r != 0;
}

// The lagged update of step k-1 by the lagged-update warps (named barrier
// 2) of the fused n1 pass, over the Krylov blocks of the CTA's tiles whose
// case has one:
//   w_{k-1} = (u_{k-1} / beta_{k-1} - delta w_{k-2} - eps w_{k-3}) / gamma
// over the slot of w_{k-3}, and on every third step the deferred x update.
// The blocks are cut into items of kX1LagChunk bytes; one thread brings an
// item's operands (u_{k-1}, w_{k-2}, w_{k-3}, and x on an x step) into a
// ring of S stages with untiled bulk copies, S items ahead, and the warps
// update it from shared memory and store w_{k-1} (and x) to HBM.  The update is the same on every real number,
// so it runs on 16-byte vectors.  Returns false after a bounded wait ran
// out (the copies in flight have been waited for, bounded).
template <typename R, int grp, int NLAG, typename LiveFrom>
__device__ __forceinline__ bool x1_lagged(const Geometry &g, const LzCoef<R> *scoef, LiveFrom live_from, int ntiles,
                                          int tpc, int per, unsigned char *ring, uint64_t *lbar,
                                          const cpx<R> *__restrict__ um, const cpx<R> *__restrict__ wa,
                                          cpx<R> *__restrict__ wb, cpx<R> *__restrict__ x) {
    using V = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
    constexpr int NR = 16 / sizeof(R);
    const int S = g.x1_lag_stages;
    const int lt = threadIdx.x - grp;
    const long long pbytes = (long long)per * sizeof(cpx<R>);
    auto next_tile = [&](int t) {
        t = live_from(t);
        while (t < ntiles && !scoef[t / tpc].lagged) t = live_from(t + gridDim.x);
        return t;
    };
    auto base_of = [&](int t) {   // byte offset of tile t's block in each Krylov vector
        return ((long long)(t / tpc) * g.kvec + (long long)(t % tpc) * per) * (long long)sizeof(cpx<R>);
    };
    int pt = next_tile(blockIdx.x), ct = pt;   // producer / consumer cursors (tile, byte offset)
    long long po = 0, co = 0;
    int issued = 0;                            // items issued (thread lt = 0)
    auto issue = [&]() {
        const int s = issued % S;
        const uint32_t nb = (uint32_t)(pbytes - po < kX1LagChunk ? pbytes - po : kX1LagChunk);
        const long long o = base_of(pt) + po;
        unsigned char *st = ring + (size_t)s * 4 * kX1LagChunk;
        const bool xs = scoef[pt / tpc].xstep;
        mbar_expect_tx(&lbar[s], (xs ? 4 : 3) * nb);
        bulk_load(st, reinterpret_cast<const char *>(um) + o, nb, &lbar[s]);
        bulk_load(st + kX1LagChunk, reinterpret_cast<const char *>(wa) + o, nb, &lbar[s]);
        bulk_load(st + 2 * kX1LagChunk, reinterpret_cast<const char *>(wb) + o, nb, &lbar[s]);
        if (xs) bulk_load(st + 3 * kX1LagChunk, reinterpret_cast<const char *>(x) + o, nb, &lbar[s]);
        ++issued;
        po += kX1LagChunk;
        if (po >= pbytes) {
            po = 0;
            pt = next_tile(pt + gridDim.x);
        }
    };
    if (lt == 0)
        for (int s = 0; s < S && pt < ntiles; ++s) issue();
    int n = 0;
    for (; ct < ntiles; ++n) {
        const int s = n % S;
        const bool got = mbar_wait_bounded(&lbar[s], (uint32_t)(n / S) & 1u);
        if (group_or<2>(!got, NLAG)) {
            if (lt == 0) {   // record, then wait (bounded) for the items in flight
                atomicExch(g.err, 1);
                for (int m = n; m < issued; ++m) mbar_wait_bounded(&lbar[m % S], (uint32_t)(m / S) & 1u);
            }
            return false;
        }
        const LzCoef<R> c = scoef[ct / tpc];
        const int nv = (int)((pbytes - co < kX1LagChunk ? pbytes - co : kX1LagChunk) / 16);
        const long long o = base_of(ct) + co;
        const V *su = reinterpret_cast<const V *>(ring + (size_t)s * 4 * kX1LagChunk);
        const V *sa = su + kX1LagChunk / 16, *sb = su + 2 * (kX1LagChunk / 16), *sx = su + 3 * (kX1LagChunk / 16);
        V *gb = reinterpret_cast<V *>(reinterpret_cast<char *>(wb) + o);
        V *gx = reinterpret_cast<V *>(reinterpret_cast<char *>(x) + o);
        if (c.xstep) {
            for (int j = lt; j < nv; j += NLAG) {
                V vu = su[j], va = sa[j], vb = sb[j], vx = sx[j], vn;
                const R *u = reinterpret_cast<const R *>(&vu);
                const R *a = reinterpret_cast<const R *>(&va);
                const R *b = reinterpret_cast<const R *>(&vb);
                R *wn = reinterpret_cast<R *>(&vn);
                R *xx = reinterpret_cast<R *>(&vx);
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    wn[r] = (u[r] * c.ib - c.d * a[r] - c.e * b[r]) * c.ig;
                    xx[r] += c.t2 * b[r] + c.t1 * a[r] + c.tau * wn[r];
                }
                gb[j] = vn;
                gx[j] = vx;
            }
        } else {
            for (int j = lt; j < nv; j += NLAG) {
                V vu = su[j], va = sa[j], vb = sb[j];
                const R *u = reinterpret_cast<const R *>(&vu);
                const R *a = reinterpret_cast<const R *>(&va);
                R *b = reinterpret_cast<R *>(&vb);
#pragma unroll
                for (int r = 0; r < NR; ++r) b[r] = (u[r] * c.ib - c.d * a[r] - c.e * b[r]) * c.ig;
                gb[j] = vb;
            }
        }
        co += kX1LagChunk;
        if (co >= pbytes) {
            co = 0;
            ct = next_tile(ct + gridDim.x);
        }
        asm volatile("bar.sync 2, %0;" ::"n"(NLAG) : "memory");   // stage s is read
        if (lt == 0 && pt < ntiles) issue();
    }
    return true;
}

// persistent TMA-staged form (FP32, the line engine's lengths), warp-
// specialised.  The first g.grp1l threads (the transform group, named
// barrier 1) take the work tiles: each comes and goes by TMA, double-
// buffered as in k_x1_tma, and the Lanczos step reads u_k and u_{k-1}
// (bulk-prefetched into L2 at the tile's start) and writes u_{k+1} with
// plain coalesced accesses.  The last one or two warps (x1l_lag_threads) run
// the lagged w update (and on one step in three the deferred x update) on
// the same tiles' Krylov blocks, streaming u_{k-1}, w_{k-2}, w_{k-3} (and x)
// while the transform group works in shared memory; the two groups share no
// written data (u_{k+1} has its own buffer), so they never wait on each
// other.  (Prefetching the next tile's blocks into L2 was measured to double
// the DRAM reads: the lines were evicted before use; the current tile's are
// used within microseconds.)  Tiles are numbered case-major over the stacked
// batch; tiles of converged cases are skipped; each transform thread keeps
// the running sum of a case, reduced over its warp into shared memory at the
// case's last tile, and the CTA writes one partial per case (partials[case * gridDim + block]).
template <typename R, int N>
__global__ void __launch_bounds__(x1l_threads(N, LinePlan<N>::TPL),
                                  LinePlan<N>::E > 16 ? 2 : (x1l_threads(N, LinePlan<N>::TPL) <= 192 ? 4 : 3))
    k_x1_lanczos_tma(Geometry g, const __grid_constant__ CUtensorMap tspec, const cpx<R> *__restrict__ uk,
                     const cpx<R> *__restrict__ um, cpx<R> *__restrict__ un, const cpx<R> *__restrict__ wa,
                     cpx<R> *__restrict__ wb, cpx<R> *__restrict__ x, const MinresState *state,
                     double *__restrict__ partials, Fold fold) {
    pdl_release();
    pdl_wait();   // predecessor complete (programmatic launch in the MINRES graph)
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ __align__(8) uint64_t lbar[kX1LagMaxStages];
    __shared__ double sacc[kNbMax * (kX1Group / 32)];   // ||u_{k+1}||^2 of each case, one running sum a warp
    __shared__ LzCoef<R> scoef[kNbMax];   // each case's coefficients, converted once
    constexpr int NC = 6;
    constexpr int T = x1l_cols(N, LinePlan<N>::TPL), L = NC * T, GRP = x1l_group(N, LinePlan<N>::TPL);
    const int cols = g.n2 * g.h;
    const int tpc = (cols + T - 1) / T;   // tiles per case
    const int ntiles = tpc * g.nb;
    constexpr int kper = krylov_tile(N, T);
    constexpr int sper = (N * L + 15) / 16 * 16;   // stage stride: a multiple of 128 bytes (FP32)
    constexpr int box = tma_box_rows(N, L * (int)sizeof(cpx<R>));
    constexpr uint32_t bytes = (uint32_t)(N * L * sizeof(cpx<R>));
    cpx<R> *base = reinterpret_cast<cpx<R> *>(smem_raw);
    const bool leader = threadIdx.x == 0;
    const bool xform = threadIdx.x < GRP;
    auto live_from = [&](int t) {
        while (t < ntiles && skip_case(state, t / tpc)) t += gridDim.x;
        return t;
    };
    if (threadIdx.x < kNbMax * (kX1Group / 32)) sacc[threadIdx.x] = 0.0;
    if (threadIdx.x < g.nb) scoef[threadIdx.x] = lz_coef<R>(state + threadIdx.x);
    if (leader) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        for (int q = 0; q < kX1LagMaxStages; ++q) mbar_init(&lbar[q], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (!xform) {
        x1_lagged<R, GRP, x1l_lag_threads(GRP)>(g, scoef, live_from, ntiles, tpc, kper, smem_raw + 2 * g.stage1l, lbar, um, wa, wb, x);
    } else {
        double run = 0.0;   // this thread's ||u_{k+1}||^2 of the running case
        int tile = live_from(blockIdx.x);
        if (leader && tile < ntiles) {
            mbar_expect_tx(&bar[0], bytes);
            tma_load_rows_2d(base, &tspec, NC * T * (tile % tpc), N * (tile / tpc), N, box, L * (int)sizeof(cpx<R>),
                             &bar[0]);
        }
        for (int i = 0; tile < ntiles; ++i) {
            const int s = i & 1;
            const int next = live_from(tile + gridDim.x);
            if (leader && next < ntiles) {
                bulk_wait_read_all();   // the store of the tile that used stage s^1 has read it
                mbar_expect_tx(&bar[s ^ 1], bytes);
                tma_load_rows_2d(base + (s ^ 1) * sper, &tspec, NC * T * (next % tpc), N * (next / tpc), N, box,
                                 L * (int)sizeof(cpx<R>), &bar[s ^ 1]);
            }
            const bool ok = mbar_wait_bounded(&bar[s], (i >> 1) & 1);
            if (group_or<1>(!ok, GRP)) {
                if (leader) {   // record, then wait (bounded) for this CTA's loads in flight
                    atomicExch(g.err, 1);
                    mbar_wait_bounded(&bar[s], (i >> 1) & 1);
                    if (next < ntiles) mbar_wait_bounded(&bar[s ^ 1], ((i + 1) >> 1) & 1);
                }
                break;
            }
            const int cs = tile / tpc, tc = tile - cs * tpc;
            const size_t ko = (size_t)cs * g.kvec;
            if (leader && g.x1_l2pf) {   // this tile's u_k and u_{k-1} blocks into L2 for the Lanczos step
                bulk_prefetch_l2(uk + ko + (size_t)tc * kper, (uint32_t)(kper * sizeof(cpx<R>)));
                bulk_prefetch_l2(um + ko + (size_t)tc * kper, (uint32_t)(kper * sizeof(cpx<R>)));
            }
            const LzCoef<R> c = scoef[cs];
            cpx<R> *buf = base + s * sper;
            // a tile's products as two floats, the tiles in FP64: two floats over all
            // tiles of a case lose 1e-13 of the thread's sum (36 tiles), 2e-15 so
            Acc<R> acc;
            x1_lanczos_line<R, N, T, GRP>(g, buf, tc * T, c, uk + ko, um + ko, un + ko, acc, fold.st + cs);
            run += acc.value();
            if (next >= ntiles || next / tpc != cs) {   // the last tile of the case here
                const double ws = warp_sum(run);
                if ((threadIdx.x & 31) == 0) sacc[cs * (kX1Group / 32) + (threadIdx.x >> 5)] += ws;
                run = 0.0;
            }
            fence_proxy_async_smem();
            group_sync(GRP);
            if (leader) {
                tma_store_rows_2d(&tspec, NC * T * tc, N * cs, N, box, buf, L * (int)sizeof(cpx<R>));
                bulk_commit();
            }
            tile = next;
        }
        if (leader) bulk_wait_all();
    }
    __syncthreads();   // both groups done
    // the cases' sums, and the last CTA's Givens steps, one case a warp: a
    // stacked batch of six coarse cells spends more time here than in its
    // tiles if one thread takes the cases in turn
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int cc = warp; cc < g.nb; cc += nw) {
        if (lane == 0) {
            double v = 0.0;
            for (int i = 0; i < kX1Group / 32; ++i) v += sacc[cc * (kX1Group / 32) + i];
            partials[cc * gridDim.x + blockIdx.x] = v;
            __threadfence();
        }
    }
    if (fold.cnt && last_of(fold.cnt + 2 * kNbMax, gridDim.x)) {   // Givens step of every case
        for (int cc = warp; cc < g.nb; cc += nw) {
            double v = 0.0;
            for (int i = lane; i < (int)gridDim.x; i += 32) v += __ldcg(partials + (size_t)cc * gridDim.x + i);
            v = warp_sum(v);
            if (lane == 0) givens_step(fold.st + cc, v);
        }
        if (threadIdx.x == 0) fold.cnt[2 * kNbMax] = 0;
    }
}

}  // namespace hom
