// net_tc.cu -- periodic 3x3x3 convolution as an implicit GEMM on the 5th-
// generation tensor cores: tcgen05.mma (kind::f16, BF16 operands, FP32
// accumulator in tensor memory), issued by one thread, completion tracked on
// mbarriers with tcgen05.commit, the result read back with tcgen05.ld.
// Kernels: column marches for up to 80 output channels (k_conv3_col and the
// weight gradient k_wgrad3_col), halo bricks for more (k_conv3_tcp, k_conv3_tcd,
// k_conv3_tch), and for grids that bricks do not tile the gathering kernel
// k_conv3_tc, described here.
//
// CTA tile: M = 128 output voxels x N = all output channels (<= 256, a
// multiple of 16) x K = 27 taps x input channels, consumed 64 K at a time
// through a 4-stage ring.  Warp-specialised: four producer warps gather the
// operands with cp.async (two chunks in flight per thread), fence them for
// the tensor core and arrive on the stage's "full" barrier; a fifth warp
// waits on it, issues the MMAs and commits to the stage's "empty" barrier,
// which the producers wait on before reusing the stage.
// Each K chunk is staged by cp.async (16-byte rows, the gathered input rows
// with periodic wrap and the half-resolution second source) into the
// canonical no-swizzle K-major layout of the MMA:
// core matrices of 8 rows x 16 bytes, K-adjacent core matrices LBO = 128 B
// apart, 8-row groups SBO = 1024 B apart.
//
// Every wait is bounded; on a timeout the kernel records it in *ConvArgs::err,
// waits (bounded) for its own MMAs, frees its tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <initializer_list>

#include "net_internal.h"
#include "per_device.h"

namespace hnet {

namespace {

constexpr int kProducers = 128;   // 4 warps: operand staging, then the epilogue (one TMEM lane quarter each)
constexpr int kThreads = kProducers + 32;   // + 1 warp that issues the MMAs
constexpr int kBM = 128;          // M per CTA (tcgen05 M = 128, cta_group::1)
constexpr int kBK = 64;           // K elements per stage (4 MMAs of K = 16)
constexpr int kStages = 4;
constexpr int kLBO = 128;         // K-adjacent core matrices
constexpr int kSBO = kBK / 8 * 128;   // 8-row groups (kBK/8 K-chunks of 128 B)
constexpr uint32_t kWaitLimit = 1u << 22;

__device__ __forceinline__ uint32_t saddr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(saddr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    for (uint32_t i = 0; i < kWaitLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// The outcome of a wait that every lane of a warp made, the same in all: lanes that
// part after a time-out would meet neither at the collectives that follow a wait
// (tcgen05.ld, __syncwarp) nor, those that stay behind at one, at the block's end.
__device__ __forceinline__ bool warp_agrees(bool ok) { return __all_sync(0xffffffffu, ok); }

// shared-memory matrix descriptor: start >> 4, LBO >> 4, SBO >> 4, version 1
// (bit 46), no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((kLBO >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((kSBO >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ uint32_t instr_desc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// 8 input channels (16 bytes) of K chunk q (K = 8q .. 8q+7) for voxel (b,z,y,x)
__device__ __forceinline__ const __nv_bfloat16 *k8_src(const ConvArgs &a, int cin_s, int b, int z, int y, int x,
                                                      int q) {
    const int k = 8 * q;
    const int t = k / cin_s, ci = k - t * cin_s;
    const int zz = wrapi(z + t / 9 - 1, a.n1), yy = wrapi(y + (t / 3) % 3 - 1, a.n2), xx = wrapi(x + t % 3 - 1, a.n3);
    if (ci < a.c0s) {
        const long long v = (((long long)b * a.n1 + zz) * a.n2 + yy) * a.n3 + xx;
        return a.src0 + v * a.c0s + ci;
    }
    const long long v = (((long long)b * (a.n1 >> 1) + (zz >> 1)) * (a.n2 >> 1) + (yy >> 1)) * (a.n3 >> 1) + (xx >> 1);
    return a.src1 + v * a.c1s + (ci - a.c0s);
}

__global__ void __launch_bounds__(kThreads) k_conv3_tc(ConvArgs a, int ncols) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], done;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = a.cout;
    const int cin_s = a.c0s + a.c1s;
    const int ktot = 27 * cin_s;                       // multiple of 16
    const int nk = (ktot + kBK - 1) / kBK;
    const int a_bytes = kBM / 8 * kSBO;                // 16 KB
    const int b_bytes = N / 8 * kSBO;
    const int stage_bytes = a_bytes + b_bytes;
    const long long V = (long long)a.n1 * a.n2 * a.n3;
    const long long total = V * a.B;
    const long long m0 = (long long)blockIdx.x * kBM;
    constexpr int kMma = kProducers / 32;              // the MMA warp

    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], kProducers);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kMma) {
        // ---- MMA issue (one thread)
        if (lane == 0) {
            int ncommit[kStages] = {};
            const uint32_t idesc = instr_desc(N);
            bool ok = true;
            for (int c = 0; c < nk && ok; ++c) {
                const int s = c % kStages;
                ok = mbar_wait(&full[s], (uint32_t)(c / kStages) & 1u) && !abort_flag;
                if (!ok) break;
                tc_fence_after();
                const uint32_t ab = saddr(smem + s * stage_bytes), bb = ab + a_bytes;
#pragma unroll
                for (int kk = 0; kk < kBK / 16; ++kk)
                    mma_bf16(tmem, smem_desc(ab + kk * 2 * kLBO), smem_desc(bb + kk * 2 * kLBO), idesc,
                             (c > 0 || kk > 0) ? 1u : 0u);
                mma_commit(&empty[s]);
                ++ncommit[s];
            }
            if (ok) {
                mma_commit(&done);
            } else {
                abort_flag = 1;
                atomicExch(a.err, 1);
                // let the issued MMAs drain (bounded) before the accumulator is freed
                for (int s = 0; s < kStages; ++s)
                    if (ncommit[s] > 0) mbar_wait(&empty[s], (uint32_t)(ncommit[s] - 1) & 1u);
            }
        }
        __syncwarp();
    } else {
        // ---- producers: operand staging
        const long long mrow = m0 + tid;
        const bool row_ok = mrow < total;
        int rb = 0, rz = 0, ry = 0, rx = 0;
        if (row_ok) {
            long long r = mrow;
            rx = (int)(r % a.n3); r /= a.n3;
            ry = (int)(r % a.n2); r /= a.n2;
            rz = (int)(r % a.n1); rb = (int)(r / a.n1);
        }
        bool ok = true;
        for (int c = 0; c < nk + kStages - 2 && ok; ++c) {
            if (c < nk) {
                const int s = c % kStages;
                if (c >= kStages) ok = warp_agrees(mbar_wait(&empty[s], (uint32_t)(c / kStages - 1) & 1u) && !abort_flag);
                if (!ok) break;
                unsigned char *base = smem + s * stage_bytes;
                const uint32_t ab = saddr(base), bb = saddr(base + a_bytes);
#pragma unroll
                for (int j = 0; j < kBK / 8; ++j) {
                    const int q = c * (kBK / 8) + j;
                    const bool in = row_ok && 8 * q < ktot;
                    const __nv_bfloat16 *src = in ? k8_src(a, cin_s, rb, rz, ry, rx, q) : a.src0;
                    cp_async16(ab + (tid >> 3) * kSBO + j * kLBO + (tid & 7) * 16, src, in ? 16 : 0);
                }
                for (int i = tid; i < N * (kBK / 8); i += kProducers) {
                    const int n = i / (kBK / 8), j = i - n * (kBK / 8);
                    const int k = 8 * (c * (kBK / 8) + j);
                    const bool in = k < ktot;
                    const int t = in ? k / cin_s : 0, ci = in ? k - t * cin_s : 0;
                    const __nv_bfloat16 *src = a.W + ((long long)t * N + n) * cin_s + ci;
                    cp_async16(bb + (n >> 3) * kSBO + j * kLBO + (n & 7) * 16, src, in ? 16 : 0);
                }
            }
            cp_async_commit();
            // chunk c - (kStages - 2) has landed for this thread: fence it for
            // the tensor core and report it
            cp_async_wait<kStages - 2>();
            const int r = c - (kStages - 2);
            if (r >= 0 && r < nk) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&full[r % kStages])) : "memory");
            }
        }
        cp_async_wait<0>();
        if (!ok) abort_flag = 1;
        // ---- epilogue: all MMAs done -> TMEM -> bias, ReLU -> global
        ok = warp_agrees(ok && mbar_wait(&done, 0u) && !abort_flag);
        if (ok) {
            tc_fence_after();
            const long long m = m0 + tid;
            for (int c0 = 0; c0 < N; c0 += 16) {
                float v[16];
                tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
                if (m < total) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        if (a.bias) v[i] += a.bias[c0 + i];
                        if (a.relu) v[i] = fmaxf(v[i], 0.f);
                    }
                    if (a.out_f32) {
                        float4 *o = reinterpret_cast<float4 *>(a.out_f32 + m * N + c0);
#pragma unroll
                        for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    } else {
                        __nv_bfloat162 h[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                        uint4 *o = reinterpret_cast<uint4 *>(a.out_bf16 + m * N + c0);
                        o[0] = *reinterpret_cast<uint4 *>(&h[0]);
                        o[1] = *reinterpret_cast<uint4 *>(&h[4]);
                    }
                }
            }
        } else if (tid == 0) {
            atomicExch(a.err, 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}


// ---------------------------------------------------------------------------
// Halo-tile variant for grids that a 4 x 4 x 8 brick tiles: the CTA's 128
// output voxels are one brick; for each 16-channel chunk of the input the
// periodic 6 x 6 x 10 halo is loaded once (cp.async), and each tap's A
// operand (128 rows x 16 K) is copied out of it in shared memory, so every
// input row leaves L2 once per CTA instead of once per tap.  One MMA
// (K = 16) per (chunk, tap) stage; A/B in the no-swizzle K-major layout with
// LBO = 128 B, SBO = 256 B.
// ---------------------------------------------------------------------------
constexpr int kHZ = 6, kHY = 6, kHX = 10, kHalo = kHZ * kHY * kHX;   // halo rows
constexpr int kHSt = 4;                      // stage ring
constexpr int kHLag = 2;                     // stages of B loads in flight per thread
constexpr int kHSBO = 256;                   // K = 16: two K core matrices per 8-row group

__device__ __forceinline__ uint64_t smem_desc_h(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((kLBO >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((kHSBO >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

__device__ __forceinline__ void bar_producers() { asm volatile("bar.sync 1, %0;" ::"n"(kProducers) : "memory"); }

__global__ void __launch_bounds__(kThreads) k_conv3_tch(ConvArgs a, int ncols) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[kHSt], empty[kHSt], done;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = a.cout;
    const int cin_s = a.c0s + a.c1s;
    const int nch = cin_s / 16;
    const int nst = nch * 27;                          // stages: (chunk, tap)
    const int a_bytes = kBM / 8 * kHSBO;               // 4 KB
    const int b_bytes = N / 8 * kHSBO;
    const int stage_bytes = a_bytes + b_bytes;
    unsigned char *halo = smem;                        // kHalo rows x 32 B
    unsigned char *ring = smem + kHalo * 32;
    // this CTA's brick
    const int bx3 = a.n3 / 8, by2 = a.n2 / 4, bz1 = a.n1 / 4;
    int r = blockIdx.x;
    const int xb = r % bx3; r /= bx3;
    const int yb = r % by2; r /= by2;
    const int zb = r % bz1;
    const int b = r / bz1;
    const int z0 = zb * 4, y0 = yb * 4, x0 = xb * 8;
    constexpr int kMma = kProducers / 32;

    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < kHSt; ++q) {
            mbar_init(&full[q], kProducers);
            mbar_init(&empty[q], 1);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kMma) {
        if (lane == 0) {
            int ncommit[kHSt] = {};
            const uint32_t idesc = instr_desc(N);
            bool ok = true;
            for (int c = 0; c < nst && ok; ++c) {
                const int q = c % kHSt;
                ok = mbar_wait(&full[q], (uint32_t)(c / kHSt) & 1u) && !abort_flag;
                if (!ok) break;
                tc_fence_after();
                const uint32_t ab = saddr(ring + q * stage_bytes), bb = ab + a_bytes;
                mma_bf16(tmem, smem_desc_h(ab), smem_desc_h(bb), idesc, c > 0 ? 1u : 0u);
                mma_commit(&empty[q]);
                ++ncommit[q];
            }
            if (ok) {
                mma_commit(&done);
            } else {
                abort_flag = 1;
                atomicExch(a.err, 1);
                for (int q = 0; q < kHSt; ++q)
                    if (ncommit[q] > 0) mbar_wait(&empty[q], (uint32_t)(ncommit[q] - 1) & 1u);
            }
        }
        __syncwarp();
    } else {
        // my output row m = tid: brick offsets (bz, by, bx)
        const int bz = tid >> 5, by = (tid >> 3) & 3, bx = tid & 7;
        bool ok = true;
        int stage = 0, arrived = 0;
        auto arrive_upto = [&](int upto) {   // stages [arrived, upto) have landed
            if (arrived < upto) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            for (; arrived < upto; ++arrived)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&full[arrived % kHSt]))
                             : "memory");
        };
        // every producer passes the same named barriers: after a failed wait a
        // thread keeps going through them and only skips the work
        for (int cc = 0; cc < nch; ++cc) {
            // the halo of channel chunk cc (all earlier copies out of it are done)
            bar_producers();
            if (ok) {
                const bool first = cc * 16 < a.c0s;
                for (int h = tid; h < kHalo; h += kProducers) {
                    const int hx = h % kHX, hy = (h / kHX) % kHY, hz = h / (kHX * kHY);
                    const int zz = wrapi(z0 - 1 + hz, a.n1), yy = wrapi(y0 - 1 + hy, a.n2),
                              xx = wrapi(x0 - 1 + hx, a.n3);
                    const __nv_bfloat16 *src;
                    if (first) {
                        const long long v = (((long long)b * a.n1 + zz) * a.n2 + yy) * a.n3 + xx;
                        src = a.src0 + v * a.c0s + cc * 16;
                    } else {
                        const long long v = (((long long)b * (a.n1 >> 1) + (zz >> 1)) * (a.n2 >> 1) + (yy >> 1)) *
                                                (a.n3 >> 1) + (xx >> 1);
                        src = a.src1 + v * a.c1s + (cc * 16 - a.c0s);
                    }
                    cp_async16(saddr(halo + h * 32), src, 16);
                    cp_async16(saddr(halo + h * 32 + 16), src + 8, 16);
                }
            }
            cp_async_commit();
            asm volatile("cp.async.wait_all;" ::: "memory");
            if (ok) arrive_upto(stage);         // B loads of earlier stages completed too
            bar_producers();
            for (int t = 0; t < 27; ++t, ++stage) {
                if (!ok) continue;
                const int q = stage % kHSt;
                if (stage >= kHSt) ok = warp_agrees(mbar_wait(&empty[q], (uint32_t)(stage / kHSt - 1) & 1u) && !abort_flag);
                if (!ok) continue;
                unsigned char *base = ring + q * stage_bytes;
                // A: my row's 16 channels at the tap's halo position
                const int dz = t / 9, dy = (t / 3) % 3, dx = t % 3;
                const int h = ((bz + dz) * kHY + (by + dy)) * kHX + (bx + dx);
                const uint4 lo = *reinterpret_cast<const uint4 *>(halo + h * 32);
                const uint4 hi = *reinterpret_cast<const uint4 *>(halo + h * 32 + 16);
                *reinterpret_cast<uint4 *>(base + (tid >> 3) * kHSBO + (tid & 7) * 16) = lo;
                *reinterpret_cast<uint4 *>(base + (tid >> 3) * kHSBO + kLBO + (tid & 7) * 16) = hi;
                // B: W[t][n][cc*16 .. +16]
                const uint32_t bb = saddr(base + a_bytes);
                for (int i = tid; i < N * 2; i += kProducers) {
                    const int n = i >> 1, j = i & 1;
                    const __nv_bfloat16 *src = a.W + ((long long)t * N + n) * cin_s + cc * 16 + j * 8;
                    cp_async16(bb + (n >> 3) * kHSBO + j * kLBO + (n & 7) * 16, src, 16);
                }
                cp_async_commit();
                cp_async_wait<kHLag>();
                arrive_upto(stage + 1 - kHLag);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (ok) arrive_upto(nst);
        if (!ok) abort_flag = 1;
        ok = warp_agrees(ok && mbar_wait(&done, 0u) && !abort_flag);
        if (ok) {
            tc_fence_after();
            const long long m = (((long long)b * a.n1 + z0 + bz) * a.n2 + y0 + by) * a.n3 + x0 + bx;
            for (int c0 = 0; c0 < N; c0 += 16) {
                float v[16];
                tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (a.bias) v[i] += a.bias[c0 + i];
                    if (a.relu) v[i] = fmaxf(v[i], 0.f);
                }
                if (a.out_f32) {
                    float4 *o = reinterpret_cast<float4 *>(a.out_f32 + m * N + c0);
#pragma unroll
                    for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                } else {
                    __nv_bfloat162 hv[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) hv[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                    uint4 *o = reinterpret_cast<uint4 *>(a.out_bf16 + m * N + c0);
                    o[0] = *reinterpret_cast<uint4 *>(&hv[0]);
                    o[1] = *reinterpret_cast<uint4 *>(&hv[4]);
                }
            }
        } else if (tid == 0) {
            atomicExch(a.err, 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}


// ---------------------------------------------------------------------------
// Halo tiles read in place.  The halo of a 16-channel chunk is stored as
// three copies, one per tap offset dy, each [6 z][4 y][10 x] rows of 16 bytes
// (channels 0-7 and 8-15 in two planes).  In copy dy the row of voxel
// (bz, by, bx) at tap (dz, dy, dx) is (bz + dz) * 40 + by * 10 + bx + dx: the
// 8 voxels of a brick row are 8 consecutive rows (one core matrix), the 16
// row groups (bz, by) lie 160 B apart, and the tap only moves the start.  So
// the A operand of every tap is a canonical K-major layout (SBO = 160 B,
// LBO = one plane) read straight from the halo: no per-tap copies, and the
// 27 MMAs of a chunk follow one another with one handoff per chunk.  B holds
// the chunk's weights for all 27 taps (K-major, N x 32 bytes per tap).
// ---------------------------------------------------------------------------
constexpr int kDY = 4;                           // y rows of one copy
constexpr int kDRows = kHZ * kDY * kHX;          // 240 rows per copy
constexpr int kDPlane = kDRows * 16;             // one channel half of one copy
constexpr int kDHalo = 3 * 2 * kDPlane;          // 23040 B
constexpr int kDSBO = kHX * 16;                  // (bz, by) row groups

__device__ __forceinline__ uint64_t smem_desc_d(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((kDPlane >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((kDSBO >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// the 27 tap MMAs of one chunk: A read in place from the halo copies, B the
// chunk's weights (32 N bytes per tap).  The descriptors are built once; a
// tap only adds its start offset (>> 4) to the address field, which stays
// inside its 14 bits because shared memory ends below 256 KB.
__device__ __forceinline__ void tap_mmas(uint32_t d, uint32_t ab, uint32_t bb, int N, uint32_t idesc, bool acc) {
    const uint64_t ad = smem_desc_d(ab), bd = smem_desc_h(bb);
    const uint64_t bstep = (uint64_t)(2 * N);          // 32 N bytes >> 4
#pragma unroll
    for (int t = 0; t < 27; ++t) {
        constexpr int kRow = kDY * kHX;
        const int off = ((t / 3) % 3) * 2 * kDPlane + ((t / 9) * kRow + t % 3) * 16;
        mma_bf16(d, ad + (uint64_t)(off >> 4), bd + bstep * t, idesc, (acc || t > 0) ? 1u : 0u);
    }
}

__global__ void __launch_bounds__(kThreads) k_conv3_tcd(ConvArgs a, int ncols, int ring) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[2], empty[2], done;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = a.cout;
    const int cin_s = a.c0s + a.c1s;
    const int nch = cin_s / 16;
    const int b_bytes = 27 * 32 * N;
    const int stage_bytes = kDHalo + b_bytes;
    const int bx3 = a.n3 / 8, by2 = a.n2 / 4, bz1 = a.n1 / 4;
    int r = blockIdx.x;
    const int xb = r % bx3; r /= bx3;
    const int yb = r % by2; r /= by2;
    const int zb = r % bz1;
    const int b = r / bz1;
    const int z0 = zb * 4, y0 = yb * 4, x0 = xb * 8;
    constexpr int kMma = kProducers / 32;

    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < 2; ++q) {
            mbar_init(&full[q], kProducers);
            mbar_init(&empty[q], 1);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kMma) {
        if (lane == 0) {
            int ncommit[2] = {0, 0};
            const uint32_t idesc = instr_desc(N);
            bool ok = true;
            for (int cc = 0; cc < nch && ok; ++cc) {
                const int q = cc % ring;
                ok = mbar_wait(&full[q], (uint32_t)(cc / ring) & 1u) && !abort_flag;
                if (!ok) break;
                tc_fence_after();
                const uint32_t ab = saddr(smem + q * stage_bytes), bb = ab + kDHalo;
                tap_mmas(tmem, ab, bb, N, idesc, cc > 0);
                mma_commit(&empty[q]);
                ++ncommit[q];
            }
            if (ok) {
                mma_commit(&done);
            } else {
                abort_flag = 1;
                atomicExch(a.err, 1);
                for (int q = 0; q < 2; ++q)
                    if (ncommit[q] > 0) mbar_wait(&empty[q], (uint32_t)(ncommit[q] - 1) & 1u);
            }
        }
        __syncwarp();
    } else {
        // my halo rows: (copy, row) pairs tid + 128 k of the 3 x 240, with the
        // periodic source voxel of each (full resolution and half resolution)
        constexpr int kMine = (3 * kDRows + kProducers - 1) / kProducers;   // 6
        int vfull[kMine], vhalf[kMine], dst[kMine];
        const int h1 = a.n1 >> 1, h2 = a.n2 >> 1, h3 = a.n3 >> 1;
#pragma unroll
        for (int k = 0; k < kMine; ++k) {
            const int i = tid + k * kProducers;
            const int dy = i / kDRows, row = i - dy * kDRows;
            const int xr = row % kHX, yr = (row / kHX) % kDY, zr = row / (kHX * kDY);
            const int zz = wrapi(z0 - 1 + zr, a.n1), yy = wrapi(y0 - 1 + yr + dy, a.n2),
                      xx = wrapi(x0 - 1 + xr, a.n3);
            vfull[k] = (zz * a.n2 + yy) * a.n3 + xx;
            vhalf[k] = ((zz >> 1) * h2 + (yy >> 1)) * h3 + (xx >> 1);
            dst[k] = dy * 2 * kDPlane + row * 16;
        }
        const __nv_bfloat16 *s0 = a.src0 + (long long)b * a.n1 * a.n2 * a.n3 * a.c0s;
        const __nv_bfloat16 *s1 = a.c1s ? a.src1 + (long long)b * h1 * h2 * h3 * a.c1s : nullptr;
        bool ok = true;
        for (int cc = 0; cc < nch; ++cc) {
            const int q = cc % ring;
            if (!ok) continue;
            if (cc >= ring) ok = warp_agrees(mbar_wait(&empty[q], (uint32_t)(cc / ring - 1) & 1u) && !abort_flag);
            if (!ok) continue;
            unsigned char *st = smem + q * stage_bytes;
            const bool first = cc * 16 < a.c0s;
#pragma unroll
            for (int k = 0; k < kMine; ++k) {
                if (tid + k * kProducers < 3 * kDRows) {
                    const __nv_bfloat16 *src = first ? s0 + (long long)vfull[k] * a.c0s + cc * 16
                                                     : s1 + (long long)vhalf[k] * a.c1s + (cc * 16 - a.c0s);
                    cp_async16(saddr(st + dst[k]), src, 16);
                    cp_async16(saddr(st + dst[k] + kDPlane), src + 8, 16);
                }
            }
            // weights of the chunk, all 27 taps: W[t][n][cc*16 .. +16]
            const uint32_t bb = saddr(st + kDHalo);
            for (int i = tid; i < 54 * N; i += kProducers) {
                const int t = i / (2 * N), rem = i - t * 2 * N, n = rem >> 1, j = rem & 1;
                const __nv_bfloat16 *src = a.W + ((long long)t * N + n) * cin_s + cc * 16 + j * 8;
                cp_async16(bb + t * 32 * N + (n >> 3) * kHSBO + j * kLBO + (n & 7) * 16, src, 16);
            }
            cp_async_commit();
            asm volatile("cp.async.wait_all;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&full[q])) : "memory");
        }
        if (!ok) abort_flag = 1;
        ok = warp_agrees(ok && mbar_wait(&done, 0u) && !abort_flag);
        if (ok) {
            tc_fence_after();
            const int bz = tid >> 5, by = (tid >> 3) & 3, bx = tid & 7;
            const long long m = (((long long)b * a.n1 + z0 + bz) * a.n2 + y0 + by) * a.n3 + x0 + bx;
            for (int c0 = 0; c0 < N; c0 += 16) {
                float v[16];
                tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (a.bias) v[i] += a.bias[c0 + i];
                    if (a.relu) v[i] = fmaxf(v[i], 0.f);
                }
                if (a.out_f32) {
                    float4 *o = reinterpret_cast<float4 *>(a.out_f32 + m * N + c0);
#pragma unroll
                    for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                } else {
                    __nv_bfloat162 hv[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) hv[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                    uint4 *o = reinterpret_cast<uint4 *>(a.out_bf16 + m * N + c0);
                    o[0] = *reinterpret_cast<uint4 *>(&hv[0]);
                    o[1] = *reinterpret_cast<uint4 *>(&hv[4]);
                }
            }
        } else if (tid == 0) {
            atomicExch(a.err, 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// Persistent form of the in-place halo convolution: a CTA keeps the weights
// of all its chunks in shared memory and walks bricks blockIdx.x, +gridDim.x,
// ...  Halo stages (brick, chunk) go through a 2-slot ring and the brick's
// accumulator alternates between two TMEM column ranges, so the loads of
// brick j overlap the MMAs of brick j-1 and the epilogue of brick j-1 runs
// while the loads of brick j are in flight.  Barriers: hfull/hempty per halo
// slot (producers / MMA commit), afull/aempty per accumulator (MMA commit /
// producers after reading it).
__global__ void __launch_bounds__(kThreads) k_conv3_tcp(ConvArgs a, int ncols) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t hfull[2], hempty[2], afull[2], aempty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = a.cout;
    const int cin_s = a.c0s + a.c1s;
    const int nch = cin_s / 16;
    const int w_bytes = nch * 27 * 32 * N;
    unsigned char *halo = smem + w_bytes;              // 2 slots of kDHalo
    const int bx3 = a.n3 / 8, by2 = a.n2 / 4, bz1 = a.n1 / 4;
    const int nbricks = bx3 * by2 * bz1 * a.B;
    const int nb = blockIdx.x < nbricks ? (nbricks - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    constexpr int kMma = kProducers / 32;
    if (nb == 0) return;

    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < 2; ++q) {
            mbar_init(&hfull[q], kProducers);
            mbar_init(&hempty[q], 1);
            mbar_init(&afull[q], 1);
            mbar_init(&aempty[q], kProducers);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kMma) {
        if (lane == 0) {
            int nh[2] = {0, 0}, na[2] = {0, 0};   // commits per barrier
            const uint32_t idesc = instr_desc(N);
            const uint32_t wb = saddr(smem);
            bool ok = true;
            for (int j = 0; j < nb && ok; ++j) {
                const int s = j & 1;
                if (j >= 2) ok = mbar_wait(&aempty[s], (uint32_t)((j >> 1) - 1) & 1u) && !abort_flag;
                if (!ok) break;
                tc_fence_after();
                for (int cc = 0; cc < nch && ok; ++cc) {
                    const int k = j * nch + cc, q = k & 1;
                    ok = mbar_wait(&hfull[q], (uint32_t)(k >> 1) & 1u) && !abort_flag;
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t ab = saddr(halo + q * kDHalo), bb = wb + cc * 27 * 32 * N;
                    tap_mmas(tmem + (uint32_t)(s * N), ab, bb, N, idesc, cc > 0);
                    mma_commit(&hempty[q]);
                    ++nh[q];
                }
                if (!ok) break;
                mma_commit(&afull[s]);
                ++na[s];
            }
            if (!ok) {
                abort_flag = 1;
                atomicExch(a.err, 1);
                for (int q = 0; q < 2; ++q) {
                    if (nh[q] > 0) mbar_wait(&hempty[q], (uint32_t)(nh[q] - 1) & 1u);
                    if (na[q] > 0) mbar_wait(&afull[q], (uint32_t)(na[q] - 1) & 1u);
                }
            }
        }
        __syncwarp();
    } else {
        // my halo rows: (copy, row) pairs tid + 128 k of the 3 x 240
        constexpr int kMine = (3 * kDRows + kProducers - 1) / kProducers;   // 6
        int rz[kMine], ry[kMine], rx[kMine], dst[kMine];
#pragma unroll
        for (int k = 0; k < kMine; ++k) {
            const int i = tid + k * kProducers;
            const int dy = i / kDRows, row = i - dy * kDRows;
            rx[k] = row % kHX - 1;
            ry[k] = (row / kHX) % kDY + dy - 1;
            rz[k] = row / (kHX * kDY) - 1;
            dst[k] = dy * 2 * kDPlane + row * 16;
        }
        const int h1 = a.n1 >> 1, h2 = a.n2 >> 1, h3 = a.n3 >> 1;
        const int bz = tid >> 5, by = (tid >> 3) & 3, bx = tid & 7;
        // weights of every chunk and tap: W[t][n][cc*16 .. +16], joined to the first halo group
        {
            const uint32_t wb = saddr(smem);
            for (int i = tid; i < 54 * N * nch; i += kProducers) {
                const int cc = i / (54 * N), i2 = i - cc * 54 * N;
                const int t = i2 / (2 * N), rem = i2 - t * 2 * N, n = rem >> 1, jj = rem & 1;
                const __nv_bfloat16 *src = a.W + ((long long)t * N + n) * cin_s + cc * 16 + jj * 8;
                cp_async16(wb + (cc * 27 + t) * 32 * N + (n >> 3) * kHSBO + jj * kLBO + (n & 7) * 16, src, 16);
            }
        }
        bool ok = true;
        int vfull[kMine], vhalf[kMine];
        int pb = 0, pz0 = 0, py0 = 0, px0 = 0;              // the previous brick, for its epilogue
        auto epilogue = [&](int j) {                        // brick j's accumulator to the output
            const int s = j & 1;
            ok = warp_agrees(mbar_wait(&afull[s], (uint32_t)(j >> 1) & 1u) && !abort_flag);
            if (!ok) return;
            tc_fence_after();
            const long long m = (((long long)pb * a.n1 + pz0 + bz) * a.n2 + py0 + by) * a.n3 + px0 + bx;
            for (int c0 = 0; c0 < N; c0 += 16) {
                float v[16];
                tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(s * N + c0), v);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (a.bias) v[i] += a.bias[c0 + i];
                    if (a.relu) v[i] = fmaxf(v[i], 0.f);
                }
                if (a.out_f32) {
                    float4 *o = reinterpret_cast<float4 *>(a.out_f32 + m * N + c0);
#pragma unroll
                    for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                } else {
                    __nv_bfloat162 hv[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) hv[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                    uint4 *o = reinterpret_cast<uint4 *>(a.out_bf16 + m * N + c0);
                    o[0] = *reinterpret_cast<uint4 *>(&hv[0]);
                    o[1] = *reinterpret_cast<uint4 *>(&hv[4]);
                }
            }
            tc_fence_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&aempty[s])) : "memory");
        };
        for (int j = 0; j < nb && ok; ++j) {
            int r = (int)blockIdx.x + j * (int)gridDim.x;
            const int xb = r % bx3; r /= bx3;
            const int yb = r % by2; r /= by2;
            const int zb = r % bz1;
            const int b = r / bz1;
            const int z0 = zb * 4, y0 = yb * 4, x0 = xb * 8;
#pragma unroll
            for (int k = 0; k < kMine; ++k) {
                const int zz = wrapi(z0 + rz[k], a.n1), yy = wrapi(y0 + ry[k], a.n2), xx = wrapi(x0 + rx[k], a.n3);
                vfull[k] = (zz * a.n2 + yy) * a.n3 + xx;
                vhalf[k] = ((zz >> 1) * h2 + (yy >> 1)) * h3 + (xx >> 1);
            }
            const __nv_bfloat16 *s0 = a.src0 + (long long)b * a.n1 * a.n2 * a.n3 * a.c0s;
            const __nv_bfloat16 *s1 = a.c1s ? a.src1 + (long long)b * h1 * h2 * h3 * a.c1s : nullptr;
            for (int cc = 0; cc < nch && ok; ++cc) {
                const int k = j * nch + cc, q = k & 1;
                if (k >= 2) ok = warp_agrees(mbar_wait(&hempty[q], (uint32_t)((k >> 1) - 1) & 1u) && !abort_flag);
                if (!ok) break;
                unsigned char *st = halo + q * kDHalo;
                const bool first = cc * 16 < a.c0s;
#pragma unroll
                for (int kk = 0; kk < kMine; ++kk) {
                    if (tid + kk * kProducers < 3 * kDRows) {
                        const __nv_bfloat16 *src = first ? s0 + (long long)vfull[kk] * a.c0s + cc * 16
                                                         : s1 + (long long)vhalf[kk] * a.c1s + (cc * 16 - a.c0s);
                        cp_async16(saddr(st + dst[kk]), src, 16);
                        cp_async16(saddr(st + dst[kk] + kDPlane), src + 8, 16);
                    }
                }
                cp_async_commit();
                if (cc == 0 && j > 0) epilogue(j - 1);   // overlaps the loads just issued
                asm volatile("cp.async.wait_all;" ::: "memory");
                if (!ok) break;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&hfull[q])) : "memory");
            }
            pb = b; pz0 = z0; py0 = y0; px0 = x0;
        }
        if (ok) epilogue(nb - 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (!ok) {
            abort_flag = 1;
            if (tid == 0) atomicExch(a.err, 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// ---------------------------------------------------------------------------
// Column convolution: a CTA marches a tile of 8 x 16 voxels (x, y) through up
// to zl planes of z.  Every input plane (its periodic halo of 10 x 18 voxels,
// one 16-channel chunk at a time) is read once and multiplied for all three
// output planes it reaches: for a tap (dy, dx) one MMA of M = 128 voxels and
// N = 3 c_out, whose B rows are the weights of dz = +1, 0, -1, and whose
// accumulator columns are those of the output planes z-1, z, z+1, side by side
// in tensor memory (plane q at column q c_out).  Nine MMAs a plane and chunk in
// place of 27: reading A (4 KB an MMA) from shared memory bounds the small-N
// products of this network, so a third of the reads is a third of the time.
// The halo of a brick (2.8 loads per voxel) becomes 1.4 (1 + 2/zl).
// Persistent: four warps load planes, one issues the MMAs, four take an item's
// accumulators to the output while the next item fills the other half of the
// tensor memory; a CTA keeps the weights of all chunks where they fit.
// A in place: plane rows of 16 bytes (8 channels), channel halves kPHalf apart;
// the 8 voxels of an x run are one core matrix, y runs 160 B apart, and a tap
// only moves the start.  The plane that a chunk-0 plane reaches first (z+1)
// starts its accumulator with that plane's first tap.
// Measured (64^3 x 8, 16 -> 16 channels, a call with its synchronisation): 76 us
// against 163 with k_conv3_tcp (27 MMAs a brick); 24 us of a call are the
// launch and the synchronisation.  An MMA of these sizes takes 85 to 100 cycles
// whatever its N, which makes 53 us of the nine a plane.
// ---------------------------------------------------------------------------
constexpr int kPX = 8, kPY = 16, kPHX = kPX + 2, kPRows = kPHX * (kPY + 2);   // tile, halo rows
constexpr int kPHalf = kPRows * 16, kPPlane = 2 * kPHalf;
constexpr int kPSlots = 12, kPDepth = 5;   // most halo planes in shared memory, loads in flight
constexpr int kColThreads = 2 * kProducers + 32;   // loads, epilogue, MMA issue

__device__ __forceinline__ uint64_t smem_desc_p(uint32_t addr) {   // K-major: LBO the channel half, SBO the next y
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((kPHalf >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((kPHX * 16 >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

__device__ __forceinline__ int wrapm(int i, int n) {   // any distance
    const int r = i % n;
    return r < 0 ? r + n : r;
}

// the nine taps of one plane: B blocks [j0, j1] (output planes), fresh: block 2
// starts its accumulator
__device__ __forceinline__ void plane_mmas(uint32_t d, uint32_t ab, uint32_t bb, int N, int j0, int j1, bool fresh) {
    const uint64_t ad = smem_desc_p(ab), bd = smem_desc_h(bb);
    const uint64_t bstep = (uint64_t)(6 * N), blk = (uint64_t)(2 * N);   // 96 N and 32 N bytes, >> 4
    const uint32_t idesc = instr_desc((j1 - j0 + 1) * N);
#pragma unroll
    for (int s = 0; s < 9; ++s) {
        const uint64_t as = ad + (uint64_t)((s / 3) * kPHX + s % 3);
        const uint64_t bs = bd + bstep * s;
        if (s == 0 && fresh) {
            if (j0 < 2) mma_bf16(d + j0 * N, as, bs + blk * j0, instr_desc((2 - j0) * N), 1u);
            mma_bf16(d + 2 * N, as, bs + blk * 2, instr_desc(N), 0u);
        } else {
            mma_bf16(d + j0 * N, as, bs + blk * j0, idesc, 1u);
        }
    }
}

// planes: halo planes in shared memory; wslots: chunks' weights there (all nch
// of them: loaded once)
template <int N>
__global__ void __launch_bounds__(kColThreads) k_conv3_col(ConvArgs a, int ncols, int zl, int nplanes, int wslots) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[kPSlots], empty[kPSlots], wempty[2], afull[2], aempty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cin_s = a.c0s + a.c1s, nch = cin_s / 16;
    const bool resident = wslots >= nch;
    constexpr int w_bytes = 27 * 32 * N;
    unsigned char *planes = smem + wslots * w_bytes;
    const int tx = (a.n3 + kPX - 1) / kPX, ty = (a.n2 + kPY - 1) / kPY, tz = (a.n1 + zl - 1) / zl;
    const int items = tx * ty * tz * a.B;
    constexpr int kMma = 2 * kProducers / 32;
    // item -> its first voxel (x0, y0, z0, b) and number of output planes
    auto decode = [&](int it, int &x0, int &y0, int &z0, int &b) {
        x0 = it % tx * kPX; it /= tx;
        y0 = it % ty * kPY; it /= ty;
        z0 = it % tz * zl;
        b = it / tz;
        return a.n1 - z0 < zl ? a.n1 - z0 : zl;
    };

    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < nplanes; ++q) {
            mbar_init(&full[q], kProducers / 32);
            mbar_init(&empty[q], 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(&wempty[q], 1);
            mbar_init(&afull[q], 1);
            mbar_init(&aempty[q], kProducers / 32);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kMma) {
        if (lane == 0) {
            bool ok = true;
            int k = 0, q = 0, c = 0, n = 0;   // stages, slot, chunks and items done
            uint32_t ph = 0;
            for (int it = blockIdx.x; it < items && ok; it += gridDim.x, ++n) {
                int x0, y0, z0, b;
                const int nz = decode(it, x0, y0, z0, b), P = nz + 2;
                if (n >= 2) ok = mbar_wait(&aempty[n & 1], (uint32_t)((n >> 1) - 1) & 1u) && !abort_flag;
                if (!ok) break;
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)((n & 1) * zl * N);
                for (int cc = 0; cc < nch && ok; ++cc, ++c) {
                    const int ws = resident ? cc : c % wslots;
                    const uint32_t wb = saddr(smem + ws * w_bytes);
                    for (int i = 0; i < P; ++i, ++k) {   // input plane z0 - 1 + i reaches outputs i - 2 + j
                        ok = mbar_wait(&full[q], ph) && !abort_flag;
                        if (!ok) break;
                        tc_fence_after();
                        const int j0 = i < 2 ? 2 - i : 0, j1 = nz + 1 - i < 2 ? nz + 1 - i : 2;
                        plane_mmas(acc + (uint32_t)((i - 2) * N), saddr(planes + q * kPPlane), wb, N, j0, j1,
                                   cc == 0 && j1 == 2);
                        mma_commit(&empty[q]);
                        if (++q == nplanes) {
                            q = 0;
                            ph ^= 1;
                        }
                    }
                    if (ok && !resident) mma_commit(&wempty[ws]);
                }
                if (ok) mma_commit(&afull[n & 1]);
            }
            if (!ok) {
                abort_flag = 1;
                atomicExch(a.err, 1);
                if (k > 0) mbar_wait(&empty[(k - 1) % nplanes], (uint32_t)((k - 1) / nplanes) & 1u);
            }
        }
        __syncwarp();
    } else if (tid < kProducers) {
        // my 16-byte pieces of a plane: piece tid + 128 m, (row, channel half)
        constexpr int kMine = (2 * kPRows + kProducers - 1) / kProducers;   // 3
        const int h2 = a.n2 >> 1, h3 = a.n3 >> 1;
        uint32_t dst[kMine];
#pragma unroll
        for (int m = 0; m < kMine; ++m) {
            const int p = tid + m * kProducers;
            dst[m] = saddr(planes) + (p & 1) * kPHalf + (p >> 1) * 16;
        }
        const bool mine2 = tid + 2 * kProducers < 2 * kPRows;
        auto load_weights = [&](int cc, int ws) {   // [tap][3 c_out rows][16 channels] of chunk cc
            const uint32_t wb = saddr(smem + ws * w_bytes);
#pragma unroll 2
            for (int p = tid; p < 54 * N; p += kProducers) {
                const int s = p / (6 * N), r6 = p - s * 6 * N, j = r6 / (2 * N), r2 = r6 - j * 2 * N;
                const int co = r2 >> 1, h = r2 & 1, n = j * N + co;
                const __nv_bfloat16 *src = a.W + (((2 - j) * 9 + s) * N + co) * cin_s + cc * 16 + h * 8;
                cp_async16(wb + s * 96 * N + (n >> 3) * kHSBO + h * kLBO + (n & 7) * 16, src, 16);
            }
        };
        bool ok = true;
        int k = 0, q = 0, c = 0, sent = 0, qs = 0;   // stage, slot, chunk; stages handed over and the next one's slot
        int kprev = 0;                               // first stage of the chunk before
        uint32_t ph = 1;                             // parity of the slot's previous round
        auto arrive = [&]() {                        // my pieces of stage `sent` are in: one arrival a warp
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&full[qs])) : "memory");
            ++sent;
            if (++qs == nplanes) qs = 0;
        };
        if (resident)
            for (int cc = 0; cc < nch; ++cc) load_weights(cc, cc);   // joined to the first plane
        for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
            int x0, y0, z0, b;
            const int P = decode(it, x0, y0, z0, b) + 2;
            int vfull[kMine], vhalf[kMine];
#pragma unroll
            for (int m = 0; m < kMine; ++m) {
                const int p = tid + m * kProducers, row = p >> 1, h = p & 1;
                const int yy = wrapm(y0 - 1 + row / kPHX, a.n2), xx = wrapm(x0 - 1 + row % kPHX, a.n3);
                vfull[m] = (yy * a.n3 + xx) * a.c0s + h * 8;
                vhalf[m] = ((yy >> 1) * h3 + (xx >> 1)) * a.c1s + h * 8;
            }
            const __nv_bfloat16 *s0 = a.src0 + (long long)b * a.n1 * a.n2 * a.n3 * a.c0s;
            const __nv_bfloat16 *s1 = a.c1s ? a.src1 + (long long)b * (a.n1 >> 1) * h2 * h3 * a.c1s : nullptr;
            const int zfirst = wrapm(z0 - 1, a.n1);
            for (int cc = 0; cc < nch && ok; ++cc, ++c) {
                if (!resident) {
                    // the buffer is free once the planes of the chunk that used it are
                    // multiplied: those of them still in flight are handed over first
                    const int need = wslots == 1 ? k : kprev;
                    kprev = k;
                    if (c >= wslots && sent < need) {
                        asm volatile("cp.async.wait_all;" ::: "memory");
                        while (sent < need) arrive();
                    }
                    if (c >= wslots)
                        ok = warp_agrees(mbar_wait(&wempty[c % wslots], (uint32_t)(c / wslots - 1) & 1u) && !abort_flag);
                    if (!ok) break;
                    load_weights(cc, c % wslots);
                }
                const bool first = cc * 16 < a.c0s;
                const int o0 = first ? vfull[0] : vhalf[0], o1 = first ? vfull[1] : vhalf[1];
                const int o2 = first ? vfull[2] : vhalf[2];
                const __nv_bfloat16 *sc = first ? s0 + cc * 16 : s1 + (cc * 16 - a.c0s);
                const long long pstride = first ? (long long)a.n2 * a.n3 * a.c0s : (long long)h2 * h3 * a.c1s;
                int zz = zfirst;
                for (int i = 0; i < P; ++i, ++k) {
                    if (k >= nplanes) ok = warp_agrees(mbar_wait(&empty[q], ph) && !abort_flag);
                    if (!ok) break;
                    const __nv_bfloat16 *src = sc + (first ? zz : zz >> 1) * pstride;
                    if (++zz == a.n1) zz = 0;
                    const uint32_t st = q * kPPlane;
                    cp_async16(dst[0] + st, src + o0, 16);
                    cp_async16(dst[1] + st, src + o1, 16);
                    if (mine2) cp_async16(dst[2] + st, src + o2, 16);
                    cp_async_commit();
                    if (k - sent >= kPDepth - 1) {
                        cp_async_wait<kPDepth - 1>();
                        arrive();
                    }
                    if (++q == nplanes) {
                        q = 0;
                        ph ^= 1;
                    }
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (ok)
            while (sent < k) arrive();
        if (!ok) {
            abort_flag = 1;
            if (tid == 0) atomicExch(a.err, 1);
        }
    } else {
        // epilogue warps: an item's planes while the next item is multiplied
        const int e = tid - kProducers, quarter = warp - kProducers / 32;
        float bias[N == 16 ? 16 : 1];   // a 16-channel output's bias stays in registers
        if constexpr (N == 16) {
#pragma unroll
            for (int i = 0; i < 16; ++i) bias[i] = a.bias ? __ldg(a.bias + i) : 0.f;
        }
        bool ok = true;
        int n = 0;
        const long long plane = (long long)a.n2 * a.n3 * N;
        for (int it = blockIdx.x; it < items && ok; it += gridDim.x, ++n) {
            int x0, y0, z0, b;
            const int nz = decode(it, x0, y0, z0, b);
            ok = warp_agrees(mbar_wait(&afull[n & 1], (uint32_t)(n >> 1) & 1u) && !abort_flag);
            if (!ok) break;
            tc_fence_after();
            const int y = y0 + (e >> 3), x = x0 + (e & 7);
            const bool live = y < a.n2 && x < a.n3;
            long long m = ((((long long)b * a.n1 + z0) * a.n2 + y) * a.n3 + x) * N;
            const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((n & 1) * zl * N);
            for (int p = 0; p < nz; ++p, m += plane) {
#pragma unroll
                for (int c0 = 0; c0 < N; c0 += 16) {
                    float v[16];
                    __syncwarp();
                    tmem_ld16(acc + (uint32_t)(p * N + c0), v);
                    if (live) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            if constexpr (N == 16) v[i] += bias[i];
                            else if (a.bias) v[i] += __ldg(a.bias + c0 + i);
                            if (a.relu) v[i] = fmaxf(v[i], 0.f);
                        }
                        if (a.out_f32) {
                            float4 *o = reinterpret_cast<float4 *>(a.out_f32 + m + c0);
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                        } else {
                            __nv_bfloat162 hv[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) hv[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                            uint4 *o = reinterpret_cast<uint4 *>(a.out_bf16 + m + c0);
                            o[0] = *reinterpret_cast<uint4 *>(&hv[0]);
                            o[1] = *reinterpret_cast<uint4 *>(&hv[4]);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&aempty[n & 1])) : "memory");
        }
        if (!ok) {
            abort_flag = 1;
            if (e == 0) atomicExch(a.err, 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// ---------------------------------------------------------------------------
// Column weight gradient: dW[t][co][ci] = sum_v G[v][co] X[v + d_t][ci] on the
// same 8 x 16 columns, 16 output channels and one 16-channel chunk of the
// input per CTA.  Rows of D are (dx, input channel), 48 of M = 64; its columns
// are (dz, dy, output channel), N = 144: the G planes z+1, z, z-1 of an X plane z,
// each as three copies shifted by dy.  So a plane takes 8 MMAs (K = the tile's
// 128 voxels, 16 at a time) for all 27 taps.  (24 of N = 48, dy in the start of
// A, took 131 us against 126 at 64^3 x 8, 16 -> 16 channels, and leave the
// copies' number to the output channels; one CTA per SM with eight stages in
// flight took 180.  What bounds it is neither: the loads alone, or a eighth of
// the MMAs, take nearly as long.)
// Both operands are MN-major in place: A three copies of the X plane, one per
// dx, [dx][channel half][16 y][8 x] rows of 16 bytes; B a ring of G planes,
// [plane][dy][channel half][16 y][8 x], whose window of three is one run of
// column groups except where the ring wraps (then two MMAs).  D stays in
// tensor memory while the CTA takes its share of columns.  (k_wgrad3_tc, which
// this replaces, copied 27 taps of every voxel between shared buffers: 258 us
// at 64^3 x 8, 16 -> 16 channels.)
// ---------------------------------------------------------------------------
constexpr int kCHalf = kPY * kPX * 16;              // 2048 B: 8 channels of one copy of a plane
constexpr int kCPlane = 6 * kCHalf;                 // three copies of 16 channels (X: dx, G: dy)
constexpr int kCSlots = 3, kCGSlots = 6, kCDepth = 2;   // X planes, G planes (each read for three stages), loads in flight
constexpr int kCPad = 2 * kCHalf;                   // rows 48..63 of A read past the last X slot
constexpr int kCRun = 4;                            // items whose products an accumulator takes at least
constexpr int kCTaps = 48;                          // columns of one G plane: dy, 16 output channels

__device__ __forceinline__ uint64_t smem_desc_c(uint32_t addr) {   // MN-major: LBO along K, SBO along MN
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((128 >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((kCHalf >> 4) & 0x3FFF) << 32) | (1ull << 46);
}
__device__ __forceinline__ uint32_t instr_desc_c(int n) {   // M = 64, both operands MN-major
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | (4u << 24);
}

// zl: planes of a work item; blockIdx = (split, input chunk, 16 output channels)
// The tensor core adds to its FP32 accumulators with about 2^-24 of them lost each
// time, in one direction, so that a sum over many voxels is off in proportion to
// their number (64 -> 64 channels, 64^3 x 8: 19 splits of 110 k voxels 1.2e-4 off the
// FP64 gradient).  So a CTA works through its split in runs of at most `run` items,
// starts the accumulators afresh in each and adds the runs up in FP32 arithmetic in
// its partial sums (7e-6; the first run is stored).  That takes 1853 us there against
// 1774 in one run, and more splits instead, of as few voxels, 2465.  Splits that are
// one run anyway (RUNS false) do without: 143 us against 149 at 16 -> 16 channels.
template <bool RUNS>
__global__ void __launch_bounds__(kThreads, 2) k_wgrad3_col(WgradArgs w, int ncols, int zl, int run) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[kCSlots], empty[kCSlots], done, taken;   // done, taken: once a run
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const ConvArgs &a = w.in;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cin_s = a.c0s + a.c1s, cc = blockIdx.y, split = blockIdx.x, co0 = blockIdx.z * 16;
    unsigned char *xs = smem, *gs = smem + kCSlots * kCPlane + kCPad;
    const int tx = (a.n3 + kPX - 1) / kPX, ty = (a.n2 + kPY - 1) / kPY, tz = (a.n1 + zl - 1) / zl;
    const long long items = (long long)tx * ty * tz * a.B;
    const long long it0 = items * split / w.S, it1 = items * (split + 1) / w.S;
    constexpr int kMma = kProducers / 32;
    if (it0 >= it1) {   // no columns in this split: its partial sums are zero
        for (int i = tid; i < 27 * 16 * 16; i += kThreads) {
            const int ci = i % 16, r = i / 16, co = r % 16, t = r / 16;
            w.partial[(((long long)split * 27 + t) * w.cout + co0 + co) * cin_s + cc * 16 + ci] = 0.f;
        }
        return;
    }
    // runs of a split, alike: their number and items
    const int n = (int)(it1 - it0), nruns = RUNS ? (n + run - 1) / run : 1, per = RUNS ? (n + nruns - 1) / nruns : n;
    auto item_z = [&](long long it) { return (int)(it % tz) * zl; };   // z fastest: neighbours share halo planes
    auto item_nz = [&](long long it) { return a.n1 - item_z(it) < zl ? a.n1 - item_z(it) : zl; };

    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < kCSlots; ++q) {
            mbar_init(&full[q], kProducers / 32);
            mbar_init(&empty[q], 1);
        }
        mbar_init(&done, 1);
        mbar_init(&taken, kProducers / 32);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the pad that A's unused rows read stays finite
    for (int i = tid; i < kCPad / 16; i += kThreads)
        reinterpret_cast<uint4 *>(smem + kCSlots * kCPlane)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kMma) {
        if (lane == 0) {
            bool ok = true;
            int k = 0, q = 0, g0 = 0;   // stage, its slot, ring slot of the item's G plane 0
            uint32_t ph = 0;
            int left = per, r = 0;      // items left of the run, runs done
            for (long long it = it0; it < it1 && ok; ++it) {
                const int nz = item_nz(it);
                if (RUNS && left == 0) {   // the next run: its accumulators once this one's are read
                    mma_commit(&done);
                    ok = mbar_wait(&taken, (uint32_t)r & 1u) && !abort_flag;
                    if (!ok) break;
                    tc_fence_after();
                    left = per;
                    ++r;
                }
                const bool starts = RUNS ? left-- == per : it == it0;
                for (int i = 0; i < nz + 2; ++i, ++k) {   // X plane z0 - 1 + i meets G planes i - 2 + j
                    ok = mbar_wait(&full[q], ph) && !abort_flag;
                    if (!ok) break;
                    tc_fence_after();
                    const int j0 = i < 2 ? 2 - i : 0, j1 = nz + 1 - i < 2 ? nz + 1 - i : 2;
                    const bool fresh = starts && i <= 2;   // block j0 starts its accumulators
                    const int s0 = (g0 + i - 2 + j0) % kCGSlots, left = kCGSlots - s0;   // planes before the ring wraps
                    const int ja = j1 - j0 + 1 > left ? j0 + left - 1 : j1;              // last block of the first run
                    const uint64_t ad = smem_desc_c(saddr(xs + q * kCPlane));
                    const uint64_t b0 = smem_desc_c(saddr(gs + s0 * kCPlane)), b1 = smem_desc_c(saddr(gs));
                    const uint32_t d = tmem + (uint32_t)(j0 * kCTaps), d1 = tmem + (uint32_t)((ja + 1) * kCTaps);
                    const uint32_t n0 = instr_desc_c((ja - j0 + 1) * kCTaps), n1 = instr_desc_c((j1 - ja) * kCTaps);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {   // 16 voxels: two y runs of 128 B
                        const uint64_t o = (uint64_t)(kk * 16);
                        if (fresh && kk == 0) {
                            mma_bf16(d, ad + o, b0 + o, instr_desc_c(kCTaps), 0u);
                            if (ja > j0)
                                mma_bf16(d + kCTaps, ad + o, b0 + o + (uint64_t)(kCPlane >> 4),
                                         instr_desc_c((ja - j0) * kCTaps), 1u);
                        } else {
                            mma_bf16(d, ad + o, b0 + o, n0, 1u);
                        }
                        if (j1 > ja) mma_bf16(d1, ad + o, b1 + o, n1, 1u);
                    }
                    mma_commit(&empty[q]);
                    if (++q == kCSlots) {
                        q = 0;
                        ph ^= 1;
                    }
                }
                g0 = (g0 + nz) % kCGSlots;
            }
            if (ok) {
                mma_commit(&done);
            } else {
                abort_flag = 1;
                atomicExch(a.err, 1);
                if (k > 0) mbar_wait(&empty[(k - 1) % kCSlots], (uint32_t)((k - 1) / kCSlots) & 1u);
            }
        }
        __syncwarp();
    } else {
        // my pieces of a plane's copies: piece p = tid + 128 m is (copy, y, x, half)
        constexpr int kMine = 3 * kPY * kPX * 2 / kProducers;   // 6
        static_assert(kMine * kProducers == 3 * kPY * kPX * 2, "whole pieces");
        const bool first = cc * 16 < a.c0s;
        const int sh = first ? 0 : 1;
        const int m1 = a.n1 >> sh, m2 = a.n2 >> sh, m3 = a.n3 >> sh;
        const int cs = first ? a.c0s : a.c1s;
        const __nv_bfloat16 *sbase = first ? a.src0 + cc * 16 : a.src1 + (cc * 16 - a.c0s);
        int off[kMine], goff[kMine];
        uint32_t dst[kMine];
#pragma unroll
        for (int m = 0; m < kMine; ++m) {
            const int p = tid + m * kProducers, v = (p >> 1) % (kPY * kPX), copy = p / (2 * kPY * kPX);
            dst[m] = (2 * copy + (p & 1)) * kCHalf + v * 16;
        }
        bool ok = true;
        int k = 0, q = 0, gq = 0, sent = 0, qs = 0;   // stage, X slot, G slot; stages handed over and the next one's slot
        uint32_t ph = 1;                              // parity of the slot's previous round
        auto arrive = [&]() {                         // my pieces of stage `sent` are in: one arrival a warp
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&full[qs])) : "memory");
            ++sent;
            if (++qs == kCSlots) qs = 0;
        };
        // the run's accumulators: M = 64, rows 16 w .. 16 w + 15 in lanes 0..15 of warp
        // w's quarter; warp w holds dx = w
        float *const out = w.partial + (((long long)split * 27 + (warp < 3 ? warp : 0)) * w.cout + co0) * cin_s + cc * 16 + (lane & 15);
        const long long tstride = (long long)w.cout * cin_s;
        auto take = [&](bool add) {
            const bool mine = warp < 3 && lane < 16;
            auto at = [&](int jd) { return out + ((2 - jd / 3) * 9 + jd % 3 * 3) * tstride; };   // (dz block, dy copy)
            float sum[16];   // of the runs before, a copy ahead
            auto fetch = [&](int jd) {
#pragma unroll
                for (int i = 0; i < 16; ++i) sum[i] = at(jd)[(long long)i * cin_s];
            };
            if (add && mine) fetch(0);
#pragma unroll 1
            for (int jd = 0; jd < 9; ++jd) {
                float v[16];
                __syncwarp();
                tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(jd * 16), v);
                if (mine) {
                    if (add) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] += sum[i];
                        if (jd < 8) fetch(jd + 1);
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) at(jd)[(long long)i * cin_s] = v[i];
                }
            }
        };
        const long long pstride = (long long)m2 * m3 * cs, gstride = (long long)a.n2 * a.n3 * w.cout;
        int left = per, nr = 0;   // items left of the run, runs done
        for (long long it = it0; it < it1 && ok; ++it, --left) {
            if (RUNS && left == 0) {   // the run before is loaded: hand it over, and take its sums
                asm volatile("cp.async.wait_all;" ::: "memory");
                while (sent < k) arrive();
                ok = warp_agrees(mbar_wait(&done, (uint32_t)nr & 1u) && !abort_flag);
                if (!ok) break;
                tc_fence_after();
                take(nr > 0);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&taken)) : "memory");
                left = per;
                ++nr;
            }
            const int z0 = item_z(it), nz = item_nz(it);
            long long r = it / tz;
            const int x0 = (int)(r % tx) * kPX; r /= tx;
            const int y0 = (int)(r % ty) * kPY;
            const int b = (int)(r / ty);
            // X row y of copy dx: X[y][x + dx]; G row y of copy dy: G[y - dy][x]; both zero
            // for y or x beyond the grid (each X row, each G column counts once, and
            // an infinite X or G there must not meet the other's zero)
            uint32_t live = 0;
#pragma unroll
            for (int m = 0; m < kMine; ++m) {
                const int p = tid + m * kProducers, v = (p >> 1) % (kPY * kPX), copy = p / (2 * kPY * kPX);
                const int y = y0 + v / kPX, x = x0 + v % kPX;
                off[m] = ((wrapm(y, a.n2) >> sh) * m3 + (wrapm(x - 1 + copy, a.n3) >> sh)) * cs + (tid & 1) * 8;
                const bool in = y < a.n2 && x < a.n3;
                goff[m] = in ? (wrapm(y + 1 - copy, a.n2) * a.n3 + x) * w.cout + co0 + (tid & 1) * 8 : 0;
                live |= (in ? 1u : 0u) << m;
            }
            const __nv_bfloat16 *src_b = sbase + (long long)b * m1 * pstride;
            const __nv_bfloat16 *g = w.G + ((long long)b * a.n1 + z0) * gstride;
            int zz = wrapm(z0 - 1, a.n1);
            for (int i = 0; i < nz + 2; ++i, ++k) {
                if (k >= kCSlots) ok = warp_agrees(mbar_wait(&empty[q], ph) && !abort_flag);
                if (!ok) break;
                const __nv_bfloat16 *src = src_b + (zz >> sh) * pstride;
                if (++zz == a.n1) zz = 0;
                const uint32_t st = saddr(xs) + q * kCPlane;
#pragma unroll
                for (int m = 0; m < kMine; ++m) cp_async16(st + dst[m], src + off[m], (live >> m) & 1 ? 16 : 0);
                if (i < nz) {   // G plane i (its slot's last reader is no later than the X slot's)
                    const uint32_t gd = saddr(gs) + gq * kCPlane;
#pragma unroll
                    for (int m = 0; m < kMine; ++m) cp_async16(gd + dst[m], g + goff[m], (live >> m) & 1 ? 16 : 0);
                    g += gstride;
                    if (++gq == kCGSlots) gq = 0;
                }
                cp_async_commit();
                if (k - sent >= kCDepth - 1) {
                    cp_async_wait<kCDepth - 1>();
                    arrive();
                }
                if (++q == kCSlots) {
                    q = 0;
                    ph ^= 1;
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (ok)
            while (sent < k) arrive();
        if (!ok) abort_flag = 1;
        ok = warp_agrees(ok && mbar_wait(&done, (uint32_t)(nruns - 1) & 1u) && !abort_flag);
        if (ok) {
            tc_fence_after();
            take(nruns > 1);
        } else if (tid == 0) {
            atomicExch(a.err, 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

}  // namespace

// The word a kernel sets when a bounded wait gives up, one per device: host memory
// that the device maps, so that reading it after a call costs no copy (the copy
// from a device symbol took about 10 us of every call).
int *conv3_tc_error_word_of(int dev) {
    static PerDevice<int *> words;
    int **w = words.get(dev, [](int *&p) {
        void *q = nullptr;
        if (cudaHostAlloc(&q, sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();   // (not for a later call to find)
            return false;
        }
        p = static_cast<int *>(q);
        *p = 0;
        return true;
    });
    return w ? *w : nullptr;
}

int *conv3_tc_error_word() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return conv3_tc_error_word_of(dev);
}

// SMs of the current device, whose kernels' shared-memory limits (and carve-outs: all
// of the unified L1/shared array, so that the CTAs that the budget allows are
// resident together) are raised at the first call on it; 0 where that failed
static int device_sms() {
    static PerDevice<int> sms;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    const int *n = sms.get(dev, [dev](int &count) {
        int lim = 0;
        cudaError_t e = cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        auto raise = [&](const void *k, bool carveout) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lim - 1024);
            if (e == cudaSuccess && carveout) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        };
        raise((const void *)k_conv3_tc, false);
        for (auto k : {k_conv3_tch, k_conv3_tcp}) raise((const void *)k, true);
        raise((const void *)k_conv3_tcd, true);
        for (auto k : {k_conv3_col<16>, k_conv3_col<32>, k_conv3_col<48>, k_conv3_col<64>, k_conv3_col<80>})
            raise((const void *)k, true);
        for (auto k : {k_wgrad3_col<false>, k_wgrad3_col<true>}) raise((const void *)k, true);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess;
    });
    return n ? *n : 0;
}

int conv3_forward_tc(const ConvArgs &in, cudaStream_t st) {
    ConvArgs a = in;
    if ((a.cout & 15) || a.cout > 256 || a.cout < 16 || (a.c0s & 15) || (a.c1s & 15) || a.c0s <= 0) return -1;
    if (a.c1s && (!a.src1 || (a.n1 | a.n2 | a.n3) & 1)) return -1;
    a.err = conv3_tc_error_word();
    if (!a.err) return -2;
    int ncols = 32;
    while (ncols < a.cout) ncols <<= 1;
    const int nsm = device_sms();
    if (!nsm) return -3;
    if (3 * a.cout <= 256) {
        // column march: two CTAs per SM up to 32 output channels, one above;
        // planes of an item by half of a CTA's tensor memory
        const int per_sm = a.cout <= 32 ? 2 : 1, nch = (a.c0s + a.c1s) / 16;
        const int zmax = a.cout <= 32 ? 128 / a.cout : 256 / a.cout, zl = a.n1 < zmax ? a.n1 : zmax;
        int nc = 32;
        while (nc < 2 * zl * a.cout) nc <<= 1;
        const size_t wb = (size_t)27 * 32 * a.cout, room = 233472 / per_sm - 3 * 1024;
        // all chunks' weights if they leave room for eight planes, else two or one
        int wslots = nch;
        while (wslots > 1 && wslots * wb + 8 * (size_t)kPPlane > room) wslots = wslots > 2 ? 2 : 1;
        int nplanes = (int)((room - wslots * wb) / kPPlane);
        nplanes = nplanes < kPSlots ? nplanes : kPSlots;
        size_t smem = wslots * wb + nplanes * (size_t)kPPlane;
        const size_t floor = 233472 / (512 / nc + 1) + 1024;   // TMEM columns per SM stay <= 512
        if (smem < floor) smem = floor;
        const long long items = (long long)((a.n3 + kPX - 1) / kPX) * ((a.n2 + kPY - 1) / kPY) * ((a.n1 + zl - 1) / zl) * a.B;
        const long long grid = items < (long long)per_sm * nsm ? items : (long long)per_sm * nsm;
        const auto k = a.cout == 16 ? k_conv3_col<16> : a.cout == 32 ? k_conv3_col<32> : a.cout == 48 ? k_conv3_col<48>
                     : a.cout == 64 ? k_conv3_col<64> : k_conv3_col<80>;
        k<<<(unsigned)grid, kColThreads, smem, st>>>(a, nc, zl, nplanes, wslots);
        return 0;
    }
    const bool bricks_tile = a.n1 % 4 == 0 && a.n2 % 4 == 0 && a.n3 % 8 == 0;
    const size_t w_bytes = (size_t)(a.c0s + a.c1s) / 16 * 27 * 32 * a.cout;
    if (bricks_tile && a.cout <= 128 && w_bytes <= 96 * 1024) {
        // persistent CTAs with the weights resident; two TMEM accumulators
        int ncols2 = 32;
        while (ncols2 < 2 * a.cout) ncols2 <<= 1;
        size_t smem = w_bytes + 2 * (size_t)kDHalo;
        const size_t floor = 233472 / (512 / ncols2 + 1) + 1024;
        if (smem < floor) smem = floor;
        // CTAs per SM that shared memory, registers and tensor memory allow
        static const int regs = [] {   // the compiler's, the same on every device
            cudaFuncAttributes fa{};
            if (cudaFuncGetAttributes(&fa, k_conv3_tcp) != cudaSuccess) cudaGetLastError();
            return fa.numRegs > 0 ? (fa.numRegs + 7) / 8 * 8 : 255;
        }();
        int per_sm = (int)(233472 / (smem + 2048));
        per_sm = per_sm < 65536 / (regs * kThreads) ? per_sm : 65536 / (regs * kThreads);
        per_sm = per_sm < 512 / ncols2 ? per_sm : 512 / ncols2;
        if (per_sm < 1) per_sm = 1;
        const long long bricks = (long long)(a.n1 / 4) * (a.n2 / 4) * (a.n3 / 8) * a.B;
        const long long grid = bricks < (long long)per_sm * nsm ? bricks : (long long)per_sm * nsm;
        k_conv3_tcp<<<(unsigned)grid, kThreads, smem, st>>>(a, ncols2);
        return 0;
    }
    if (bricks_tile && a.cout <= 128) {
        // halo tiles read in place: two chunk stages where they fit in about
        // half of the shared memory, else one
        const size_t stage = (size_t)kDHalo + 27 * 32 * (size_t)a.cout;
        const int ring = (a.c0s + a.c1s > 16 && 2 * stage <= 116 * 1024) ? 2 : 1;
        size_t smem = ring * stage;
        const size_t floor = 233472 / (512 / ncols + 1) + 1024;
        if (smem < floor) smem = floor;
        const long long bricks = (long long)(a.n1 / 4) * (a.n2 / 4) * (a.n3 / 8) * a.B;
        k_conv3_tcd<<<(unsigned)bricks, kThreads, smem, st>>>(a, ncols, ring);
        return 0;
    }
    if (a.n1 % 4 == 0 && a.n2 % 4 == 0 && a.n3 % 8 == 0) {
        // halo tiles; at least enough shared memory per CTA that the CTAs
        // resident on an SM never ask for more than its 512 TMEM columns
        size_t smem = (size_t)kHalo * 32 + (size_t)kHSt * (kBM / 8 * kHSBO + a.cout / 8 * kHSBO);
        const size_t floor = 233472 / (512 / ncols + 1) + 1024;
        if (smem < floor) smem = floor;
        const long long bricks = (long long)(a.n1 / 4) * (a.n2 / 4) * (a.n3 / 8) * a.B;
        k_conv3_tch<<<(unsigned)bricks, kThreads, smem, st>>>(a, ncols);
        return 0;
    }
    const size_t smem = (size_t)kStages * (kBM / 8 * kSBO + a.cout / 8 * kSBO);
    const long long total = (long long)a.n1 * a.n2 * a.n3 * a.B;
    k_conv3_tc<<<(unsigned)((total + kBM - 1) / kBM), kThreads, smem, st>>>(a, ncols);
    return 0;
}

bool conv3_wgrad_takes(const WgradArgs &w) {
    const ConvArgs &a = w.in;
    if ((w.cout & 15) || w.cout > 64 || w.cout < 16 || a.c0s < 0 || a.c1s < 0 || ((a.c0s | a.c1s) & 15)) return false;
    if (a.c0s + a.c1s <= 0) return false;
    return !(a.c1s && ((a.n1 | a.n2 | a.n3) & 1));
}

int conv3_wgrad(const WgradArgs &in, cudaStream_t st) {
    WgradArgs w = in;
    w.in.err = conv3_tc_error_word();
    const ConvArgs &a = w.in;
    if (w.S <= 0 || !conv3_wgrad_takes(w)) return -1;
    if (!a.err) return -2;
    if (!device_sms()) return -3;
    const int nc = 256;   // 144 columns; two CTAs per SM by tensor and shared memory
    const int zl = a.n1 < 8 ? a.n1 : 8;
    size_t smem = (size_t)(kCSlots + kCGSlots) * kCPlane + kCPad;
    const size_t floor = 233472 / (512 / nc + 1) + 1024;    // TMEM columns per SM stay <= 512
    if (smem < floor) smem = floor;
    // four items of 1024 voxels, or 1/256 of all voxels where that is more
    const long long vox = (long long)a.B * a.n1 * a.n2 * a.n3, per256 = vox / (256 * 1024);
    const int run = (int)(per256 < kCRun ? kCRun : (per256 > 1 << 20 ? 1 << 20 : per256));
    const long long items = (long long)((a.n3 + kPX - 1) / kPX) * ((a.n2 + kPY - 1) / kPY) * ((a.n1 + zl - 1) / zl) * a.B;
    const auto k = (items + w.S - 1) / w.S > run ? k_wgrad3_col<true> : k_wgrad3_col<false>;
    k<<<dim3(w.S, (a.c0s + a.c1s) / 16, w.cout / 16), kThreads, smem, st>>>(w, nc, zl, run);
    return 0;
}

int conv3_tc_error(int clear) {
    int *f = conv3_tc_error_word();
    if (!f) return 0;
    return clear ? __atomic_exchange_n(f, 0, __ATOMIC_ACQ_REL) : __atomic_load_n(f, __ATOMIC_ACQUIRE);
}

}  // namespace hnet
