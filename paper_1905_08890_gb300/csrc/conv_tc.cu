// conv_tc.cu - the U-Net's circular 3^3 convolution on the 5th-generation
// tensor cores (tcgen05.mma, FP32 accumulators in tensor memory), for grids of
// 128^3 voxels (rows of exactly 128 voxels: the network's finest level, where
// two thirds of its arithmetic sits) with 16 or 48 input channels.
//
// Implicit GEMM with M = the 128 voxels of a row.  An input row (d', h') takes
// part in the nine output rows (d' - dd, h' - dh), so one MMA multiplies it
// (shifted by dw, 16 of its channels) with the weights of all nine (dd, dh) at
// once: N = 9 x 16 output channels, accumulated in nine neighbouring blocks of
// 16 tensor-memory columns; 3 cin / 16 MMAs per input row.  With one tap per MMA (N =
// 16, 27 cin / 16 per output row) the tensor core read 4 KB of A for 512 B of B: 178 us for
// 16 -> 16 channels and 701 us for 48 -> 16 at 128^3, now 54 and 110 us (the
// mma.sync kernel: 108 and 437).  The issue of the MMAs bounds it: about 70 clocks
// each, as long as their 8.7 KB of operands take to read, and the mbarrier
// waits of the issuing thread, so rows are handed over in pairs.
//
// A block works on 8 output rows (h0 .. h0 + 7) of a range of planes d.  Row r
// of plane q accumulates in columns 48 r + 16 (q mod 3): while the input rows of
// plane d' arrive, planes d' - 1, d' and d' + 1 are open, and with row h' their
// rows h' - 1 .. h' + 1, which are neighbouring columns.  The slot of a plane
// rotates with d', so the weights sit in shared memory in three rotations.  Per
// output element the products are summed in the order of the taps (dd, dh, dw),
// then of the channels.  Outside the range (two further input planes, two further
// input rows) the blocks of output rows that the range does not have sum up
// values nobody reads.
//
// Input rows are staged in shared memory in the canonical no-swizzle K-major
// layout (core matrices of 8 voxels x 16 bytes; plane p holds channels 8p ..
// 8p + 7 of every voxel), with one wrapped halo voxel on each side, so that tap dw is
// the same row read from a start address 16 (dw + 1) bytes further on.  Roles:
// warps 8..11 copy rows into a ring (cp.async), one thread of warp 12 issues the
// MMAs, warps 0..7 read finished rows back (tcgen05.ld; thread t of four owns
// tensor-memory lane t = voxel w), clear their columns for the plane three further on,
// and write BF16 (bias and ReLU, or the ReLU mask of the data gradient).
// mbarriers between them, per pair of rows: slots full, slots empty (and output
// rows complete), output rows drained.
//
// Every wait is bounded (2 s); a wait that runs out sets g_conv_tc_err, the
// other waits of the block then give up as well, and the block goes on to
// release its tensor memory and return.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "gr_internal.cuh"
#include "unet_internal.cuh"

namespace gr {

__device__ int g_conv_tc_err = 0;

namespace {

constexpr int kRowVox = 128;         // voxels per output row (= MMA M)
constexpr int kRows = 8;             // output rows of a block
constexpr int kInRows = kRows + 2;   // input rows of a plane
constexpr int kN = 9 * 16;           // columns of one MMA
constexpr uint32_t kMatB = kN * 32;  // bytes of one weight matrix (kN x 16 BF16)
constexpr uint32_t kTmemCols = 512;  // 8 x 48 used; a power of two is allocated
constexpr int kThreads = 13 * 32;
constexpr int kUnits = 128 / kRows * 128;  // (row group, plane) pairs of the grid

// per number of 16-channel chunks of the input: ring slots (rows; handed over in pairs), rows a
// copying warp (every fourth row) has in flight before it waits for one, and 16-byte pieces per
// 8-channel plane of a staged row (130 used; the stride spreads one warp's copies over the banks)
template <int NCH>
struct Ring {
    static constexpr int kSlots = NCH == 1 ? 16 : 8, kAhead = kSlots / 4 - 1;
    static constexpr uint32_t kPlaneB = (NCH == 1 ? 132 : 133) * 16, kRowB = 2 * NCH * kPlaneB;
    static constexpr uint32_t kWeights = 512, kStage = kWeights + 9 * NCH * kMatB;
    static constexpr uint32_t kSmem = kStage + kSlots * kRowB;
};

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: no swizzle, K-major; start, leading
// (K-direction core-matrix) and stride (M/N-direction 8-row group) byte offsets
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of the 5th-generation tensor cores
    return d;                // base offset 0, swizzle none
}

// instruction descriptor of kind::f16: D FP32, A and B BF16, both K-major, M = 128
__device__ __forceinline__ constexpr uint32_t idesc_bf16(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRowVox >> 4) << 24);
}

__device__ __forceinline__ void mma_tc(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t id, uint32_t accum)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
        "l"(ad), "l"(bd), "r"(id), "r"(accum));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// bounded wait for the completion of phase `parity` of the mbarrier; quit: the block's give-up flag
__device__ __forceinline__ void mbar_wait(uint32_t mbar, uint32_t parity, volatile int *quit)
{
    long long start = 0;
    for (int it = 0;; it++) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return;
        if (it == 0) start = clock64();
        else if ((it & 63) == 0 && (*quit || clock64() - start > 4000000000ll)) {
            *quit = 1;
            atomicExch(&g_conv_tc_err, 1);
            return;
        }
    }
}

__device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// zeros into 16 columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_zero16(uint32_t taddr)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(
                     taddr),
                 "r"(0)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16(lo)) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16(hi)) << 16);
}

__device__ __forceinline__ void cp16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory");
}

// x: [128^3][16 NCH] BF16, w: [27][cout][16 NCH] BF16, bias [cout] (CONV_RELU), mask
// [128^3][cout] (CONV_MASK), y: [128^3][cout] BF16; blockIdx.y: group of 16 output channels.
template <int NCH>
__global__ void __launch_bounds__(kThreads, 1)
    k_conv3d_tc(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ w, const float *__restrict__ bias,
                int cout, int mode, const __nv_bfloat16 *__restrict__ mask, __nv_bfloat16 *__restrict__ y)
{
    pdl_begin();
    extern __shared__ __align__(128) uint8_t sm[];
    using R = Ring<NCH>;
    constexpr int cin = 16 * NCH, planes = 2 * NCH;
    const int tid = threadIdx.x, warp = tid >> 5, co0 = 16 * blockIdx.y;
    const uint32_t base = smem_u32(sm), slot = base, bs = base + R::kWeights, as = base + R::kStage;
    volatile int *quit = reinterpret_cast<volatile int *>(sm + 4);
    constexpr int kPairs = R::kSlots / 2;  // pairs of rows: one wait and one commit for 6 NCH MMAs
    const uint32_t full = base + 16, empty = full + 8 * kPairs, drained = empty + 8 * kPairs,
                   fin = drained + 8 * (kRows / 2);  // 16 + 8 (2 x 8 + 5) bytes at most
    if (tid == 0) {
        quit[0] = quit[1] = 0;
        for (int k = 0; k < kPairs; k++) {
            mbar_init(full + 8 * k, 64);
            mbar_init(empty + 8 * k, 1);
        }
        for (int k = 0; k < kRows / 2; k++) mbar_init(drained + 8 * k, 256);
        mbar_init(fin, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // weights: matrix (v 3 + dw) NCH + c for planes d' = v mod 3; its row n = 48 k + 16 s + co is
    // output row h' - 1 + k (dh = 1 - k) of the plane in slot s (d' + j with (v + j) mod 3 = s, dd = -j)
    for (int e = tid; e < 9 * NCH * kN * 2; e += kThreads) {
        const int p = e & 1, n = (e >> 1) % kN, m = (e >> 1) / kN;
        const int c = m % NCH, dw = m / NCH % 3, v = m / NCH / 3;
        const int k = n / 48, sl = n / 16 % 3, co = n & 15;
        const int j = (sl - v + 4) % 3 - 1, tap = (1 - j) * 9 + (2 - k) * 3 + dw;
        cp16(bs + m * kMatB + p * kN * 16 + n * 16, w + ((size_t)tap * cout + co0 + co) * cin + 16 * c + 8 * p);
    }
    cp_commit();
    cp_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    fence_before();
    __syncthreads();  // weights, mbarriers and the tensor-memory address are visible
    fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(sm);
    if (warp < 4) {
        for (int k = 0; k < 3 * kRows; k++) tmem_zero16(tmem + ((uint32_t)(warp * 32) << 16) + 16 * k);
        tmem_wait_st();
    }
    fence_before();
    __syncthreads();  // the accumulators are zero
    fence_after();
    const int u0 = (int)((int64_t)blockIdx.x * kUnits / gridDim.x), u1 = (int)((int64_t)(blockIdx.x + 1) * kUnits / gridDim.x);
    // every role walks the same input planes: f(first row of the group, input plane, first and one past
    // the last output plane); planes d0 - 1 .. d1 of each run d0 .. d1 - 1 within one row group
    auto walk = [&](auto &&f) {
        for (int u = u0; u < u1;) {
            const int d0 = u & 127, run = min(u1 - u, 128 - d0), h0 = (u >> 7) * kRows;
            for (int d = d0 - 1; d <= d0 + run; d++) f(h0, d, d0, d0 + run);
            u += run;
        }
    };
    if (warp >= 8 && warp < 12) {  // each copies every fourth row
        const int lane = tid & 31, mine = warp - 8;
        int k = 0, i = 0, done = 0;  // rows passed, copied here, handed over
        walk([&](int h0, int d, int, int) {
            for (int h = h0 - 1; h <= h0 + kRows; h++, k++) {
                if ((k & 3) != mine) continue;
                const int sl = k % R::kSlots, pair = sl >> 1;
                if (k >= R::kSlots) {
                    const uint32_t parity = (k / R::kSlots - 1) & 1;
                    // no free slot: hand over what is in flight before waiting for one
                    if (done < i && !mbar_test(empty + 8 * pair, parity)) {
                        cp_wait<0>();
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        for (; done < i; done++) mbar_arrive(full + 8 * ((4 * done + mine) / 2 % kPairs));
                    }
                    mbar_wait(empty + 8 * pair, parity, quit);
                }
                const __nv_bfloat16 *row = x + ((size_t)((d & 127) << 7 | (h & 127)) << 7) * cin;
                const uint32_t dst = as + sl * R::kRowB;
#pragma unroll
                for (int j = 0; j < 4 * planes; j++) {
                    const int e = j * 32 + lane, p = e % planes, v = e / planes;
                    cp16(dst + p * R::kPlaneB + 16 * (v + 1), row + 8 * e);
                }
                if (lane < 2 * planes) {  // the wrapped halo voxels
                    const int p = lane >> 1, hi = lane & 1;
                    cp16(dst + p * R::kPlaneB + (hi ? 16 * 129 : 0), row + (hi ? 0 : 127 * cin) + 8 * p);
                }
                cp_commit();
                if (++i - done > R::kAhead) {
                    cp_wait<R::kAhead>();  // this lane's part of all but the kAhead latest rows has landed
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    for (; done < i - R::kAhead; done++) mbar_arrive(full + 8 * ((4 * done + mine) / 2 % kPairs));
                }
            }
        });
        cp_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (; done < i; done++) mbar_arrive(full + 8 * ((4 * done + mine) / 2 % kPairs));
    } else if (warp == 12) {
        if (tid == 384) {
            int k = 0;  // pairs consumed
            const uint64_t a0 = sdesc(as, R::kPlaneB, 128), b0 = sdesc(bs, kN * 16, 128);
            walk([&](int, int d, int, int) {
                const uint64_t bv = b0 + (uint64_t)(((d + 3) % 3) * 3 * NCH * (kMatB >> 4));
#pragma unroll
                for (int g = 0; g < kInRows / 2; g++, k++) {
                    const int sl = k % kPairs;
                    mbar_wait(full + 8 * sl, (k / kPairs) & 1, quit);
                    // output rows 2 g and 2 g + 1 of plane d + 1 begin: their columns have been read and cleared
                    if (k >= kInRows / 2 && g < kRows / 2) mbar_wait(drained + 8 * g, (k / (kInRows / 2) - 1) & 1, quit);
                    fence_after();
                    const uint64_t ap = a0 + (uint64_t)(2 * sl * (R::kRowB >> 4));
#pragma unroll
                    for (int hp = 0; hp < 2; hp++) {
                        // input row h of the group's; output rows h - 1 .. h + 1 within the group: MMA columns
                        // from 48 first, weight rows from 48 skip
                        const int h = 2 * g - 1 + hp, first = h > 0 ? h - 1 : 0, last = h < kRows - 1 ? h + 1 : kRows - 1;
                        const int skip = first - (h - 1);
#pragma unroll
                        for (int dw = 0; dw < 3; dw++)
#pragma unroll
                            for (int c = 0; c < NCH; c++)
                                mma_tc(tmem + 48 * first, ap + (uint64_t)((hp * R::kRowB + 16 * dw + c * 2 * R::kPlaneB) >> 4),
                                       bv + (uint64_t)(((dw * NCH + c) * kMatB + skip * 48 * 16) >> 4),
                                       idesc_bf16(48 * (last - first + 1)), 1u);
                    }
                    mma_commit(empty + 8 * sl);  // the slots are free; rows 2 g - 2, 2 g - 1 of plane d - 1 are complete
                }
            });
            mma_commit(fin);
            mbar_wait(fin, 0, quit + 1);  // its own flag: waits for the MMAs in flight also after a give-up
        }
        __syncwarp();
    } else {
        const uint32_t lane0 = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const int vox = tid & 127;
        float bv[16];
#pragma unroll
        for (int k = 0; k < 16; k++) bv[k] = mode == CONV_RELU ? bias[co0 + k] : 0.0f;
        int seq = 0;
        walk([&](int h0, int d, int d0, int d1) {
            const int q = d - 1, sl = (q + 3) % 3;
            for (int r = warp >> 2; r < kRows; r += 2) {  // warps 0..3 the even rows, 4..7 the odd
                // complete with the pair after its own; the pair four later waits for this read
                const int k = seq * (kInRows / 2) + r / 2 + 1;
                mbar_wait(empty + 8 * (k % kPairs), (k / kPairs) & 1, quit);
                fence_after();
                uint32_t a[16];
                tmem_ld16(lane0 + 48 * r + 16 * sl, a);
                tmem_zero16(lane0 + 48 * r + 16 * sl);
                if (d == d1) {  // the run ends: nothing of it stays in the other two slots
                    tmem_zero16(lane0 + 48 * r + 16 * ((sl + 1) % 3));
                    tmem_zero16(lane0 + 48 * r + 16 * ((sl + 2) % 3));
                }
                tmem_wait_st();
                fence_before();
                mbar_arrive(drained + 8 * (r / 2));
                if (q < d0) continue;
                const size_t o0 = (((size_t)(q << 7 | (h0 + r)) << 7) + vox) * cout + co0;
                float o[16];
#pragma unroll
                for (int k = 0; k < 16; k++) o[k] = __uint_as_float(a[k]);
                if (mode == CONV_RELU) {
#pragma unroll
                    for (int k = 0; k < 16; k++) o[k] = fmaxf(o[k] + bv[k], 0.0f);
                } else if (mode == CONV_MASK) {
                    const uint4 m0 = *reinterpret_cast<const uint4 *>(mask + o0);
                    const uint4 m1 = *reinterpret_cast<const uint4 *>(mask + o0 + 8);
                    const __nv_bfloat16 *mb0 = reinterpret_cast<const __nv_bfloat16 *>(&m0);
                    const __nv_bfloat16 *mb1 = reinterpret_cast<const __nv_bfloat16 *>(&m1);
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        o[k] = __bfloat162float(mb0[k]) > 0.0f ? o[k] : 0.0f;
                        o[8 + k] = __bfloat162float(mb1[k]) > 0.0f ? o[8 + k] : 0.0f;
                    }
                }
                uint4 s0, s1;
                s0.x = pack_bf16(o[0], o[1]);
                s0.y = pack_bf16(o[2], o[3]);
                s0.z = pack_bf16(o[4], o[5]);
                s0.w = pack_bf16(o[6], o[7]);
                s1.x = pack_bf16(o[8], o[9]);
                s1.y = pack_bf16(o[10], o[11]);
                s1.z = pack_bf16(o[12], o[13]);
                s1.w = pack_bf16(o[14], o[15]);
                *reinterpret_cast<uint4 *>(y + o0) = s0;
                *reinterpret_cast<uint4 *>(y + o0 + 8) = s1;
            }
            seq++;
        });
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

template <int NCH>
void launch_tc(const __nv_bfloat16 *x, const __nv_bfloat16 *w, const float *bias, int cout, int mode,
               const __nv_bfloat16 *mask, __nv_bfloat16 *y, cudaStream_t st)
{
    static const int sms = [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? n : 1;
    }();
    per_device([] {
        return cudaFuncSetAttribute(k_conv3d_tc<NCH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)Ring<NCH>::kSmem) == cudaSuccess;
    });
    // one block per SM (its tensor memory) and group of 16 output channels
    const dim3 grid(sms < kUnits ? sms : kUnits, cout / 16);
    GR_LAUNCH_SMEM((k_conv3d_tc<NCH>), grid, kThreads, (int)Ring<NCH>::kSmem, st, x, w, bias, cout, mode, mask, y);
}

}  // namespace

bool conv3d_tc_fits(int cin, int cout, int lg)
{
    // 48 input channels fill shared memory (221 KB of weights and ring), and only 48 -> 16 occurs
    if (lg != 7) return false;
    if (cin == 16) return cout == 16 || cout == 32 || cout == 48 || cout == 64;
    return cin == 48 && cout == 16;
}

void conv3d_tc(const __nv_bfloat16 *x, int cin, const __nv_bfloat16 *w, const float *bias, int cout, int mode,
               const __nv_bfloat16 *mask, __nv_bfloat16 *y, cudaStream_t st)
{
    if (cin == 16) launch_tc<1>(x, w, bias, cout, mode, mask, y, st);
    else launch_tc<3>(x, w, bias, cout, mode, mask, y, st);
}

int conv3d_tc_error(cudaStream_t st)
{
    int e = 0;
    if (cudaMemcpyFromSymbolAsync(&e, g_conv_tc_err, sizeof(int), 0, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return -1;
    return e;
}

}  // namespace gr
