// unet_kernels.cu - kernels of the learned initial guess: a 3D U-Net with
// circular 3^3 convolutions on channels-last BF16 activations [v][c],
// v = (d n + h) n + w, FP32 accumulation on the tensor cores (mma.sync
// m16n8k16 BF16; 128^3 grids on tcgen05, conv_tc.cu).  Convolutions are
// implicit GEMMs: output voxels x output channels, reduced over input channels x
// 27 taps, from boxes of voxels staged with their halo in shared memory.
//
// Weights: FP32 master and BF16 copies [27][cout][cin] (tap = (dd+1)*9 +
// (dh+1)*3 + (dw+1)); the data gradient is the same convolution with the
// flipped, transposed copy [27][cin][cout] (tap' = 26 - tap).
#include <cuda_bf16.h>

#include <cstdlib>

#include "gr_internal.cuh"
#include "unet_internal.cuh"

namespace gr {
namespace {

inline int cdiv(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 lo, __nv_bfloat16 hi)
{
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// ---------------------------------------------------------------- convolution
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// A box of 2^lw x 2^lh x 2^ld voxels (w fastest) of a 2^lg grid and its halo of
// one voxel per side: the unit of work of the convolution and its weight gradient.
struct Box {
    int lg, lw, lh, ld;
    __host__ __device__ int hw() const { return (1 << lw) + 2; }
    __host__ __device__ int hh() const { return (1 << lh) + 2; }
    __host__ __device__ int hd() const { return (1 << ld) + 2; }
    __host__ __device__ int halo() const { return hw() * hh() * hd(); }
    // origin of box b (boxes in w, h, d order)
    __device__ void origin(int b, int &d0, int &h0, int &w0) const
    {
        const int nw = lg - lw, nh = lg - lh;
        w0 = (b & ((1 << nw) - 1)) << lw;
        h0 = ((b >> nw) & ((1 << nh) - 1)) << lh;
        d0 = (b >> (nw + nh)) << ld;
    }
    // voxel q of the box: its halo index at tap (0, 0, 0) (the corner of its 3^3 neighbourhood)
    __device__ int corner(int q) const
    {
        const int w = q & ((1 << lw) - 1), h = (q >> lw) & ((1 << lh) - 1), dd = q >> (lw + lh);
        return (dd * hh() + h) * hw() + w;
    }
    __device__ int voxel(int q, int d0, int h0, int w0) const
    {
        const int w = q & ((1 << lw) - 1), h = (q >> lw) & ((1 << lh) - 1), dd = q >> (lw + lh);
        return ((((d0 + dd) << lg) + h0 + h) << lg) + w0 + w;
    }
};

// 2^lb voxels per box: rows along w of up to 16, then h and d in turn
Box make_box(int lg, int lb)
{
    Box x;
    x.lg = lg;
    x.lw = lg < 4 ? lg : 4;
    const int rest = lb - x.lw;
    x.lh = (rest + 1) / 2 < lg ? (rest + 1) / 2 : lg;
    x.ld = rest - x.lh;
    return x;
}

// a 32-byte row (16 channels) holds its two 16-byte halves swapped on every
// second group of four rows, so that eight consecutive rows' halves fall on all 32 banks
__device__ __forceinline__ uint32_t row_half(int row, int half) { return (uint32_t)(32 * row + ((half ^ (row >> 2 & 1)) << 4)); }

// the halo's 16 channels from c0 into shared memory (asynchronous copies)
__device__ __forceinline__ void load_halo(uint32_t dst, const __nv_bfloat16 *x, int cin, int c0, const Box &bx, int d0, int h0,
                                          int w0)
{
    const int m = (1 << bx.lg) - 1, hw = bx.hw(), hh = bx.hh(), n = 2 * bx.halo();
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int r = e >> 1, half = e & 1;
        const int w = r % hw, t = r / hw, h = t % hh, dd = t / hh;
        const int v = ((((d0 + dd - 1) & m) << bx.lg) + ((h0 + h - 1) & m)) * (1 << bx.lg) + ((w0 + w - 1) & m);
        cp16(dst + row_half(r, half), x + (size_t)v * cin + c0 + 8 * half);
    }
}

// Block: WARPS warps along the voxels of one box; warp tile MT*16 voxels x NT*8
// channels; grid.y walks the output channels in steps of NT*8.  Per 16 input
// channels the box with its halo and the 27 taps' weights are staged in shared
// memory, one chunk ahead, and the fragments come from there (ldmatrix):
// gathered straight from global memory in 4-byte loads they cost 16 loads and 40 index
// instructions per eight MMAs.  The ten layers of a 128^3 pass took 1467 us that way and
// take 437 us.  The products are summed in the order input channels, taps, as
// the order of a layer's arithmetic is part of its result.  Epilogue modes:
//   CONV_RELU  y = relu(acc + bias) (BF16)
//   CONV_MASK  y = acc * (mask > 0) (BF16; data gradient through a ReLU)
//   CONV_PLAIN y = acc (BF16)
template <int WARPS, int MT, int NT>
__global__ void __launch_bounds__(32 * WARPS)
    k_conv3d(const __nv_bfloat16 *__restrict__ x, int cin, const __nv_bfloat16 *__restrict__ w,
             const float *__restrict__ bias, int cout, Box bx, int mode, const __nv_bfloat16 *__restrict__ mask,
             __nv_bfloat16 *__restrict__ y)
{
    pdl_begin();
    static_assert(NT % 2 == 0, "two 8-channel tiles per ldmatrix");
    extern __shared__ __align__(128) unsigned char csm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int cb = blockIdx.y * (NT * 8);
    int d0, h0, w0;
    bx.origin(blockIdx.x, d0, h0, w0);
    const int halo = bx.halo(), hw = bx.hw(), hh = bx.hh();
    const uint32_t base = smem_addr(csm), stage = 32u * (uint32_t)(halo + 27 * NT * 8);
    auto load = [&](int c0, uint32_t buf) {
        load_halo(buf, x, cin, c0, bx, d0, h0, w0);
        const uint32_t wb = buf + 32u * (uint32_t)halo;
        for (int e = threadIdx.x; e < 2 * 27 * NT * 8; e += 32 * WARPS) {
            const int half = e & 1, r = e >> 1, co = r % (NT * 8), tap = r / (NT * 8);
            cp16(wb + row_half(r, half), w + ((size_t)tap * cout + cb + co) * cin + c0 + 8 * half);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[MT][NT][4];
#pragma unroll
    for (int a = 0; a < MT; a++)
#pragma unroll
        for (int b = 0; b < NT; b++)
#pragma unroll
            for (int r = 0; r < 4; r++) acc[a][b][r] = 0.0f;
    // this lane's row of each A tile (lanes 0..15: channels 0..7, 16..31: 8..15) and of each B pair
    int arow[MT];
#pragma unroll
    for (int a = 0; a < MT; a++) arow[a] = bx.corner((warp * MT + a) * 16 + (lane & 15));
    const int ahalf = lane >> 4, brow = (lane & 7) + ((lane >> 4) << 3), bhalf = (lane >> 3) & 1;
    load(0, base);
    for (int c0 = 0, k = 0; c0 < cin; c0 += 16, k ^= 1) {
        const uint32_t buf = base + (k ? stage : 0u);
        if (c0 + 16 < cin) {
            load(c0 + 16, base + (k ? 0u : stage));
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const uint32_t wb = buf + 32u * (uint32_t)halo;
        int tap = 0;
        for (int dd = 0; dd < 3; dd++)
            for (int dh = 0; dh < 3; dh++) {
                const int off = (dd * hh + dh) * hw;
#pragma unroll
                for (int dw = 0; dw < 3; dw++, tap++) {
                    uint32_t bf[NT / 2][4];
#pragma unroll
                    for (int b = 0; b < NT / 2; b++) ldsm4(bf[b], wb + row_half(tap * NT * 8 + 16 * b + brow, bhalf));
#pragma unroll
                    for (int a = 0; a < MT; a++) {
                        uint32_t af[4];
                        ldsm4(af, buf + row_half(arow[a] + off + dw, ahalf));
#pragma unroll
                        for (int b = 0; b < NT; b++) {
                            const uint32_t bb[2] = {bf[b >> 1][2 * (b & 1)], bf[b >> 1][2 * (b & 1) + 1]};
                            mma_bf16(acc[a][b], af, bb);
                        }
                    }
                }
            }
        __syncthreads();  // before the next chunk's copies overwrite this buffer
    }
#pragma unroll
    for (int a = 0; a < MT; a++)
#pragma unroll
        for (int hrow = 0; hrow < 2; hrow++) {
            const int v = bx.voxel((warp * MT + a) * 16 + g + 8 * hrow, d0, h0, w0);
#pragma unroll
            for (int b = 0; b < NT; b++) {
                const int co = cb + b * 8 + 2 * t;
                float r0 = acc[a][b][2 * hrow], r1 = acc[a][b][2 * hrow + 1];
                const size_t o = (size_t)v * cout + co;
                if (mode == CONV_RELU) {
                    r0 = fmaxf(r0 + bias[co], 0.0f);
                    r1 = fmaxf(r1 + bias[co + 1], 0.0f);
                } else if (mode == CONV_MASK) {
                    r0 = __bfloat162float(mask[o]) > 0.0f ? r0 : 0.0f;
                    r1 = __bfloat162float(mask[o + 1]) > 0.0f ? r1 : 0.0f;
                }
                *reinterpret_cast<uint32_t *>(y + o) = pack2(__float2bfloat16(r0), __float2bfloat16(r1));
            }
        }
}

template <int WARPS, int MT, int NT>
void launch_conv3d(const __nv_bfloat16 *x, int cin, const __nv_bfloat16 *w, const float *bias, int cout, int lg, int lb,
                   int mode, const __nv_bfloat16 *mask, __nv_bfloat16 *y, cudaStream_t st)
{
    // the largest halo of these boxes: 2^8 voxels as 4 x 4 x 16 or 4 x 8 x 8
    constexpr int kMost = 2 * 32 * (720 + 27 * NT * 8);
    per_device([] {
        return cudaFuncSetAttribute(k_conv3d<WARPS, MT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost) ==
               cudaSuccess;
    });
    const Box bx = make_box(lg, lb);
    const int smem = (cin > 16 ? 2 : 1) * 32 * (bx.halo() + 27 * NT * 8);
    const dim3 grid(1u << (3 * lg - lb), cout / (NT * 8));
    GR_LAUNCH_SMEM((k_conv3d<WARPS, MT, NT>), grid, 32 * WARPS, smem, st, x, cin, w, bias, cout, bx, mode, mask, y);
}

// ---------------------------------------------------------------- weight gradient
// dw[tap][co][ci] += sum_v dy[v][co] x[v's neighbour at tap][ci]: GEMM with M = co,
// N = ci, K = voxels.  Block: 16 output x 16 input channels (grid.y), a range of
// voxel boxes (grid.x), all 27 taps, three per warp.  Per box the 16 channels of
// dy and of x with its halo are staged in shared memory, one box ahead; both
// operands are read transposed (ldmatrix .trans) from the voxel rows, A once
// for a warp's three taps.  The taps' sums stay in registers over the block's
// boxes and end in one FP32 atomic per weight.  The blocks of the first 16 input
// channels also sum dy itself, the bias's gradient (4.4 us a layer as a launch of its own).  (One tap per block with
// two-byte gathers took 957 us over the layers at 64^3; these take 304.)
constexpr int kWgWarps = 9, kWgBox = 8;  // boxes of 2^8 voxels (or the grid)
__global__ void __launch_bounds__(32 * kWgWarps)
    k_conv3d_wgrad(const __nv_bfloat16 *__restrict__ x, int cin, const __nv_bfloat16 *__restrict__ dy, int cout, Box bx,
                   int nbox, float *__restrict__ dw, float *__restrict__ db)
{
    pdl_begin();
    extern __shared__ __align__(128) unsigned char csm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int nci = cin >> 4, co0 = ((int)blockIdx.y / nci) << 4, ci0 = ((int)blockIdx.y % nci) << 4;
    const int halo = bx.halo(), hw = bx.hw(), hh = bx.hh(), nv = 1 << (bx.lw + bx.lh + bx.ld);
    const uint32_t base = smem_addr(csm), stage = 32u * (uint32_t)(halo + nv);
    const int first = (int)((int64_t)blockIdx.x * nbox / gridDim.x), last = (int)((int64_t)(blockIdx.x + 1) * nbox / gridDim.x);
    auto load = [&](int b, uint32_t buf) {
        int d0, h0, w0;
        bx.origin(b, d0, h0, w0);
        load_halo(buf, x, cin, ci0, bx, d0, h0, w0);
        for (int e = threadIdx.x; e < 2 * nv; e += 32 * kWgWarps) {
            const int q = e >> 1, half = e & 1;
            cp16(buf + 32u * (uint32_t)halo + row_half(q, half), dy + (size_t)bx.voxel(q, d0, h0, w0) * cout + co0 + 8 * half);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[3][2][4] = {};
    int toff[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const int tap = 3 * warp + j;
        toff[j] = ((tap / 9) * hh + (tap / 3) % 3) * hw + tap % 3;
    }
    // this lane's row and half of the four 8 x 8 matrices.  A (co x voxels, from
    // dy's voxel rows): voxels 0..7 co 0..7, voxels 0..7 co 8..15, then voxels
    // 8..15; B (voxels x ci): voxels 0..7 and 8..15 of ci 0..7, then of ci 8..15
    const int arow = (lane & 7) + ((lane >> 4) << 3), ahalf = (lane >> 3) & 1;
    const int brow = (lane & 7) + (((lane >> 3) & 1) << 3), bhalf = lane >> 4;
    // bias: thread t < 256 sums channel t mod 16 over every 16th voxel
    const bool bias = ci0 == 0 && threadIdx.x < 256;
    const int bc = threadIdx.x & 15;
    float bsum = 0.0f;
    if (first < last) load(first, base);
    for (int b = first, k = 0; b < last; b++, k ^= 1) {
        const uint32_t buf = base + (k ? stage : 0u);
        if (b + 1 < last) {
            load(b + 1, base + (k ? 0u : stage));
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        for (int q = 0; q < nv; q += 16) {
            uint32_t af[4];
            ldsm4t(af, buf + 32u * (uint32_t)halo + row_half(q + arow, ahalf));
            const int c = bx.corner(q + brow);
#pragma unroll
            for (int j = 0; j < 3; j++) {
                uint32_t bf[4];
                ldsm4t(bf, buf + row_half(c + toff[j], bhalf));
                const uint32_t b0[2] = {bf[0], bf[1]}, b1[2] = {bf[2], bf[3]};
                mma_bf16(acc[j][0], af, b0);
                mma_bf16(acc[j][1], af, b1);
            }
        }
        if (bias) {
            const unsigned char *dyb = csm + (buf - base) + 32 * halo + 2 * (bc & 7);
            for (int q = threadIdx.x >> 4; q < nv; q += 16)
                bsum += __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(dyb + row_half(q, bc >> 3)));
        }
        __syncthreads();  // before the next box's copies overwrite this buffer
    }
    if (first >= last) return;
    if (ci0 == 0) {
        float *sb = reinterpret_cast<float *>(csm);
        bsum += __shfl_xor_sync(0xffffffffu, bsum, 16);
        if (threadIdx.x < 256 && lane < 16) sb[16 * warp + lane] = bsum;
        __syncthreads();
        if (threadIdx.x < 16) {
            float v = 0.0f;
            for (int k = 0; k < 8; k++) v += sb[16 * k + threadIdx.x];
            atomicAdd(db + co0 + threadIdx.x, v);
        }
    }
    // acc[j][n][0..1]: co g, ci 8 n + 2 t (+ 1); [2..3]: co g + 8
#pragma unroll
    for (int j = 0; j < 3; j++)
#pragma unroll
        for (int n = 0; n < 2; n++)
#pragma unroll
            for (int r = 0; r < 4; r++)
                atomicAdd(dw + ((size_t)(3 * warp + j) * cout + co0 + g + 8 * (r >> 1)) * cin + ci0 + 8 * n + 2 * t + (r & 1),
                          acc[j][n][r]);
}

// cell-centred trilinear x2 upsampling (weights 3/4, 1/4 per axis) into
// channels [0, c) of a buffer with channel stride cstride
__global__ void k_upsample(const __nv_bfloat16 *__restrict__ x, int c, int lgc, __nv_bfloat16 *__restrict__ y,
                           int cstride)
{
    pdl_begin();
    const int lgf = lgc + 1, mf = (1 << lgf) - 1, mc = (1 << lgc) - 1;
    const int64_t total = ((int64_t)1 << (3 * lgf)) * c;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(e % c);
        const int v = (int)(e / c);
        const int k = v & mf, j = (v >> lgf) & mf, i = v >> (2 * lgf);
        int I[2], J[2], K[2];
        I[0] = i >> 1;
        I[1] = (i & 1) ? ((I[0] + 1) & mc) : ((I[0] - 1) & mc);
        J[0] = j >> 1;
        J[1] = (j & 1) ? ((J[0] + 1) & mc) : ((J[0] - 1) & mc);
        K[0] = k >> 1;
        K[1] = (k & 1) ? ((K[0] + 1) & mc) : ((K[0] - 1) & mc);
        const float wt[2] = {0.75f, 0.25f};
        float s = 0.0f;
        for (int a = 0; a < 2; a++)
            for (int b = 0; b < 2; b++)
                for (int q = 0; q < 2; q++)
                    s += wt[a] * wt[b] * wt[q] *
                         __bfloat162float(x[(size_t)((((I[a] << lgc) + J[b]) << lgc) + K[q]) * c + ch]);
        y[(size_t)v * cstride + ch] = __float2bfloat16(s);
    }
}

// y[v][yoff + ch] = x[v][xoff + ch] (copy into a channel slice)
__global__ void k_copy_slice(const __nv_bfloat16 *__restrict__ x, int c, int xs, int xoff, __nv_bfloat16 *__restrict__ y,
                             int ys, int yoff, int64_t nv)
{
    pdl_begin();
    const int64_t total = nv * c;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(e % c);
        const int64_t v = e / c;
        y[v * ys + yoff + ch] = x[v * xs + xoff + ch];
    }
}

// Eight channels per thread (c and the channel strides and offsets multiples
// of 8, 16-byte aligned rows): the same per-channel arithmetic as k_upsample
// and k_copy_slice with 16-byte loads and stores and the weights and indices
// formed once per eight channels.
__device__ __forceinline__ void bf8_unpack(uint4 r, float f[8])
{
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&r);
#pragma unroll
    for (int m = 0; m < 4; m++) {
        const float2 t = __bfloat1622float2(h[m]);
        f[2 * m] = t.x, f[2 * m + 1] = t.y;
    }
}

__device__ __forceinline__ uint4 bf8_pack(const float f[8])
{
    uint4 r;
    __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&r);
#pragma unroll
    for (int m = 0; m < 4; m++) h[m] = __floats2bfloat162_rn(f[2 * m], f[2 * m + 1]);
    return r;
}

// Eight channels of the four fine voxels (j, k) = (2 J + 0..1, 2 K + 0..1) of a fine plane i per
// thread: 18 coarse voxels are read and unpacked for them (8 per fine voxel on its own:
// 74 us for 32 channels to 128^3, so 55).  Per voxel the eight products are added in the
// order own cell first, then neighbour, along i, j, k.
__global__ void __launch_bounds__(256)
    k_upsample8(const __nv_bfloat16 *__restrict__ x, int lgc8, int lgc, __nv_bfloat16 *__restrict__ y, int cstride)
{
    pdl_begin();
    const int lgf = lgc + 1, mc = (1 << lgc) - 1, c = 8 << lgc8;
    const int total = 1 << (3 * lgc + 1 + lgc8);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int ch = (e & ((1 << lgc8) - 1)) << 3;
        const int v = e >> lgc8;
        const int K = v & mc, J = (v >> lgc) & mc, i = v >> (2 * lgc);
        const int I[2] = {i >> 1, ((i >> 1) + ((i & 1) ? 1 : -1)) & mc};
        const int js[3] = {J, (J - 1) & mc, (J + 1) & mc}, ks[3] = {K, (K - 1) & mc, (K + 1) & mc};
        const float wt[2] = {0.75f, 0.25f};
        float s[2][2][8] = {};
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int b = 0; b < 3; b++)
#pragma unroll
                for (int q = 0; q < 3; q++) {
                    float xv[8];
                    bf8_unpack(*reinterpret_cast<const uint4 *>(x + (size_t)((((I[a] << lgc) + js[b]) << lgc) + ks[q]) * c + ch), xv);
                    // the own cell serves both fine voxels of its axis, J - 1 the lower and J + 1 the upper one
#pragma unroll
                    for (int fj = 0; fj < 2; fj++)
#pragma unroll
                        for (int fk = 0; fk < 2; fk++) {
                            if ((b != 0 && b != fj + 1) || (q != 0 && q != fk + 1)) continue;
                            const float w = wt[a] * wt[b != 0] * wt[q != 0];
#pragma unroll
                            for (int m = 0; m < 8; m++) s[fj][fk][m] += w * xv[m];
                        }
                }
#pragma unroll
        for (int fj = 0; fj < 2; fj++)
#pragma unroll
            for (int fk = 0; fk < 2; fk++)
                *reinterpret_cast<uint4 *>(y + (size_t)((((i << lgf) + 2 * J + fj) << lgf) + 2 * K + fk) * cstride + ch) =
                    bf8_pack(s[fj][fk]);
    }
}

// 2^3 average pooling, channels-last, channel stride c = 8 2^lgc8; fine extent 2^lgf (16 channels at
// 128^3: 11 us, 23 with one channel per thread)
__global__ void k_pool8(const __nv_bfloat16 *__restrict__ x, int lgc8, int lgf, __nv_bfloat16 *__restrict__ y)
{
    pdl_begin();
    const int lgc = lgf - 1, mc = (1 << lgc) - 1, c = 8 << lgc8;
    const int64_t total = (int64_t)1 << (3 * lgc + lgc8);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(e & ((1 << lgc8) - 1)) << 3;
        const int V = (int)(e >> lgc8);
        const int K = V & mc, J = (V >> lgc) & mc, I = V >> (2 * lgc);
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int b = 0; b < 2; b++)
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const int v = ((((2 * I + a) << lgf) + 2 * J + b) << lgf) + 2 * K + k;
                    float xv[8];
                    bf8_unpack(*reinterpret_cast<const uint4 *>(x + (size_t)v * c + ch), xv);
#pragma unroll
                    for (int m = 0; m < 8; m++) s[m] += xv[m];
                }
#pragma unroll
        for (int m = 0; m < 8; m++) s[m] *= 0.125f;
        *reinterpret_cast<uint4 *>(y + (size_t)V * c + ch) = bf8_pack(s);
    }
}

// Gradient of a level's last encoder activation act: through the skip connection
// (channels [soff, soff + c) of the concatenation's gradient, stride ss) plus the
// pooling's, dy / 8 of the parent, through act's ReLU
__global__ void k_skip_back8(const __nv_bfloat16 *__restrict__ dy, int lgc8, int lgf, const __nv_bfloat16 *__restrict__ skip,
                             int ss, int soff, const __nv_bfloat16 *__restrict__ act, __nv_bfloat16 *__restrict__ dx)
{
    pdl_begin();
    const int mf = (1 << lgf) - 1, lgc = lgf - 1, c = 8 << lgc8;
    const int64_t total = (int64_t)1 << (3 * lgf + lgc8);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(e & ((1 << lgc8) - 1)) << 3;
        const int v = (int)(e >> lgc8);
        const int k = v & mf, j = (v >> lgf) & mf, i = v >> (2 * lgf);
        const int V = ((((i >> 1) << lgc) + (j >> 1)) << lgc) + (k >> 1);
        float g[8], s[8], a[8];
        bf8_unpack(*reinterpret_cast<const uint4 *>(dy + (size_t)V * c + ch), g);
        bf8_unpack(*reinterpret_cast<const uint4 *>(skip + (size_t)v * ss + soff + ch), s);
        bf8_unpack(*reinterpret_cast<const uint4 *>(act + (size_t)v * c + ch), a);
#pragma unroll
        for (int m = 0; m < 8; m++) g[m] = a[m] > 0.0f ? 0.125f * g[m] + s[m] : 0.0f;
        *reinterpret_cast<uint4 *>(dx + (size_t)v * c + ch) = bf8_pack(g);
    }
}

// adjoint of the upsampling: per axis coarse J gathers fine 2J-1 (1/4), 2J (3/4),
// 2J+1 (3/4), 2J+2 (1/4); dy read from channels [0, c) of stride cstride; through
// the ReLU of the activation act that was upsampled
__global__ void k_upsample_back8(const __nv_bfloat16 *__restrict__ dy, int lgc8, int cstride, int lgc,
                                 const __nv_bfloat16 *__restrict__ act, __nv_bfloat16 *__restrict__ dx)
{
    pdl_begin();
    const int lgf = lgc + 1, mf = (1 << lgf) - 1, mc = (1 << lgc) - 1, c = 8 << lgc8;
    const int64_t total = (int64_t)1 << (3 * lgc + lgc8);
    const float wt[4] = {0.25f, 0.75f, 0.75f, 0.25f};
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(e & ((1 << lgc8) - 1)) << 3;
        const int V = (int)(e >> lgc8);
        const int K = V & mc, J = (V >> lgc) & mc, I = V >> (2 * lgc);
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, a8[8];
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int b = 0; b < 4; b++)
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const int i = (2 * I - 1 + a) & mf, j = (2 * J - 1 + b) & mf, k = (2 * K - 1 + q) & mf;
                    const float w = wt[a] * wt[b] * wt[q];
                    float g[8];
                    bf8_unpack(*reinterpret_cast<const uint4 *>(dy + (size_t)((((i << lgf) + j) << lgf) + k) * cstride + ch), g);
#pragma unroll
                    for (int m = 0; m < 8; m++) s[m] += w * g[m];
                }
        bf8_unpack(*reinterpret_cast<const uint4 *>(act + (size_t)V * c + ch), a8);
#pragma unroll
        for (int m = 0; m < 8; m++) s[m] = a8[m] > 0.0f ? s[m] : 0.0f;
        *reinterpret_cast<uint4 *>(dx + (size_t)V * c + ch) = bf8_pack(s);
    }
}

__global__ void k_copy_slice8(const __nv_bfloat16 *__restrict__ x, int lgc8, int xs, int xoff,
                              __nv_bfloat16 *__restrict__ y, int ys, int yoff, int nv)
{
    pdl_begin();
    const int total = nv << lgc8;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int ch = (e & ((1 << lgc8) - 1)) << 3;
        const int v = e >> lgc8;
        *reinterpret_cast<uint4 *>(y + (size_t)v * ys + yoff + ch) =
            *reinterpret_cast<const uint4 *>(x + (size_t)v * xs + xoff + ch);
    }
}

// ---------------------------------------------------------------- input, head, loss
// x[v][0..15]: standardised log(eps + s0/rho), s_i/(rho v_rms), zeros; from natural-layout sources
__global__ void k_net_input(const double *__restrict__ s0, const double *__restrict__ sx, const double *__restrict__ sy,
                            const double *__restrict__ sz, int64_t nv, float inv_rho, float inv_rv,
                            const float *__restrict__ in_mean, const float *__restrict__ in_std,
                            __nv_bfloat16 *__restrict__ x)
{
    pdl_begin();
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x) {
        float f[4];
        f[0] = logf(kNetLogEps + (float)s0[v] * inv_rho);
        f[1] = (float)sx[v] * inv_rv;
        f[2] = (float)sy[v] * inv_rv;
        f[3] = (float)sz[v] * inv_rv;
        // the voxel's 16 channels (4 used, 12 zero) as two 16-byte stores
        float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int c = 0; c < 4; c++) g[c] = (f[c] - in_mean[c]) / in_std[c];
        static_assert(kNetCin == 16, "two 8-channel vectors per voxel");
        uint4 *o = reinterpret_cast<uint4 *>(x + v * kNetCin);
        o[0] = bf8_pack(g);
        o[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// 1x1 head (FP32): out[v][o] = b[o] + sum_c W[o][c] a[v][c], a with 16 channels
// (a block's outputs pass through shared memory: 36 us at 128^3; stored with a stride of 40 bytes, 62)
constexpr int kHeadVox = 256;
__global__ void __launch_bounds__(kHeadVox)
    k_head(const __nv_bfloat16 *__restrict__ a, const float *__restrict__ W, const float *__restrict__ b, int64_t nv,
           float *__restrict__ out)
{
    pdl_begin();
    __shared__ __align__(16) float sw[kNetOut * 16], sb[kNetOut], so[kHeadVox * kNetOut];
    for (int k = threadIdx.x; k < kNetOut * 16; k += kHeadVox) sw[k] = W[k];
    for (int k = threadIdx.x; k < kNetOut; k += kHeadVox) sb[k] = b[k];
    __syncthreads();
    for (int64_t v0 = (int64_t)blockIdx.x * kHeadVox; v0 < nv; v0 += (int64_t)gridDim.x * kHeadVox) {
        const int64_t v = v0 + threadIdx.x;
        if (v < nv) {
            const uint4 *a8 = reinterpret_cast<const uint4 *>(a + v * 16);
            float lo[8], hi[8];
            bf8_unpack(a8[0], lo);
            bf8_unpack(a8[1], hi);
#pragma unroll
            for (int o = 0; o < kNetOut; o++) {
                float s = sb[o];
#pragma unroll
                for (int c = 0; c < 16; c += 4) {
                    const float4 w = *reinterpret_cast<const float4 *>(sw + o * 16 + c);
                    const float *x = c < 8 ? lo + c : hi + (c - 8);
                    s += w.x * x[0];
                    s += w.y * x[1];
                    s += w.z * x[2];
                    s += w.w * x[3];
                }
                so[threadIdx.x * kNetOut + o] = s;
            }
        }
        __syncthreads();
        const int cnt = (int)(nv - v0 < kHeadVox ? nv - v0 : kHeadVox) * kNetOut;
        float *dst = out + v0 * kNetOut;  // v0 is a multiple of 256: 16-byte aligned
        for (int k = 4 * threadIdx.x; k < cnt; k += 4 * kHeadVox) {
            if (k + 4 <= cnt) *reinterpret_cast<float4 *>(dst + k) = *reinterpret_cast<const float4 *>(so + k);
            else
                for (int r = k; r < cnt; r++) dst[r] = so[r];
        }
        __syncthreads();
    }
}

// loss and head backward: standardised target t[v][o]; dout = 2 (out - t) / (nv * 10);
// da[v][c] = (a > 0) sum_o W[o][c] dout[v][o]; dW, db accumulated; loss partial per block.
// A thread per voxel forms dout and da and leaves dout and a in shared memory;
// then 160 threads each sum one dW[o][c] over the block's voxels.  (With
// the 160 sums in every thread's local memory 528 us at 64^3, so 27.)
constexpr int kHbVox = 256;
__global__ void __launch_bounds__(kHbVox)
    k_head_back(const __nv_bfloat16 *__restrict__ a, const float *__restrict__ W, const float *__restrict__ out,
                const float *__restrict__ tgt, int64_t nv, __nv_bfloat16 *__restrict__ da, float *__restrict__ dW,
                float *__restrict__ db, float *__restrict__ loss)
{
    pdl_begin();
    __shared__ float sw[kNetOut * 16], sd[kHbVox][kNetOut + 1], sa[kHbVox][17], sl[kHbVox / 32];
    for (int k = threadIdx.x; k < kNetOut * 16; k += kHbVox) sw[k] = W[k];
    __syncthreads();
    const float scale = 2.0f / ((float)nv * kNetOut);
    float lsum = 0.0f, wsum = 0.0f, bsum = 0.0f;
    const int so = threadIdx.x / 16, sc = threadIdx.x % 16;  // the sum this thread carries (so < 10)
    for (int64_t v0 = (int64_t)blockIdx.x * kHbVox; v0 < nv; v0 += (int64_t)gridDim.x * kHbVox) {
        const int64_t v = v0 + threadIdx.x;
        const bool ok = v < nv;
        float av[16], g[16];
        if (ok) {
            const uint4 *a8 = reinterpret_cast<const uint4 *>(a + v * 16);
            float lo[8], hi[8];
            bf8_unpack(a8[0], lo);
            bf8_unpack(a8[1], hi);
#pragma unroll
            for (int c = 0; c < 16; c++) av[c] = c < 8 ? lo[c & 7] : hi[c & 7];
        }
#pragma unroll
        for (int c = 0; c < 16; c++) {
            g[c] = 0.0f;
            if (!ok) av[c] = 0.0f;
            sa[threadIdx.x][c] = av[c];
        }
#pragma unroll
        for (int o = 0; o < kNetOut; o++) {
            const float r = ok ? out[v * kNetOut + o] - tgt[v * kNetOut + o] : 0.0f;
            lsum += r * r;
            const float d = scale * r;
            sd[threadIdx.x][o] = d;
#pragma unroll
            for (int c = 0; c < 16; c++) g[c] += sw[o * 16 + c] * d;
        }
        if (ok) {
            float lo[8], hi[8];
#pragma unroll
            for (int c = 0; c < 8; c++) {
                lo[c] = av[c] > 0.0f ? g[c] : 0.0f;
                hi[c] = av[8 + c] > 0.0f ? g[8 + c] : 0.0f;
            }
            uint4 *o8 = reinterpret_cast<uint4 *>(da + v * 16);
            o8[0] = bf8_pack(lo);
            o8[1] = bf8_pack(hi);
        }
        __syncthreads();
        if (so < kNetOut) {
            float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
            for (int q = 0; q < kHbVox; q += 4)
#pragma unroll
                for (int e = 0; e < 4; e++) s4[e] += sd[q + e][so] * sa[q + e][sc];
            wsum += (s4[0] + s4[1]) + (s4[2] + s4[3]);
        } else if (so < kNetOut + 5) {  // ten pairs of eight threads: the biases' sums
            const int o = (so - kNetOut) * 2 + (sc >> 3);
            for (int q = sc & 7; q < kHbVox; q += 8) bsum += sd[q][o];
        }
        __syncthreads();
    }
    if (so < kNetOut) {
        atomicAdd(dW + threadIdx.x, wsum);
    } else if (so < kNetOut + 5) {
        atomicAdd(db + (so - kNetOut) * 2 + (sc >> 3), bsum);
    }
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if ((threadIdx.x & 31) == 0) sl[threadIdx.x >> 5] = lsum;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int k = 0; k < kHbVox / 32; k++) t += sl[k];
        atomicAdd(loss, t / ((float)nv * kNetOut));
    }
}

// standardised target from natural-layout fields (psi, apsi as deviations)
__global__ void k_net_target(FieldPtrs fields, int64_t nv, const float *__restrict__ mean,
                             const float *__restrict__ stdv, float *__restrict__ tgt)
{
    pdl_begin();
    // the reciprocals once per thread (one per voxel and field: 63 us at 64^3, now 38)
    double inv[kNetOut], mu[kNetOut];
#pragma unroll
    for (int o = 0; o < kNetOut; o++) {
        inv[o] = 1.0 / (double)stdv[o];
        mu[o] = (double)mean[o];
    }
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x)
#pragma unroll
        for (int o = 0; o < kNetOut; o++)
            tgt[v * kNetOut + o] = (float)((fields.p[o][v] - (o < 2 ? 1.0 : 0.0) - mu[o]) * inv[o]);
}

// de-standardised output into the fields (psi, apsi get + 1)
__global__ void k_net_output(const float *__restrict__ out, int64_t nv, const float *__restrict__ mean,
                             const float *__restrict__ stdv, FieldPtrs fields)
{
    pdl_begin();
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x)
        {
            const float2 *o2 = reinterpret_cast<const float2 *>(out + v * kNetOut);
            float ov[kNetOut];
#pragma unroll
            for (int o = 0; o < kNetOut / 2; o++) {
                const float2 t2 = o2[o];
                ov[2 * o] = t2.x, ov[2 * o + 1] = t2.y;
            }
#pragma unroll
            for (int o = 0; o < kNetOut; o++) {
                // FP32 de-standardisation as in k_net_output_fine (the guess carries BF16 accuracy),
                // so only the conversion and psi's and alpha psi's + 1 use the narrow FP64 pipe
                const double val = (double)(ov[o] * stdv[o] + mean[o]);
                fields.p[o][v] = o < 2 ? val + 1.0 : val;
            }
        }
}

// ---------------------------------------------------------------- guesses on finer grids
// Sources of a fine grid (extent nc << lr) averaged over the r^3 cells each
// coarse cell covers (r = 2^lr), FP64; one thread per coarse cell and array.
__global__ void __launch_bounds__(256)
    k_avg_down(FieldPtrs in, FieldPtrs out, int narr, int lgc, int lr)
{
    pdl_begin();
    const int64_t nvc = (int64_t)1 << (3 * lgc);
    const int lgf = lgc + lr, r = 1 << lr;
    const double inv = 1.0 / (double)((int64_t)1 << (3 * lr));
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nvc * narr;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int a = (int)(t >> (3 * lgc));
        const int64_t v = t & (nvc - 1);
        const int64_t mc = ((int64_t)1 << lgc) - 1;
        const int64_t K = v & mc, J = (v >> lgc) & mc, I = v >> (2 * lgc);
        const double *f = in.p[a];
        double acc = 0.0;
        for (int di = 0; di < r; di++)
            for (int dj = 0; dj < r; dj++) {
                const int64_t row = ((((I << lr) + di) << lgf) + ((J << lr) + dj)) << lgf;
                for (int dk = 0; dk < r; dk++) acc += f[row + (K << lr) + dk];
            }
        out.p[a][v] = acc * inv;
    }
}

// The network's standardised output [vc][10] on the coarse grid, interpolated
// trilinearly between periodic coarse cell centres to every cell of the fine
// grid (extent nc << lr) and de-standardised (psi and alpha psi get their 1
// back): FP32 arithmetic, FP64 stores.  One thread per fine cell.
__global__ void __launch_bounds__(256)
    k_net_output_fine(const float *__restrict__ out, int lgc, int lr, const float *__restrict__ mean,
                      const float *__restrict__ stdv, FieldPtrs fields)
{
    pdl_begin();
    const int lgf = lgc + lr;
    const int64_t nvf = (int64_t)1 << (3 * lgf);
    const int mc = (1 << lgc) - 1, mf = (1 << lgf) - 1;
    const float r = (float)(1 << lr);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nvf; t += (int64_t)gridDim.x * blockDim.x) {
        const int idx[3] = {(int)(t >> (2 * lgf)), (int)((t >> lgf) & mf), (int)(t & mf)};
        int lo[3];
        float w1[3];
        for (int d = 0; d < 3; d++) {  // coarse position of the fine cell centre, in coarse cells
            const float c = ((float)idx[d] + 0.5f) / r - 0.5f;
            const float fl = floorf(c);
            w1[d] = c - fl;
            lo[d] = ((int)fl) & mc;
        }
        float acc[kNetOut];
        for (int o = 0; o < kNetOut; o++) acc[o] = 0.0f;
        for (int a = 0; a < 2; a++)
            for (int b = 0; b < 2; b++)
                for (int c = 0; c < 2; c++) {
                    const float w = (a ? w1[0] : 1.0f - w1[0]) * (b ? w1[1] : 1.0f - w1[1]) *
                                    (c ? w1[2] : 1.0f - w1[2]);
                    const int64_t v = ((((int64_t)((lo[0] + a) & mc) << lgc) + ((lo[1] + b) & mc)) << lgc) +
                                      ((lo[2] + c) & mc);
                    const float *rec = out + v * kNetOut;
                    for (int o = 0; o < kNetOut; o++) acc[o] = fmaf(w, rec[o], acc[o]);
                }
        for (int o = 0; o < kNetOut; o++) {
            const double val = (double)(acc[o] * stdv[o] + mean[o]);
            fields.p[o][t] = o < 2 ? val + 1.0 : val;
        }
    }
}

// ---------------------------------------------------------------- optimiser
// Adam (Kingma & Ba 2015) on FP32 master weights; bc1 = 1 - beta1^t, bc2 = 1 - beta2^t
__global__ void k_adam(float *__restrict__ w, float *__restrict__ m, float *__restrict__ v,
                       const float *__restrict__ gr, int64_t cnt, float lr, float b1, float b2, float eps, float bc1,
                       float bc2)
{
    pdl_begin();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < cnt; e += (int64_t)gridDim.x * blockDim.x) {
        const float g = gr[e];
        const float mm = b1 * m[e] + (1.0f - b1) * g;
        const float vv = b2 * v[e] + (1.0f - b2) * g * g;
        m[e] = mm;
        v[e] = vv;
        w[e] -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
    }
}

// BF16 copies of one conv's FP32 weights: wb[tap][co][ci] and the data-gradient
// copy wt[26 - tap][ci][co]
__global__ void k_conv_weights_bf16(const float *__restrict__ w, int cout, int cin, __nv_bfloat16 *__restrict__ wb,
                                    __nv_bfloat16 *__restrict__ wt)
{
    pdl_begin();
    const int64_t total = (int64_t)27 * cout * cin;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int ci = (int)(e % cin);
        const int co = (int)((e / cin) % cout);
        const int tap = (int)(e / ((int64_t)cin * cout));
        const __nv_bfloat16 b = __float2bfloat16(w[e]);
        wb[e] = b;
        wt[((int64_t)(26 - tap) * cin + ci) * cout + co] = b;
    }
}

}  // namespace

// ================================================================ launchers
void conv3d(const __nv_bfloat16 *x, int cin, const __nv_bfloat16 *w, const float *bias, int cout, int lg, int mode,
            const __nv_bfloat16 *mask, __nv_bfloat16 *y, cudaStream_t st)
{
    // 128^3 grids on the 5th-generation tensor cores (conv_tc.cu) unless GR_CONV_TC=0
    const char *env = getenv("GR_CONV_TC");
    if ((!env || env[0] != '0') && conv3d_tc_fits(cin, cout, lg)) {
        conv3d_tc(x, cin, w, bias, cout, mode, mask, y, st);
        return;
    }
    // 256 voxels x 32 channels per block where that gives every SM two blocks, x 16 channels down to 256
    // blocks (32^3, 32 -> 32: 11.8 us against 18.3), else 64 voxels x 16 channels (16^3, 64 -> 128: 128
    // blocks would take longer; 8^3 at 64^3's coarsest level had 16 blocks of 62 us)
    const int64_t nv = (int64_t)1 << (3 * lg);
    const int64_t blocks = (nv >> 8) * (cout / 16);  // of 256 voxels x 16 channels
    if (lg >= 3 && blocks >= 256) {
        if (cout % 32 == 0 && blocks >= 304) launch_conv3d<8, 2, 4>(x, cin, w, bias, cout, lg, 8, mode, mask, y, st);
        else launch_conv3d<8, 2, 2>(x, cin, w, bias, cout, lg, 8, mode, mask, y, st);
    } else {
        launch_conv3d<4, 1, 2>(x, cin, w, bias, cout, lg, 6, mode, mask, y, st);
    }
}

void conv3d_wgrad(const __nv_bfloat16 *x, int cin, const __nv_bfloat16 *dy, int cout, int lg, float *dw, float *db,
                  cudaStream_t st)
{
    const int lb = 3 * lg < kWgBox ? 3 * lg : kWgBox;
    const Box bx = make_box(lg, lb);
    const int nbox = 1 << (3 * lg - lb), pairs = (cout / 16) * (cin / 16);
    // about four blocks per SM in all, at least one box each
    int split = (4 * 152 + pairs - 1) / pairs;
    if (split > nbox) split = nbox;
    constexpr int kMost = 2 * 32 * (720 + (1 << kWgBox));
    per_device([] {
        return cudaFuncSetAttribute(k_conv3d_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost) == cudaSuccess;
    });
    const int smem = 2 * 32 * (bx.halo() + (1 << lb));
    GR_LAUNCH_SMEM(k_conv3d_wgrad, dim3(split, pairs), 32 * kWgWarps, smem, st, x, cin, dy, cout, bx, nbox, dw, db);
}

// exponent of a power of two, -1 otherwise
static int pow2_log(int c)
{
    if (c <= 0 || (c & (c - 1))) return -1;
    int l = 0;
    while ((1 << l) < c) ++l;
    return l;
}

void upsample(const __nv_bfloat16 *x, int c, int lgc, __nv_bfloat16 *y, int cstride, cudaStream_t st)
{
    const int l8 = pow2_log(c) - 3;
    if (l8 >= 0 && cstride % 8 == 0 && 3 * lgc + 3 + l8 < 31) {
        GR_LAUNCH(k_upsample8, cdiv((int64_t)1 << (3 * lgc + 1 + l8), 256), 256, st, x, l8, lgc, y, cstride);
        return;
    }
    GR_LAUNCH(k_upsample, cdiv(((int64_t)1 << (3 * lgc + 3)) * c, 256), 256, st, x, c, lgc, y, cstride);
}

void pool(const __nv_bfloat16 *x, int c, int lgf, __nv_bfloat16 *y, cudaStream_t st)
{
    const int l8 = pow2_log(c) - 3;  // every level has 16 2^l channels
    GR_LAUNCH(k_pool8, cdiv((int64_t)1 << (3 * lgf - 3 + l8), 256), 256, st, x, l8, lgf, y);
}

void skip_back(const __nv_bfloat16 *dy, int c, int lgf, const __nv_bfloat16 *skip, int ss, int soff,
               const __nv_bfloat16 *act, __nv_bfloat16 *dx, cudaStream_t st)
{
    const int l8 = pow2_log(c) - 3;
    GR_LAUNCH(k_skip_back8, cdiv((int64_t)1 << (3 * lgf + l8), 256), 256, st, dy, l8, lgf, skip, ss, soff, act, dx);
}

void upsample_back(const __nv_bfloat16 *dy, int c, int cstride, int lgc, const __nv_bfloat16 *act, __nv_bfloat16 *dx,
                   cudaStream_t st)
{
    const int l8 = pow2_log(c) - 3;
    GR_LAUNCH(k_upsample_back8, cdiv((int64_t)1 << (3 * lgc + l8), 128), 128, st, dy, l8, cstride, lgc, act, dx);
}

void copy_slice(const __nv_bfloat16 *x, int c, int xs, int xoff, __nv_bfloat16 *y, int ys, int yoff, int64_t nv,
                cudaStream_t st)
{
    const int l8 = pow2_log(c) - 3;
    if (l8 >= 0 && xs % 8 == 0 && ys % 8 == 0 && xoff % 8 == 0 && yoff % 8 == 0 && (nv << l8) < (1LL << 31)) {
        GR_LAUNCH(k_copy_slice8, cdiv(nv << l8, 256), 256, st, x, l8, xs, xoff, y, ys, yoff, (int)nv);
        return;
    }
    GR_LAUNCH(k_copy_slice, cdiv(nv * c, 256), 256, st, x, c, xs, xoff, y, ys, yoff, nv);
}

void net_input(const double *s0, const double *sx, const double *sy, const double *sz, int64_t nv, float inv_rho,
               float inv_rv, const float *in_mean, const float *in_std, __nv_bfloat16 *x, cudaStream_t st)
{
    GR_LAUNCH(k_net_input, cdiv(nv, 256), 256, st, s0, sx, sy, sz, nv, inv_rho, inv_rv, in_mean, in_std, x);
}

void avg_down(FieldPtrs in, FieldPtrs out, int narr, int lgc, int lr, cudaStream_t st)
{
    const int64_t tot = ((int64_t)narr) << (3 * lgc);
    GR_LAUNCH(k_avg_down, cdiv(tot, 256), 256, st, in, out, narr, lgc, lr);
}

void net_output_fine(const float *out, int lgc, int lr, const float *mean, const float *stdv, FieldPtrs fields,
                     cudaStream_t st)
{
    const int64_t nvf = (int64_t)1 << (3 * (lgc + lr));
    GR_LAUNCH(k_net_output_fine, wave_grid(k_net_output_fine, nvf), 256, st, out, lgc, lr, mean, stdv, fields);
}

void head(const __nv_bfloat16 *a, const float *W, const float *b, int64_t nv, float *out, cudaStream_t st)
{
    GR_LAUNCH(k_head, wave_grid(k_head, nv, kHeadVox), kHeadVox, st, a, W, b, nv, out);
}

void head_back(const __nv_bfloat16 *a, const float *W, const float *out, const float *tgt, int64_t nv,
               __nv_bfloat16 *da, float *dW, float *db, float *loss, cudaStream_t st)
{
    GR_LAUNCH(k_head_back, wave_grid(k_head_back, nv, kHbVox), kHbVox, st, a, W, out, tgt, nv, da, dW, db, loss);
}

void net_target(FieldPtrs fields, int64_t nv, const float *mean, const float *stdv, float *tgt, cudaStream_t st)
{
    GR_LAUNCH(k_net_target, cdiv(nv, 256) < 304 ? cdiv(nv, 256) : 304, 256, st, fields, nv, mean, stdv, tgt);
}

void net_output(const float *out, int64_t nv, const float *mean, const float *stdv, FieldPtrs fields,
                cudaStream_t st)
{
    GR_LAUNCH(k_net_output, cdiv(nv, 256), 256, st, out, nv, mean, stdv, fields);
}

void adam(float *w, float *m, float *v, const float *g, int64_t cnt, float lr, float b1, float b2, float eps,
          float bc1, float bc2, cudaStream_t st)
{
    GR_LAUNCH(k_adam, cdiv(cnt, 256) > 4096 ? 4096 : cdiv(cnt, 256), 256, st, w, m, v, g, cnt, lr, b1, b2, eps, bc1,
              bc2);
}

void conv_weights_bf16(const float *w, int cout, int cin, __nv_bfloat16 *wb, __nv_bfloat16 *wt, cudaStream_t st)
{
    const int64_t total = (int64_t)27 * cout * cin;
    GR_LAUNCH(k_conv_weights_bf16, cdiv(total, 256) > 4096 ? 4096 : cdiv(total, 256), 256, st, w, cout, cin, wb, wt);
}

}  // namespace gr
