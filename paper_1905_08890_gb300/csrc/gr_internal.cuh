// gr_internal.cuh - shared definitions of the CUDA library (not part of the C ABI).
//
// Multigrid level arrays use a red-black split layout: on a level of extent
// n (a power of two, n >= 2) the cell (i, j, k) of colour c = (i + j + k) & 1
// lives at
//     c * n^3/2 + (i * n + j) * (n/2) + (k >> 1).
// A red cell's six neighbours are black cells at the same half-index q = k>>1
// in rows (i +- 1, j) and (i, j +- 1), and at q and q + (p ? 1 : -1) in its own
// row, p = (i + j + c) & 1 the parity of k.  A colour pass therefore reads one
// contiguous half-array and writes the other, with no idle threads, and the
// 8 children of a coarse cell (I, J, K) all sit at q = K in rows (2I + a, 2J + b).
// Caller-facing fields and sources use the natural [n][n][n] layout.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include <atomic>
#include <mutex>
#include <unordered_map>

#include "device_once.cuh"
#include "df64.cuh"

namespace gr {

// kernels launched by this library since load; every launch goes through GR_LAUNCH
extern std::atomic<long long> g_launches;

// Every kernel is launched with programmatic dependent launch: the next kernel
// of the stream may be scheduled onto the SMs while its predecessor drains
// (its launch latency and block start-up overlap the predecessor's last
// blocks), and every kernel begins with pdl_begin(), which waits for the
// predecessor's completion and memory before anything else, so the stream's
// order of effects is that of plain launches.
template <class T>
struct ident {
    using type = T;
};
template <typename... KArgs>
inline void launch_pdl(void (*k)(KArgs...), dim3 g, dim3 b, size_t smem, cudaStream_t st,
                       typename ident<KArgs>::type... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = b;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k, args...) != cudaSuccess) {
        // a stream that takes no programmatic serialization (the legacy default
        // stream may not): a plain launch, whose error, if any, stays recorded
        cudaGetLastError();
        cfg.numAttrs = 0;
        cudaLaunchKernelEx(&cfg, k, args...);
    }
}
#define GR_LAUNCH(kernel, grid, block, stream, ...)                              \
    do {                                                                         \
        ::gr::launch_pdl(kernel, (grid), (block), 0, (stream), __VA_ARGS__);      \
        ::gr::g_launches.fetch_add(1, std::memory_order_relaxed);                \
    } while (0)
#define GR_LAUNCH_SMEM(kernel, grid, block, smem, stream, ...)                   \
    do {                                                                         \
        ::gr::launch_pdl(kernel, (grid), (block), (smem), (stream), __VA_ARGS__); \
        ::gr::g_launches.fetch_add(1, std::memory_order_relaxed);                \
    } while (0)

// f() once for each device it is called on (a kernel's attributes, such as its dynamic shared
// memory, belong to one device), its result on every call.  One set-up per type F: call it with a lambda.
template <class F>
bool per_device(F &&f)
{
    static DeviceOnce once;
    int dev = 0;
    cudaGetDevice(&dev);
    return once(dev, f);
}

#ifdef __CUDACC__
// First statement of every kernel: let the stream's next kernel launch, then
// wait for the previous one (a no-op for a kernel launched without the attribute).
// The wait alone does not hold back every load that follows it: what a kernel reads
// through const __restrict__ pointers or __ldg counts as constant while it runs, and the
// compiler moved such loads above the wait (a list's length was read before the kernel that
// writes it had ended).  A load may not be moved above a branch that decides whether it is made,
// so a branch the compiler cannot decide follows the wait: no SM has the number 2^32 - 1.
__device__ __forceinline__ void pdl_begin()
{
    unsigned sm;
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;\n\tmov.u32 %0, %%smid;" : "=r"(sm)::"memory");
    if (sm == 0xffffffffu) {
        asm volatile("exit;");
        __builtin_unreachable();
    }
}
#endif

// Kernels of the finest level take `rev`: nonzero walks their index range
// from the end, so a launch that follows one walking forward starts where it
// stopped, on data still in L2.

// Blocks for a grid-stride kernel over `threads` threads: one full wave (as
// many blocks per SM as the kernel's registers allow, on every SM) or fewer
// when the work is smaller.  Every block then takes the same number of
// grid-stride iterations to within one, where a fixed block count that is not
// a multiple of the wave leaves a partial last wave with most SMs idle.
inline int wave_grid_of(const void *kernel, int64_t threads, int block)
{
    static std::mutex mu;
    static std::unordered_map<const void *, int> per_sm;
    static int sms = 0;
    int b = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (sms == 0) {
            int dev = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (sms <= 0) sms = 1;
        }
        auto it = per_sm.find(kernel);
        if (it == per_sm.end()) {
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, block, 0) != cudaSuccess || b <= 0) {
                cudaGetLastError();
                b = 1;
            }
            per_sm[kernel] = b;
        } else {
            b = it->second;
        }
    }
    const int64_t need = (threads + block - 1) / block;
    const int64_t wave = (int64_t)sms * b;
    return (int)(need < 1 ? 1 : (need < wave ? need : wave));
}

template <class Kernel>
int wave_grid(Kernel kernel, int64_t threads, int block = 256)
{
    return wave_grid_of(reinterpret_cast<const void *>(kernel), threads, block);
}

// sets the thread's message returned by gr_last_error()
void set_last_error(const char *msg);

constexpr double kPi = 3.14159265358979323846;

enum Kind : int { KPOISSON = 0, KHELM = 1, KPSI = 2 };

constexpr int kBlock = 256;
constexpr int kMaxRedBlocks = 152 * 16;  // blocks of the norm/mean reductions (16 per SM)
constexpr int kCoarsestSweeps = 32;  // red-black sweeps on the 2^3 level

// Where a kernel that reduces leaves its two sums: per-block partials, whose
// sum (in a fixed order) the last block to finish writes to out[0], out[1]
// and, if given, to mapped[0], mapped[1] (device alias of pinned host memory),
// then seq to *flag (likewise).  A launch of its own for that sum cost 2.3 us
// behind every residual, and another 2 us for the store to the host.  ticket:
// a counter that is zero between launches; launches that share it must be
// ordered.  partials == nullptr: no sums are wanted.
struct Sums {
    double *partials = nullptr, *out = nullptr;
    unsigned *ticket = nullptr;
    double *mapped = nullptr, *flag = nullptr;
    double seq = 0.0;
};

#ifdef __CUDACC__
// the first red relaxation of a Poisson correction from e = 0 (rounded as if stored: not contracted into the sum it enters)
__device__ __forceinline__ float first_red(float r, float h2) { return __fmul_rn(__fmul_rn(-h2, r), 1.0f / 6.0f); }

// The divisions for recip64's rare operands, out of line so that they do not occupy the common path
static __device__ __noinline__ double recip64_any(double x) { return 1.0 / x; }

// 1/x by Newton's iteration r <- r + r (1 - x r) from the hardware's 20-bit
// estimate: two steps leave at most one unit in the last place.  The iteration has no zeros, infinities
// and subnormals (of x or of the result): those x are divided
__device__ __forceinline__ double recip64(double x)
{
    const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    if (ex - 1u > 2043u) return recip64_any(x);
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// 1/sqrt(a), a >= 1: the FP32 estimate and one third-order step
// y <- y (1 + e/2 + 3 e^2/8), e = 1 - a y^2 (the binomial series of (1 - e)^-1/2): at most two units in the last place
__device__ __forceinline__ double rsqrt64(double a)
{
    if (!(a < 0x1p120)) return rsqrt(a);
    // a's leading 24 bits as a float and y back, by moving exponent and mantissa
    const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
    const float f = __uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29));
    const unsigned yb = __float_as_uint(rsqrtf(f));
    const double y = __hiloint2double((int)((yb >> 3) + (896u << 20)), (int)(yb << 29));
    const double e = fma(-a * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Sums of a and b over the warp's lanes: lane 0 returns a's, lane 16 b's.  The lower half goes on with a
// and the upper with b: five FP64 additions a warp instead of ten, each of which holds the FP64 pipe
// for 16 cycles.
__device__ __forceinline__ double warp_sum2(double a, double b)
{
    const bool up = (threadIdx.x & 16) != 0;
    const double o = __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
    double v = (up ? b : a) + o;
#pragma unroll
    for (int k = 8; k > 0; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
    return v;
}

// the same over the kBlock threads of a block, returned by lanes 0 and 16 of the first warp (which
// alone continues: the others return false); s: 2 kBlock / 32 doubles
__device__ __forceinline__ bool block_sum_pair(double a, double b, double *s, double *v)
{
    constexpr int W = kBlock / 32;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const double t = warp_sum2(a, b);
    if ((l & 15) == 0) s[(l >> 4) * W + w] = t;
    __syncthreads();
    if (w != 0) return false;
    double u = (l & 15) < W ? s[(l >> 4) * W + (l & 15)] : 0.0;
#pragma unroll
    for (int k = W / 2; k > 0; k >>= 1) u += __shfl_xor_sync(0xffffffffu, u, k);
    *v = u;
    return true;
}

// the end of a reducing kernel, by every thread of the block, after lanes 0 and 16 of
// the first warp wrote the block's partials
__device__ __forceinline__ void last_block_sum(const Sums &S)
{
    __shared__ bool last;
    __shared__ double la[2 * (kBlock / 32)];
    if (threadIdx.x < 32) {
        __threadfence();
        __syncwarp();
        if (threadIdx.x == 0) last = atomicInc(S.ticket, gridDim.x - 1) == gridDim.x - 1;  // wraps to zero
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double a = 0.0, b = 0.0;
    for (unsigned q = threadIdx.x; q < gridDim.x; q += kBlock) {
        const double2 p = __ldcg(reinterpret_cast<const double2 *>(S.partials) + q);
        a += p.x;
        b += p.y;
    }
    double v;
    if (!block_sum_pair(a, b, la, &v)) return;
    const double vb = __shfl_sync(0xffffffffu, v, 16);
    if (threadIdx.x == 0) {
        S.out[0] = v;
        S.out[1] = vb;
        if (S.mapped) {
            S.mapped[0] = v;
            S.mapped[1] = vb;
            __threadfence_system();
            if (S.flag) *(volatile double *)S.flag = S.seq;
        }
    }
}

// Block sums of a and b (blockDim.x == kBlock) into out[2 blockIdx.x + 0/1],
// in a fixed order.
__device__ __forceinline__ void block_sum2(double a, double b, double *out)
{
    __shared__ double sa[2 * (kBlock / 32)];
    double v;
    if (block_sum_pair(a, b, sa, &v) && (threadIdx.x & 15) == 0) out[2 * blockIdx.x + (threadIdx.x >> 4)] = v;
}

// Sums of a and b over the grid
__device__ __forceinline__ void block_sum2(double a, double b, const Sums &S)
{
    block_sum2(a, b, S.partials);
    last_block_sum(S);
}

// The same for FP32 inputs: warp sums in FP32 (for norms, where the rounding
// of partial sums is harmless), the per-warp totals in FP64.  GB300's FP64
// pipe is narrow enough that a full FP64 warp reduction per thread costs a
// noticeable share of a memory-sized kernel.
__device__ __forceinline__ void block_sum2f(float a, float b, const Sums &S)
{
    constexpr int W = kBlock / 32;
    __shared__ double sa[2 * W];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        sa[w] = (double)a;
        sa[W + w] = (double)b;
    }
    __syncthreads();
    if (w == 0) {
        double u = (l & 15) < W ? sa[(l >> 4) * W + (l & 15)] : 0.0;
#pragma unroll
        for (int k = W / 2; k > 0; k >>= 1) u += __shfl_xor_sync(0xffffffffu, u, k);
        if ((l & 15) == 0) S.partials[2 * blockIdx.x + (l >> 4)] = u;
    }
    last_block_sum(S);
}
#endif

// ---- multigrid kernels (templated on the working precision T) ---------------
// One Gauss-Seidel pass over colour `color` of a level.  KPOISSON: f;
// KHELM: f and c1 = 1/(6 + h^2 m); KPSI (double only): f, c0 = s0, c1 = AA,
// unknown u = psi - 1, one Newton step per cell.
template <typename T>
void sweep_colour(int kind, int n, T *u, const T *f, const T *c0, const T *c1, double h2, double ih2, double rho,
                  int color, cudaStream_t st, int rev = 0);
// KPOISSON, n >= 8: the black pass that follows the first red one from e = 0, with the red values
// -h^2 r / 6 formed here from r instead of read from e (whose red half nothing need write)
void sweep_black_from_r(int n, float *e, const float *r, double h2, cudaStream_t st, int rev = 0);

// Residual eps = L(u) - f of the fine level restricted to the coarse level.
// Correction form (fas = 0): fc = -R eps, uc = 0.  FAS (fas = 1, KPSI):
// fc = R eps, uc = urc = R u.  c0 is m for KHELM (the operator), s0 for KPSI.
// red_only (linear kinds, right after a black relaxation pass): the black
// children's residuals, zero up to rounding, count as zero.
template <typename T>
void resid_restrict(int kind, int nf, const T *u, const T *f, const T *c0, const T *c1, double ih2, double rho, T *uc,
                    T *fc, T *urc, int fas, cudaStream_t st, bool red_only = false);
// FP32 correction form of the same (KPOISSON or KHELM with m) right after a
// black relaxation pass: only the red children's residuals enter the average,
// the black ones being zero up to rounding.  h2c > 0: the coarse correction
// ec receives the coarse level's first red relaxation from zero instead of
// zeros (cinv: the coarse KHELM inverse diagonal), so that pass is skipped.
void resid_restrict_red(int kind, int nf, const float *e, const float *r, const float *m, double ih2, float *ec,
                        float *rc, const float *cinv, double h2c, cudaStream_t st, int rev = 0);

// FAS coarse right-hand side: fc = N(uc) - fc (KPSI, double).
void fas_rhs(int nc, const double *uc, double *fc, const double *c0, const double *c1, double ih2, double rho,
             cudaStream_t st);
// uc -= urc (the FAS coarse correction).
void fas_diff(int nc, double *uc, const double *urc, cudaStream_t st);

// Fine u += P(uc), cell-centred trilinear.
template <typename T>
void prolong_add(int nf, T *u, const T *uc, cudaStream_t st);
// FP64, black_only when a red pass of a linear equation follows
void prolong_add64(int nf, double *u, const double *uc, bool black_only, cudaStream_t st);
// FP32, black children only (a red relaxation of a linear equation follows)
void prolong_add_black(int nf, float *u, const float *uc, cudaStream_t st, int rev = 0);
// FP32 coarse = 8-child average of fine (a right-hand side going down)
void restrict_avg(int nf, const float *fine, float *coarse, cudaStream_t st);

// The 2^3 level in FP64 (any T storage).  KPOISSON, KHELM: solved exactly
// (Walsh-Hadamard diagonalisation; Gauss-Jordan elimination), Poisson with
// the source mean removed before and the solution mean after; KHELM reads
// c0 = m.  KPSI: kCoarsestSweeps Newton red-black sweeps, each followed by
// the constant shift that zeroes the sum of the eight residuals to first
// order (the Laplacian leaves that mode to the weak non-Laplacian terms).
template <typename T>
void coarsest(int kind, T *u, T *f, const T *c0, const T *c1, double h2, double ih2, double rho, cudaStream_t st);

// Coarse coefficients.  KPSI: c0c = R c0f, c1c = R c1f.  KHELM: c0c = R c0f
// (m) and c1c = 1/(6 + h2c c0c).
template <typename T>
void restrict_coef(int kind, int nf, const T *c0f, const T *c1f, T *c0c, T *c1c, double h2c, cudaStream_t st);
// KHELM inverse diagonal on one level: c1 = 1/(6 + h2 c0).
template <typename T>
void helm_invdiag(int n, const T *c0, T *c1, double h2, cudaStream_t st);

// Sums of eps^2 and of u over a level (split layout);
// eps_nat (may be null) receives eps in natural layout (double).
template <typename T>
void resid_norm(int kind, int n, const T *u, const T *f, const T *c0, const T *c1, double ih2, double rho,
                const Sums &sums, double *eps_nat, cudaStream_t st);
// The FP32 correction cycle's levels coarse_tail_n()^3 .. 2^3 in one thread
// block (shared memory): e/r/m/inv of levels 2^3, 4^3, 8^3, 16^3 (index 0 =
// 2^3); e and r of the top tail level in and e out; h2 per level.
int coarse_tail_n();
void coarse_tail(int kind, float *const *e, float *const *r, const float *const *m, const float *const *inv,
                 const double *h2, int nu1, int nu2, cudaStream_t st);

// The FP32 correction cycle's levels 64^3 .. 2^3 in one 16-CTA thread-block
// cluster (coarse_cluster.cu): arrays of levels 2^3 .. 64^3 (index 0 = 2^3);
// e and r of 64^3 in (its first red pass made by the restriction), e out.
// Needs nu1, nu2 >= 1.  coarse_cluster_ok: the device runs such a cluster
// (KPOISSON, KHELM).
bool coarse_cluster_ok(int kind);
void coarse_cluster(int kind, float *const *e, float *const *r, const float *const *m, const float *const *inv,
                    const double *h2, const double *ih2, int nu1, int nu2, cudaStream_t st);

// A level of 32^3 or 64^3 smoothed in one launch per direction
// (level_fused.cu; linear kinds, nu1 = nu2 = 2).  level_down: the pre-smoothing
// and the restriction: from_r starts from e = 0 (first red pass from r),
// otherwise e's red half holds the first red pass; eb receives the black half,
// rc the coarse right-hand side and ec (may be null) the coarse correction's
// start as resid_restrict_red writes it (h2c = 0: zeros).  level_up: the
// black half eb corrected from ec, then the post-smoothing; the result goes to
// e or, with uh and ul, is added to the double-float unknown.
bool level_fused_fits(int kind, int n, int nu1, int nu2);
void level_down(int kind, int n, bool from_r, const float *e, float *eb, const float *r, const float *m,
                const float *inv, double h2, double ih2, float *ec, float *rc, const float *cinv, double h2c,
                cudaStream_t st);
void level_up(int kind, int n, float *e, const float *eb, const float *r, const float *inv, const float *ec, double h2,
              float *uh, float *ul, cudaStream_t st);

// Levels 2 << top .. 2^3 (top = 1 .. 3) of an FP64 V-cycle in one 16-CTA
// cluster launch (fp64_tail.cu): u and f of the top level in, u out; c0, c1, h2
// and ih2 of levels 2^3 (index 0) .. top.  tail64_ok: the device runs such a cluster.
bool tail64_ok(int kind);
void tail64(int kind, int top, double *u, const double *f, const double *const *c0, const double *const *c1,
            const double *h2, const double *ih2, double rho, int nu1, int nu2, cudaStream_t st);

// ---- mixed precision -------------------------------------------------------
// FP64 residual on the fine level; writes r32 = -eps (split), and for KPSI
// the Jacobian coefficient m32 = -dN/du > 0 and its inverse diagonal inv32.
void mixed_resid(int kind, int n, const double *u, const double *f, const double *c0, const double *c1, double ih2,
                double h2, double rho, float *r32, float *m32, float *inv32, const Sums &sums, cudaStream_t st);
// u64 += e32 (split layout).
void mixed_update(int n, double *u, const float *e, cudaStream_t st);
// c32 = (float) c64.
void to_float(int64_t cnt, const double *a, float *b, cudaStream_t st);

// ---- double-float fine level (df_kernels.cu) -------------------------------
// hi/lo = a split into FP32 pairs; a = hi + lo.
// Fine residual in double-float: r32 = -eps, KPSI also m32/inv32 (Newton
// coefficient and FP32 inverse diagonal).  f, a = c0, b = c1 are pairs
// premultiplied by h^2 (KPOISSON, KHELM: h^2 f, h^2 m; KPSI: f' = h^2 f,
// a' = 2 pi h^2 s0, b' = h^2 AA / 8).  When e32 is not null it also writes the
// first red relaxation of the correction cycle from e = 0 (inv_in: the KHELM
// inverse diagonal).  Sums: of (eps/ref)^2.
void df_resid(int kind, int n, const float *uh, const float *ul, const float *fh, const float *fl, const float *ah,
             const float *al, const float *bh, const float *bl, double h2, double rho, double ref, float *r32,
             float *m32, float *inv32, const float *inv_in, float *e32, const Sums &sums, cudaStream_t st, int rev = 0,
             const double *fshift = nullptr);
void df_update(int n, float *uh, float *ul, const float *e, cudaStream_t st);
// last black pass of the FP32 correction cycle (KPOISSON or KHELM, n >= 8)
// fused with u += e on both colours; e's black half is left unwritten
void df_black_update(int kind, int n, const float *e, const float *r, const float *inv, double h2, float *uh,
                     float *ul, cudaStream_t st, int rev = 0);

// ---- double-float set-up and write-back (df_setup.cu) -----------------------
// Natural FP64 inputs -> split-layout hi/lo pairs, right-hand sides and
// coefficients premultiplied by h^2 as df_resid takes them (the callers pass
// the scales with h^2 folded in).  sums: sum and sum of squares of the high
// parts of the quantity named.
void dfs_sum(int64_t cnt, const double *a, const Sums &sums, cudaStream_t st);                      // a
void dfs_pair_sum(int64_t cnt, const float *h, const float *l, const Sums &sums, cudaStream_t st);  // h + l
// f = scale (s - sum[0]/n^3), u = fld; sums of f
void dfs_mean_rhs(int n, const double *s, const double *sum, double scale, const double *fld, float *uh, float *ul,
                 float *fh, float *fl, const Sums &sums, cudaStream_t st);
// f = scale sum_l (F_l(+l) - F_l(-l)), u = fld; sums of f
void dfs_div_rhs(int n, double scale, const double *Fx, const double *Fy, const double *Fz, const double *fld,
                float *uh, float *ul, float *fh, float *fl, const Sums &sums, cudaStream_t st);
// f = scale sum_l ((A^{comp l} w)(+l) - (A^{comp l} w)(-l)), u = fld; sums of f
void dfs_shift_rhs(int n, double scale, const float *A, const float *wh, const float *wl, int comp, const double *fld,
                  float *uh, float *ul, float *fh, float *fl, const Sums &sums, cudaStream_t st);
// A_ij (12 n^3 floats: component c hi at A + 2c n^3, lo at A + (2c+1) n^3) and AA pairs, natural layout;
// scratch: four arrays of 2 n^3 floats for the pairs of V_x, V_y, V_z, U
void dfs_aij(int n, double inv2h, double ih2, const double *Vx, const double *Vy, const double *Vz, const double *U,
             float *const scratch[4], float *A, float *AAh, float *AAl, cudaStream_t st);
// psi: u = psi - 1, a = 2 pi h^2 s0, b = h^2 AA / 8, f = 0; sums of s0
void dfs_psi(int n, double h2, const double *psi, const double *s0, const float *AAh, const float *AAl, float *uh,
            float *ul, float *ah, float *al, float *bh, float *bl, float *fh, float *fl, const Sums &sums,
            cudaStream_t st);
// alpha psi: u = alpha psi - 1, a = h^2 m, f = h^2 (m - psi^5 Kdot), m32, inv32; sums of psi^5 Kdot
void dfs_apsi(int n, double h2, const double *psi, const double *apsi, const double *s0, const double *sig,
             const float *AAh, const float *AAl, double K2, double Kdot, float *uh, float *ul, float *ah, float *al,
             float *fh, float *fl, float *m32, float *inv32, const Sums &sums, cudaStream_t st);
// w = alpha psi psi^-7 pairs, natural layout
void dfs_weight(int n, const double *psi, const double *apsi, float *wh, float *wl, cudaStream_t st);
// out (natural) = hi + lo - sum[0]/n^3 (sum may be null) + (dev ? 1 : 0)
void dfs_store(int n, const float *uh, const float *ul, const double *sum, int dev, double *out, cudaStream_t st);

// ---- sources, coefficients, layouts (field_kernels.cu) ---------------------
// zeros into the five source arrays of cnt (even) doubles each: one launch (five memsets cost a small
// deposit of 12345 particles on 32^3 cells 28.7 us, so 13.0)
void clear5(int64_t cnt, double *const f[5], cudaStream_t st);
// the deposit kernel, one thread per particle, adding to the five arrays (no zeroing)
void deposit_add(int n, double L, int64_t np, const double *x, const double *u, double mass, double *s0, double *sx,
                 double *sy, double *sz, double *sig, cudaStream_t st);
// The same over tiles of 8^3 cells (deposit_tiles.cu), psi null: the plain
// deposit, else with the metric's Lorentz factor; x, u: [3][stride], np of them;
// adds to the five arrays (add: other launches have added to them already;
// otherwise they hold zeros).  scratch: device memory.  deposit_tiles_fit: the
// particles fill the grid well enough for it, the charge mass / h^3 is in its
// range and the scratch suffices.
bool deposit_tiles_fit(int n, double L, int64_t np, double mass, bool metric, size_t scratch);
void deposit_tiles(int n, double L, int64_t np, int64_t stride, const double *x, const double *u, double mass,
                   const double *psi, double *s0, double *sx, double *sy, double *sz, double *sig, void *scratch,
                   size_t bytes, bool add, cudaStream_t st);
// Sums of a and a^2 over cnt doubles.
void sum_sq(int64_t cnt, const double *a, const Sums &sums, cudaStream_t st);
// a[i] = scale * (a[i] - s[0] / cnt_total), s a device scalar (a sum).
void scale_sub_mean(int64_t cnt, double *a, const double *sum, double inv_cnt, double scale, cudaStream_t st);
// natural -> split with a shift: split = nat + shift; split -> natural:
// nat = split + shift - sum[0] * inv_cnt (sum may be null).
void to_split(int n, const double *nat, double *split, double shift, cudaStream_t st);
void from_split(int n, const double *split, double *nat, double shift, const double *sum, double inv_cnt,
                cudaStream_t st);
// f (split) = scale * div3(F) from natural F (3-point central differences).
void div_to_split(int n, double inv2h, const double *Fx, const double *Fy, const double *Fz, double scale, double *f,
                  cudaStream_t st);
// A_ij (6 natural arrays: xx yy zz xy xz yz; A null: not stored) and AA (natural) from V, U.
void aij_aa(int n, double inv2h, double ih2, const double *Vx, const double *Vy, const double *Vz, const double *U,
            double *A, double *AA, cudaStream_t st);
// psi equation: u = psi - 1, c0 = s0, c1 = AA, f = 0 (split); sums of s0 and s0^2.
void psi_setup(int n, const double *psi, const double *s0, const double *AA, double *u, double *c0, double *c1,
               double *f, const Sums &sums, cudaStream_t st);
// alpha psi equation: u = apsi - 1, c0 = m, c1 = 1/(6 + h^2 m), f = m - psi^5 Kdot (split);
// g = psi^5 Kdot (natural scratch) for the reference norm.
void apsi_setup(int n, double h2, const double *psi, const double *apsi, const double *s0, const double *sig,
                const double *AA, double K2, double Kdot, double *u, double *c0, double *c1, double *f, double *g,
                cudaStream_t st);
// B^i source: f (split) = 2 sum_j D_j (w A^ij), w = apsi psi^-7 (natural scratch).
void shift_weight(int n, const double *psi, const double *apsi, double *w, cudaStream_t st);
void shift_source(int n, double inv2h, const double *A, const double *w, int comp, double *f, cudaStream_t st);

// ---- particles (particle_kernels.cu) ----------------------------------------
// The per-cell records of the particle update: 20 FP32 quantities (alpha - 1,
// psi - 1, beta^j, D_i alpha, D_i psi, D_i beta^j at 11 + 3 j + i), 80 bytes
// per cell (rec: 20 n^3 floats, 16-byte aligned), from the natural FP64
// fields; dev is FP32 scratch of 5 n^3 floats.
void particle_fields(int n, double L, const double *psi, const double *apsi, const double *Bx, const double *By,
                     const double *Bz, const double *b, float *dev, float *rec, cudaStream_t st);
// Kicks and drift of np particles (x, u: [3][np] device SoA) with the flags
// GR_KICK_SYNC, GR_KICK_OPEN, GR_DRIFT.
void particle_update(int n, double L, int64_t np, double *x, double *u, const float *rec, double dt, int flags,
                     cudaStream_t st);
// The deposit with W = sqrt(1 + psi^-4 |u|^2), psi interpolated at the particle.
// One thread per particle, adding to the five arrays.
void deposit_metric_add(int n, double L, int64_t np, const double *x, const double *u, double mass, const double *psi,
                        double *s0, double *sx, double *sy, double *sz, double *sig, cudaStream_t st);

// ---- code units (codeunits.cu) ----------------------------------------------
struct CuPtrs {
    double *p[10];  // sources: s0 s_x s_y s_z sigma; fields: psi apsi V_x V_y V_z U B^x B^y B^z b
};
struct CuScale {
    double s[5];   // source scales (code units -> the a = 1 problem)
    double f[10];  // field scales of the potentials (entries 2..9)
};
// code-unit sources -> scaled copies; code-unit fields -> the a = 1 form, in place
void code_units_in(int64_t N, const CuPtrs &src_in, const CuPtrs &src_out, const CuScale &sc, const CuPtrs &fld,
                   double a2c2, cudaStream_t st);
// the a = 1 solution -> code-unit fields, in place
void code_units_out(int64_t N, const CuScale &sc, const CuPtrs &fld, double a2c2, cudaStream_t st);

// ---------------------------------------------------------------- nested patches
// Base level as the patch kernels see it: natural FP64 fields (PB_NAT, nat),
// the FP64 split-layout arrays of a solve (PB_SPLIT: u, f, c0, c1 as the
// FP64 relaxation uses them) or the double-float split-layout arrays
// (PB_DF: uh/ul, fh/fl = h^2 f, ah/al, bh/bl = the h^2-scaled coefficients).
enum PatchBaseFmt : int { PB_NAT = 0, PB_SPLIT = 1, PB_DF = 2 };
struct PBase {
    int lgn = 0;
    const double *nat = nullptr;
    double *u = nullptr, *f = nullptr;
    const double *c0 = nullptr, *c1 = nullptr;
    float *uh = nullptr, *ul = nullptr, *fh = nullptr, *fl = nullptr;
    const float *ah = nullptr, *al = nullptr, *bh = nullptr, *bl = nullptr;
    double h2 = 0, ih2 = 0, rho = 0;
};
// One patch level: ghosted (n + 4)^3 arrays; co/cnc the block its child
// covers (cnc = 0: none); lam the Poisson solvability constant (NULL: none).
// The working unknown is u (FP64) or the pair uh/ul (the double-float
// relaxation of the mixed modes, with the h^2-scaled pairs fh/fl, ah/al,
// bh/bl of the right-hand side and coefficients, cpr = 2 pi rho h^2 and
// c5 = 10 pi rho h^2); f, c0, c1 are the FP64 right-hand side and
// coefficients (Helmholtz c1: 1 / (6 + h^2 m)).
struct PPatch {
    int lgn = 0, m = 0;
    double *u = nullptr, *f = nullptr;
    const double *c0 = nullptr, *c1 = nullptr;
    float *uh = nullptr, *ul = nullptr, *fh = nullptr, *fl = nullptr;
    float *ah = nullptr, *al = nullptr, *bh = nullptr, *bl = nullptr;
    df cpr = {0.0f, 0.0f};
    float c5 = 0.0f;
    double h2 = 0, ih2 = 0, rho = 0;
    int co[3] = {0, 0, 0}, cnc = 0;
    const double *lam = nullptr;
};
struct PSetSrc {
    double *s[5];  // s0 s_x s_y s_z sigma, natural n^3
};
struct PSetFld {
    const double *g[10];  // ghosted fields, setup order V_x V_y V_z U psi apsi B^x B^y B^z b
};
void patch_deposit(int64_t np, const double *x, const double *u, double mass, double L, int N, const int O[3], int nw,
                   const PSetSrc &out, cudaStream_t st);
// indices of the particles in base cells [lo, lo + len) (mod n0) per axis -> list, their number -> count
void patch_select(int64_t np, const double *x, double L, int n0, const int lo[3], int len, int *list,
                  unsigned *count, cudaStream_t st);
// patch_deposit over the particles of such a list (np: the particle arrays' length)
void patch_deposit_list(int64_t np, const int *list, const unsigned *count, const double *x, const double *u,
                        double mass, double L, int N, const int O[3], int nw, const PSetSrc &out, cudaStream_t st);
// win = the parent's window; with dold, also dold := win - dold (and d32 its FP32 copy)
void patch_gather_base(int fmt, const PBase &B, const int o[3], int w, double *win, cudaStream_t st,
                       double *dold = nullptr, float *d32 = nullptr);
void patch_gather_patch(const PPatch &par, bool pdf, const int o[3], int w, double *win, cudaStream_t st,
                        double *dold = nullptr, float *d32 = nullptr);
// ghosts of the unknown = P(win); with d (or its FP32 copy d32 for pdf), the interior += P(d)
void patch_interp(const PPatch &P, bool pdf, const double *win, const double *d, const float *d32, cudaStream_t st);
void patch_gs(int kind, const PPatch &P, bool pdf, int color, cudaStream_t st);
void patch_resid(int kind, const PPatch &P, bool pdf, double *eps, const Sums &sums, cudaStream_t st);
void patch_restrict(const PPatch &P, bool pdf, const double *eps, double *Ru, double *Re, cudaStream_t st);
void patch_inject_u_base(int fmt, const PBase &B, const int o[3], int nc, const double *Ru, cudaStream_t st);
void patch_inject_f_base(int fmt, int kind, const PBase &B, const int o[3], int nc, const double *Re, const double *lam,
                        const Sums &sums, cudaStream_t st);
void patch_sum_f_base(int fmt, const PBase &B, const int o[3], int nc, const Sums &sums, cudaStream_t st);
void patch_inject_u_patch(const PPatch &par, bool pdf, const int o[3], int nc, const double *Ru, cudaStream_t st);
void patch_inject_f_patch(int kind, const PPatch &par, bool pdf, const int o[3], int nc, const double *Re,
                          cudaStream_t st);
void patch_reflux(int parent_fmt, const PBase &B, const PPatch &par, const PPatch &ch, bool pdf, const int o[3],
                  double hc, double *flux, cudaStream_t st);
void patch_lambda(double *sc, const double *flux, int nq, double N, double Ncov, double *lam, cudaStream_t st);
void sub_scalar(int64_t cnt, double *a, const double *m, cudaStream_t st);
void patch_to_ghosted(int n, const double *in, double *out, double add, cudaStream_t st);
void patch_u_load(const PPatch &P, bool pdf, const double *in, double add, cudaStream_t st);
void patch_u_store(const PPatch &P, bool pdf, double *out, double *keep, double add, const double *usum, double scale,
                   cudaStream_t st);
void patch_coef_df(int kind, const PPatch &P, cudaStream_t st);
// A_ij of the ghosted V, U on the interior and first ghost layer (six ghosted arrays)
void patch_aij(int n, double nh, const PSetFld &G, double *A6, cudaStream_t st);
void patch_setup(int eq, int n, double nh, const PSetSrc &S, const PSetFld &G, const double *A6, double smean,
                double K2, double Kdot, double *f, double *c0, double *c1, const Sums &sums, cudaStream_t st);

// Three FP32 colour passes of the correction equation (KPOISSON, KHELM) in
// one pass over memory: colour c1 from the other colour of ein, then the other
// colour, then c1 again; both colours of the result go to eout (smooth3.cu).
// inv: KHELM's 1/(6 + h^2 m).  rt: row tiles (smooth3_row_tiles).
bool smooth3_fits(int kind, int n);
int smooth3_row_tiles(int n, int sms);
void smooth3(int kind, int n, const float *ein, float *eout, const float *f, const float *inv, double h2, int c1,
             int rt, cudaStream_t st);

}  // namespace gr
