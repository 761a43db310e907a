// particle_kernels.cu - the particle update around the constraint solve (kick
// and drift in the solved metric) and the deposit with the metric's Lorentz
// factor.
//
// Geometric units, a = 1, c = 1: the metric is psi^4 delta_ij, the lapse
// alpha = (alpha psi) / psi and the shift beta^i = B^i + d_i b (Sec. 4.3.1).
// With the paper's code-unit potentials Phi = alpha - 1 and Psi = 2 (1 - psi)
// the kick splits the force of Sec. 4.4 (Eqs. force, coeff_j, coeff_4,
// coeff_5) into five substeps, each using the velocity the previous one left:
//     j = 1, 2, 3:  du_i += dt/2 (-u_j)(-D_i beta^j)
//     j = 4:        du_i += dt/2 (W^2 - 1)/W alpha/psi (2 D_i psi)
//     j = 5:        du_i += dt/2 W (-D_i alpha)
// with W = sqrt(1 + psi^-4 |u|^2) (Eq. Lorentz-factor) at the current
// velocity; the synchronising kick of the previous step runs j = 1..5 and the
// opening kick j = 5..1 (Sec. 4.4; App. A Eqs. GR-K1, GR-K2).  The drift
// moves x by dt (alpha psi^-4 u / W - beta) with the fields at the old
// position (App. A Eqs. GR-D, V_exp).
//
// Design.  Pass 1 forms alpha - 1 = (alpha psi - psi)/psi, psi - 1 and
// beta^j = B^j + D_j b per cell (the differences in FP64, the quotient and the
// stores in FP32: deviations keep their relative precision); pass 2 forms the
// 3-point central differences (the paper's gradient stencil) of those FP32
// arrays and stores, per cell, one 80-byte record of the 20 quantities
// (alpha - 1, psi - 1, beta^j, D_i alpha, D_i psi, D_i beta^j).  The
// cloud-in-cell gather of a particle reads eight records; five lanes read one
// record (16 bytes each), six particles at a time per warp, so that a load
// touches the few cache lines of six records instead of a line per lane.
// Each particle runs the substeps in FP32, accumulating its
// velocity change in FP32 and adding it to the FP64 velocity once;
// positions, the cell index and the cloud-in-cell fractions stay FP64 (a
// fraction loses nothing when rounded to FP32 afterwards).  GB300 issues
// FP64 at 1/58 of the FP32 rate, so this keeps the per-cell and per-particle
// work off the FP64 pipe, and so do conversions, cell indices and fractions
// made by integer operations.  Error: the gathered values carry a few 2^-24 of
// their own size; a central difference of FP32 deviations carries 2^-24 of
// the deviation over kh (the field's wavenumber times h), about 1e-6 of the
// gradient for grid-scale structure, far below the O(h^2) of the
// interpolation.
#include <cuda_runtime.h>

#include <cmath>

#include "../../include/gr.h"
#include "gr_internal.cuh"

namespace gr {

namespace {

// index of the 20 gathered quantities
enum : int { Q_ALPHA = 0, Q_PSI = 1, Q_BETA = 2, Q_DALPHA = 5, Q_DPSI = 8, Q_DBETA = 11, Q_N = 20 };

int log2i(int n)
{
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

// The FP64 forms of the helpers below, out of line: inlined, they would be
// predicated into the common path and occupy the FP64 pipe for every element.
static __device__ __noinline__ float to_float_fp64(double x) { return (float)x; }
static __device__ __noinline__ double to_double_fp64(float x) { return (double)x; }
static __device__ __noinline__ double wrap_fp64(double x, double L, double invL) { return fma(-L, floor(x * invL), x); }
struct Cloud {
    int lo;
    float w0, w1;
};
static __device__ __noinline__ Cloud cloud_fp64(double x, double invh)
{
    const double t = fma(x, invh, -0.5), fl = floor(t), fr = t - fl;
    return {(int)(long long)fl, (float)(1.0 - fr), (float)fr};
}

// (float)x by integer operations: the mantissa's 29 lowest bits rounded off to
// nearest even; results outside FP32's normal range take the conversion
__device__ __forceinline__ float to_float_rn(double x)
{
    // on the two 32-bit halves: a test of the 64 bits for zero would become an FP64 comparison
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if (((hi << 1) | lo) == 0u) return __uint_as_float(hi);  // +-0
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e - 897u > 252u) return to_float_fp64(x);
    // leading 23 stored bits, the 29 others rounded; a carry moves into the exponent
    const unsigned t = ((hi & 0x7fffffffu) - (896u << 20) << 3) | (lo >> 29);
    const unsigned rest = lo & 0x1fffffffu;
    return __uint_as_float((hi & 0x80000000u) | (t + (rest + (t & 1u) > 0x10000000u ? 1u : 0u)));
}

// (double)x by moving exponent and mantissa (normal x and zeros)
__device__ __forceinline__ double to_double(float x)
{
    const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    if (e - 1u > 253u) return (b << 1) == 0u ? __hiloint2double((int)b, 0) : to_double_fp64(x);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}

// four consecutive values of a natural-layout array, ALIGNED: on a 16-byte boundary
template <bool ALIGNED>
__device__ __forceinline__ void ld4d(const double *p, double (&v)[4])
{
    if (!ALIGNED) {
#pragma unroll
        for (int e = 0; e < 4; e++) v[e] = p[e];
        return;
    }
    const double2 a = *reinterpret_cast<const double2 *>(p), b = *reinterpret_cast<const double2 *>(p + 2);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}

// pass 1 (natural layout): d[0] = alpha - 1, d[1] = psi - 1,
// d[2 + j] = beta^j = B^j + D_j b, FP32 (n^3 each); four cells of a row per
// thread, FP64 issue bound (8 operations per cell: 2.1 ms at 512^3; 14 with
// the conversions on the FP64 pipe, 3.5 ms)
template <bool ALIGNED>
__global__ void __launch_bounds__(kBlock)
    k_pf_dev(int lgn, double inv2h, const double *__restrict__ psi, const double *__restrict__ apsi,
             const double *__restrict__ Bx, const double *__restrict__ By, const double *__restrict__ Bz,
             const double *__restrict__ b, float *__restrict__ d)
{
    pdl_begin();
    const int m = (1 << lgn) - 1;
    const int64_t N = (int64_t)1 << (3 * lgn);
    for (int64_t t4 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t4 < N / 4; t4 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = 4 * t4;
        const int k = (int)(t & m), j = (int)((t >> lgn) & m), i = (int)(t >> (2 * lgn));
        const int64_t row = t - k, plane = t - ((int64_t)j << lgn) - k;
        const int64_t ro = ((int64_t)j << lgn) + k;
        double ps[4], ap[4], xp[4], xm[4], yp[4], ym[4], z[4], f[4];
        ld4d<ALIGNED>(psi + t, ps);
        ld4d<ALIGNED>(apsi + t, ap);
        ld4d<ALIGNED>(b + ((int64_t)((i + 1) & m) << (2 * lgn)) + ro, xp);
        ld4d<ALIGNED>(b + ((int64_t)((i - 1) & m) << (2 * lgn)) + ro, xm);
        ld4d<ALIGNED>(b + plane + ((int64_t)((j + 1) & m) << lgn) + k, yp);
        ld4d<ALIGNED>(b + plane + ((int64_t)((j - 1) & m) << lgn) + k, ym);
        ld4d<ALIGNED>(b + t, z);
        const double zm = b[row + ((k - 1) & m)], zp = b[row + ((k + 4) & m)];
        float o[4];
#pragma unroll
        for (int e = 0; e < 4; e++) o[e] = to_float_rn(ap[e] - ps[e]) / to_float_rn(ps[e]);
        *reinterpret_cast<float4 *>(d + t) = make_float4(o[0], o[1], o[2], o[3]);
#pragma unroll
        for (int e = 0; e < 4; e++) o[e] = to_float_rn(ps[e] - 1.0);
        *reinterpret_cast<float4 *>(d + N + t) = make_float4(o[0], o[1], o[2], o[3]);
        ld4d<ALIGNED>(Bx + t, f);
#pragma unroll
        for (int e = 0; e < 4; e++) o[e] = to_float_rn(fma(xp[e] - xm[e], inv2h, f[e]));
        *reinterpret_cast<float4 *>(d + 2 * N + t) = make_float4(o[0], o[1], o[2], o[3]);
        ld4d<ALIGNED>(By + t, f);
#pragma unroll
        for (int e = 0; e < 4; e++) o[e] = to_float_rn(fma(yp[e] - ym[e], inv2h, f[e]));
        *reinterpret_cast<float4 *>(d + 3 * N + t) = make_float4(o[0], o[1], o[2], o[3]);
        ld4d<ALIGNED>(Bz + t, f);
#pragma unroll
        for (int e = 0; e < 4; e++)
            o[e] = to_float_rn(fma((e < 3 ? z[e < 3 ? e + 1 : 0] : zp) - (e > 0 ? z[e > 0 ? e - 1 : 0] : zm), inv2h, f[e]));
        *reinterpret_cast<float4 *>(d + 4 * N + t) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

// pass 2: the 80-byte record of every cell from the five FP32 arrays of pass 1.
// Four cells of a row per thread, each neighbour row one 16-byte load; the
// records of 64 cells at a time (5120 contiguous bytes) go through shared memory so
// that the stores are consecutive (a slot in forty is skipped, which spreads the
// lanes over the banks).  32-bit offsets: n <= 1024.  Memory bound: 100 bytes per
// cell, 3.2 ms at 512^3 (6.9 with one cell per thread and 35 scalar loads).
__global__ void __launch_bounds__(kBlock)
    k_pf_grad(int lgn, float inv2h, const float *__restrict__ d, float4 *__restrict__ rec)
{
    pdl_begin();
    __shared__ float4 stage[kBlock / 32][320 + 8];
    const int m = (1 << lgn) - 1;
    const int N = 1 << (3 * lgn);
    const int lane = threadIdx.x & 31;
    float4 *const st = stage[threadIdx.x >> 5];
    // whole warps step through the cells; on 4^3 the upper lanes repeat the last cells
    for (int base = 4 * (blockIdx.x * blockDim.x + (threadIdx.x & ~31)); base < N; base += 4 * gridDim.x * blockDim.x) {
        const int t = min(base + 4 * lane, N - 4);
        const int k = t & m, j = (t >> lgn) & m, i = t >> (2 * lgn);
        const int row = t - k, plane = t - (j << lgn) - k, ro = (j << lgn) + k;
        const int nx0 = (((i + 1) & m) << (2 * lgn)) + ro, nx1 = (((i - 1) & m) << (2 * lgn)) + ro;
        const int ny0 = plane + (((j + 1) & m) << lgn) + k, ny1 = plane + (((j - 1) & m) << lgn) + k;
        const int nz0 = row + ((k + 4) & m), nz1 = row + ((k - 1) & m);
        float q[4][Q_N];
#pragma unroll
        for (int v = 0; v < 5; v++) {  // alpha - 1, psi - 1, beta^x, beta^y, beta^z
            const float *f = d + (int64_t)v * N;
            const float4 c4 = *reinterpret_cast<const float4 *>(f + t);
            const float4 a4 = *reinterpret_cast<const float4 *>(f + nx0), b4 = *reinterpret_cast<const float4 *>(f + nx1);
            const float4 e4 = *reinterpret_cast<const float4 *>(f + ny0), g4 = *reinterpret_cast<const float4 *>(f + ny1);
            const float zp = f[nz0], zm = f[nz1];
            const float c[4] = {c4.x, c4.y, c4.z, c4.w};
            const float dx[4] = {a4.x - b4.x, a4.y - b4.y, a4.z - b4.z, a4.w - b4.w};
            const float dy[4] = {e4.x - g4.x, e4.y - g4.y, e4.z - g4.z, e4.w - g4.w};
            const float dz[4] = {c[1] - zm, c[2] - c[0], c[3] - c[1], zp - c[2]};
            const int o = v == 0 ? Q_DALPHA : (v == 1 ? Q_DPSI : Q_DBETA + 3 * (v - 2));
#pragma unroll
            for (int e = 0; e < 4; e++) {
                q[e][v] = c[e];
                q[e][o] = dx[e] * inv2h;
                q[e][o + 1] = dy[e] * inv2h;
                q[e][o + 2] = dz[e] * inv2h;
            }
        }
#pragma unroll
        for (int half = 0; half < 2; half++) {
            if ((lane >> 4) == half)
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const int c = 4 * (lane & 15) + e;
#pragma unroll
                    for (int v = 0; v < 5; v++)
                        st[5 * c + v + (c >> 3)] =
                            make_float4(q[e][4 * v], q[e][4 * v + 1], q[e][4 * v + 2], q[e][4 * v + 3]);
                }
            __syncwarp();
            float4 *const r = rec + 5 * (int64_t)(base + 64 * half);
            const int cnt = 5 * min(64, N - base - 64 * half);
#pragma unroll
            for (int v = 0; v < 10; v++) {
                const int o = 32 * v + lane;
                if (o < cnt) r[o] = st[o + o / 40];
            }
            __syncwarp();
        }
    }
}

// one substep j (1..5) of a kick by hdt = dt/2 in FP32; the velocity is
// u0 + du with the change du accumulated here; q holds alpha - 1 and psi - 1
__device__ __forceinline__ void substep(int j, float hdt, const float *q, const float u0[3], float du[3])
{
    const float ux = u0[0] + du[0], uy = u0[1] + du[1], uz = u0[2] + du[2];
    if (j <= 3) {
        const float c = -(j == 1 ? ux : (j == 2 ? uy : uz));  // c_j = -u_j
        const float *g = q + Q_DBETA + 3 * (j - 1);             // D_i beta^j, (f_j)_i = -D_i beta^j
        du[0] = fmaf(hdt * c, -g[0], du[0]);
        du[1] = fmaf(hdt * c, -g[1], du[1]);
        du[2] = fmaf(hdt * c, -g[2], du[2]);
        return;
    }
    const float ip = 1.0f / (1.0f + q[Q_PSI]);
    const float ip2 = ip * ip;
    const float g = ip2 * ip2 * fmaf(ux, ux, fmaf(uy, uy, uz * uz));  // psi^-4 |u|^2 = W^2 - 1
    const float W = sqrtf(1.0f + g);
    if (j == 4) {  // c_4 = (W^2 - 1)/W alpha/psi, (f_4)_i = 2 D_i psi
        const float c = g / W * (1.0f + q[Q_ALPHA]) * ip;
        du[0] = fmaf(hdt * c, 2.0f * q[Q_DPSI + 0], du[0]);
        du[1] = fmaf(hdt * c, 2.0f * q[Q_DPSI + 1], du[1]);
        du[2] = fmaf(hdt * c, 2.0f * q[Q_DPSI + 2], du[2]);
    } else {  // c_5 = W, (f_5)_i = -D_i alpha
        du[0] = fmaf(hdt * W, -q[Q_DALPHA + 0], du[0]);
        du[1] = fmaf(hdt * W, -q[Q_DALPHA + 1], du[1]);
        du[2] = fmaf(hdt * W, -q[Q_DALPHA + 2], du[2]);
    }
}

// f 2^-64 rounded to FP32 (to nearest even); one: f stands for 2^64
__device__ __forceinline__ float unit_fraction(unsigned long long f, bool one)
{
    if (one) return 1.0f;
    if (f == 0ull) return 0.0f;
    const int z = __clzll((long long)f);
    const unsigned long long n = f << z;  // leading bit at 63
    const unsigned r = (unsigned)((n + 0x7fffffffffull + ((n >> 40) & 1ull)) >> 40);  // 24 bits; zero on a carry out
    // r's leading bit adds one to the exponent
    return r ? __uint_as_float(((unsigned)(125 - z) << 23) + r) : __uint_as_float((unsigned)(127 - z) << 23);
}

// Cell and FP32 weights of coordinate x: t = x / h - 1/2, lo = floor(t), the
// fraction and one minus it rounded to FP32.  lgh >= 0: 1/h = 2^lgh, and the
// fraction of a t >= 0 is x's mantissa shifted (t and 1 - fraction are then
// exact in FP64 too, so the weights are the same); FP64 otherwise.
__device__ __forceinline__ Cloud cloud(double x, double invh, int lgh)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)(b >> 52) - 1023 + lgh;  // negative x: beyond 2^10
    if (lgh < 0 || ex < -1 || ex > 20) return cloud_fp64(x, invh);
    const unsigned long long mant = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const unsigned long long f = mant << (ex + 12);  // fraction of x / h in units of 2^-64
    const int c = ex < 0 ? 0 : (int)(mant >> (52 - ex));
    const unsigned long long fr = f - (1ull << 63);  // of t = x / h - 1/2
    return {c - (f < (1ull << 63) ? 1 : 0), unit_fraction(0ull - fr, fr == 0ull), unit_fraction(fr, false)};
}

// One thread per particle for positions, kicks and drift (blocks start in index
// order, so for lattice-ordered particles the cells in flight are a few planes
// that L2 holds); the gather in between is the warp's: lane 5 s + v reads
// quadruple v of the records around particle s of six, with that particle's cells and
// weights from shared memory, and leaves the interpolated quadruple there.
// top: below L by a relative 2^-40.  Latency and L1 bound (L1 75% busy, records of
// scattered particles; 4 blocks of 64 registers, 5 spill): 12.6 -> 10.4 ms for
// 134M particles.
__global__ void __launch_bounds__(kBlock, 4)
    k_particle_update(int lgn, double invh, int lgh, double L, double invL, double top, int64_t np,
                      double *__restrict__ x, double *__restrict__ u, const float4 *__restrict__ rec, float hdt, double dt,
                      int flags)
{
    pdl_begin();
    __shared__ float4 wt_s[2][kBlock];  // the eight weights, corners (a, b, c) at 4 a + 2 b + c
    __shared__ int4 xy_s[kBlock];       // the two cells' offsets along x and along y
    __shared__ int2 z_s[kBlock];        // and along z
    __shared__ float4 q_s[kBlock * 5];
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool ok = p < np;
    const int m = (1 << lgn) - 1;
    double xd[3] = {0.0, 0.0, 0.0};
    {
        Cloud cl[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (ok) xd[d] = x[d * np + p];
            cl[d] = cloud(xd[d], invh, lgh);
        }
        float w[8];
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int b = 0; b < 2; b++) {
                const float wab = (a ? cl[0].w1 : cl[0].w0) * (b ? cl[1].w1 : cl[1].w0);
                w[4 * a + 2 * b] = wab * cl[2].w0;
                w[4 * a + 2 * b + 1] = wab * cl[2].w1;
            }
        wt_s[0][threadIdx.x] = make_float4(w[0], w[1], w[2], w[3]);
        wt_s[1][threadIdx.x] = make_float4(w[4], w[5], w[6], w[7]);
        xy_s[threadIdx.x] = make_int4((cl[0].lo & m) << (2 * lgn), ((cl[0].lo + 1) & m) << (2 * lgn), (cl[1].lo & m) << lgn,
                                      ((cl[1].lo + 1) & m) << lgn);
        z_s[threadIdx.x] = make_int2(cl[2].lo & m, (cl[2].lo + 1) & m);
    }
    __syncwarp();
    {
        const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
        const int s6 = lane / 5, v = lane - 5 * s6;
        const int live = (int)min((int64_t)32, np - (p - lane));  // particles of this warp (may be none)
        for (int r = 0; r < live; r += 6) {
            const int s = r + s6;
            if (s6 < 6 && s < live) {
                const int t = w0 + s;
                const int4 xy = xy_s[t];
                const int2 z = z_s[t];
                const int row[4] = {xy.x + xy.z, xy.x + xy.w, xy.y + xy.z, xy.y + xy.w};
                float4 g[8];
#pragma unroll
                for (int ab = 0; ab < 4; ab++) {
                    g[2 * ab] = __ldg(rec + 5 * (int64_t)(row[ab] + z.x) + v);
                    g[2 * ab + 1] = __ldg(rec + 5 * (int64_t)(row[ab] + z.y) + v);
                }
                const float4 wa = wt_s[0][t], wb = wt_s[1][t];
                const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
                float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    q.x = fmaf(w[c], g[c].x, q.x);
                    q.y = fmaf(w[c], g[c].y, q.y);
                    q.z = fmaf(w[c], g[c].z, q.z);
                    q.w = fmaf(w[c], g[c].w, q.w);
                }
                q_s[5 * t + v] = q;
            }
        }
    }
    __syncwarp();
    if (!ok) return;
    float q[Q_N];
#pragma unroll
    for (int v = 0; v < 5; v++) {
        const float4 g = q_s[5 * threadIdx.x + v];
        q[4 * v] = g.x;
        q[4 * v + 1] = g.y;
        q[4 * v + 2] = g.z;
        q[4 * v + 3] = g.w;
    }
    const double ud[3] = {u[p], u[np + p], u[2 * np + p]};
    const float u0[3] = {to_float_rn(ud[0]), to_float_rn(ud[1]), to_float_rn(ud[2])};
    float du[3] = {0.0f, 0.0f, 0.0f};
    if (flags & GR_KICK_SYNC)
#pragma unroll
        for (int j = 1; j <= 5; j++) substep(j, hdt, q, u0, du);
    if (flags & GR_KICK_OPEN)
#pragma unroll
        for (int j = 5; j >= 1; j--) substep(j, hdt, q, u0, du);
    if (flags & (GR_KICK_SYNC | GR_KICK_OPEN))
#pragma unroll
        for (int d = 0; d < 3; d++) u[d * np + p] = ud[d] + to_double(du[d]);
    if (flags & GR_DRIFT) {
        const float ux = u0[0] + du[0], uy = u0[1] + du[1], uz = u0[2] + du[2];
        const float ip = 1.0f / (1.0f + q[Q_PSI]);
        const float ip4 = (ip * ip) * (ip * ip);
        const float W = sqrtf(1.0f + ip4 * fmaf(ux, ux, fmaf(uy, uy, uz * uz)));
        const float fac = (1.0f + q[Q_ALPHA]) * ip4 / W;
        const float v[3] = {fmaf(fac, ux, -q[Q_BETA + 0]), fmaf(fac, uy, -q[Q_BETA + 1]),
                            fmaf(fac, uz, -q[Q_BETA + 2])};
#pragma unroll
        for (int d = 0; d < 3; d++) {
            // back into [0, L) (x - L floor(x / L); for L = 1 exactly x - floor(x))
            double xn = fma(dt, to_double(v[d]), xd[d]);
            // inside the box and not within rounding of L: floor(xn / L) = 0 (compared as integers)
            if ((unsigned long long)__double_as_longlong(xn) >= (unsigned long long)__double_as_longlong(top))
                xn = wrap_fp64(xn, L, invL);
            x[d * np + p] = xn;
        }
    }
}

// Deposit with the Lorentz factor at psi: W = sqrt(1 + psi^-4 |u|^2), psi
// at the particle by cloud-in-cell in FP64.  Charges as k_deposit:
// s0 += q W w, s_l += q u_l w, sigma += q |u|^2 / W w, the forty products
// charge x weight as double-float products (relative error about 2^-46)
// joined for the FP64 atomic adds, as in the plain deposit.
__global__ void __launch_bounds__(kBlock)
    k_deposit_metric(int lgn, double invh, int64_t np, const double *__restrict__ x, const double *__restrict__ u,
                     double q, const double *__restrict__ psi, double *__restrict__ s0, double *__restrict__ sx,
                     double *__restrict__ sy, double *__restrict__ sz, double *__restrict__ sig)
{
    pdl_begin();
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= np) return;
    const int m = (1 << lgn) - 1;
    int lo[3];
    double fw[3][2];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const double t = fma(x[d * np + p], invh, -0.5);
        const double fl = floor(t);
        const double fr = t - fl;
        fw[d][0] = 1.0 - fr;
        fw[d][1] = fr;
        lo[d] = (int)((long long)fl & m);
    }
    double ps = 0.0;
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int b = 0; b < 2; b++) {
            const double wab = fw[0][a] * fw[1][b];
            const int64_t row = ((int64_t)((((lo[0] + a) & m) << lgn) + ((lo[1] + b) & m))) << lgn;
#pragma unroll
            for (int c = 0; c < 2; c++) ps = fma(wab * fw[2][c], __ldg(psi + row + ((lo[2] + c) & m)), ps);
        }
    const double ip2 = 1.0 / (ps * ps);
    const double ux = u[p], uy = u[np + p], uz = u[2 * np + p];
    const double u2 = fma(ux, ux, fma(uy, uy, uz * uz));
    const double w2 = fma(ip2 * ip2, u2, 1.0);
    const double rw = rsqrt(w2);
    const df Q[5] = {split_double(q * (w2 * rw)), split_double(q * ux), split_double(q * uy), split_double(q * uz),
                     split_double((q * u2) * rw)};
    double *const out[5] = {s0, sx, sy, sz, sig};
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int b = 0; b < 2; b++) {
            const double wab = fw[0][a] * fw[1][b];
            const int64_t row = ((int64_t)((((lo[0] + a) & m) << lgn) + ((lo[1] + b) & m))) << lgn;
#pragma unroll
            for (int c = 0; c < 2; c++) {
                const df w = split_double(wab * fw[2][c]);
                const int64_t id = row + ((lo[2] + c) & m);
#pragma unroll
                for (int k = 0; k < 5; k++) atomicAdd(out[k] + id, join_double(df_mul(Q[k], w)));
            }
        }
}

}  // namespace

void particle_fields(int n, double L, const double *psi, const double *apsi, const double *Bx, const double *By,
                     const double *Bz, const double *b, float *dev, float *rec, cudaStream_t st)
{
    const int lgn = log2i(n);
    const int64_t N = (int64_t)n * n * n;
    const double inv2h = 0.5 * n / L;
    // the caller's fields need not lie on 16-byte boundaries here
    const double *f[6] = {psi, apsi, Bx, By, Bz, b};
    bool aligned = true;
    for (int k = 0; k < 6; k++) aligned = aligned && ((uintptr_t)f[k] & 15u) == 0;
    if (aligned)
        GR_LAUNCH(k_pf_dev<true>, wave_grid(k_pf_dev<true>, N / 4), kBlock, st, lgn, inv2h, psi, apsi, Bx, By, Bz, b, dev);
    else
        GR_LAUNCH(k_pf_dev<false>, wave_grid(k_pf_dev<false>, N / 4), kBlock, st, lgn, inv2h, psi, apsi, Bx, By, Bz, b,
                  dev);
    GR_LAUNCH(k_pf_grad, wave_grid(k_pf_grad, N / 4), kBlock, st, lgn, (float)inv2h, (const float *)dev, (float4 *)rec);
}

void particle_update(int n, double L, int64_t np, double *x, double *u, const float *rec, double dt, int flags,
                     cudaStream_t st)
{
    if (np <= 0) return;
    const int64_t blocks = (np + kBlock - 1) / kBlock;
    const int g = (int)(blocks < 0x7fffffff ? blocks : 0x7fffffff);
    const double invh = (double)n / L;
    int hx;
    const int lgh = std::frexp(invh, &hx) == 0.5 && hx >= 1 && hx < 1000 ? hx - 1 : -1;
    GR_LAUNCH(k_particle_update, g, kBlock, st, log2i(n), invh, lgh, L, 1.0 / L, L * (1.0 - 0x1p-40), np, x, u,
              (const float4 *)rec, (float)(0.5 * dt), dt, flags);
}

void deposit_metric_add(int n, double L, int64_t np, const double *x, const double *u, double mass, const double *psi,
                        double *s0, double *sx, double *sy, double *sz, double *sig, cudaStream_t st)
{
    if (np <= 0) return;
    const double h = L / n;
    const int64_t blocks = (np + kBlock - 1) / kBlock;
    const int g = (int)(blocks < 0x7fffffff ? blocks : 0x7fffffff);
    GR_LAUNCH(k_deposit_metric, g, kBlock, st, log2i(n), 1.0 / h, np, x, u, mass / (h * h * h), psi, s0, sx, sy, sz,
              sig);
}

}  // namespace gr
