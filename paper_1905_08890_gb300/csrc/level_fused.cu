// level_fused.cu - one level's whole smoothing in one launch per direction, for
// the FP32 correction cycle's levels 32^3 and 64^3 with nu = 2.
//
// Such a level holds 0.1 to 1 MB per array, so its passes run from L2 and cost
// their latency, not bandwidth: measured back to back, a colour pass takes 1.5
// us at 32^3 and 1.6 us at 64^3, of which 1.4 us is the launch itself.  Here a block
// owns a tile of TI x TJ full rows (k whole, so the periodic wrap along k
// stays inside the row) and recomputes what its neighbours' passes would give
// it: its region is the tile with four rows more on every side, and each pass is valid
// on one row less than the one before.  Going down (k_level_down): [first red
// from the right-hand side,] black, red, black, red residual, restriction.
// Going up (k_level_up): prolongation onto the black cells, red, black, red,
// black[, u += e].  Both colours of the region live in shared memory, the
// right-hand sides of all passes in registers, fetched at the start.  Every
// cell's arithmetic is that of the separate kernels (k_sweep4, k_restrict_red2,
// k_prolong_black4), bit for bit.
//
// Tiles: the grid should fill the SMs once and the redundant rows stay few:
// 32^3 takes 4 x 4 rows (64 blocks, 18 KB), 64^3 4 x 8 (128 blocks, 49 KB).
// Measured, down + up back to back: 32^3 6.3 us against 15.5 in ten launches,
// 64^3 8.4 against 16; a 128^3 double-float solve 12.83 -> 11.05 ms.  128^3
// stays on separate launches: its tile of 8 x 16 rows (192 KB) took 12.3 + 20.9 us
// against 12.2 + 19.5 (a pass there is 3 us of L2 bandwidth, and the redundant
// rows cost more of it than the launches saved).
#include "df64.cuh"
#include "df_stencil.cuh"
#include "gr_internal.cuh"

namespace gr {
namespace {

constexpr int kHalo = 4;

template <int LGN_, int TI_, int TJ_, int T_>
struct Tile {
    static constexpr int LGN = LGN_, TI = TI_, TJ = TJ_, T = T_;
    static constexpr int N = 1 << LGN, HN = N / 2, Q4 = HN / 4;  // half-indices and float4 per row and colour
    static constexpr int RI = TI + 2 * kHalo, RJ = TJ + 2 * kHalo;
    static constexpr int HALF = N * N * HN;
    static constexpr int SMEM = 2 * RI * RJ * HN * (int)sizeof(float);
    static constexpr int BLOCKS = (N / TI) * (N / TJ);
    static_assert(TI % 2 == 0 && TJ % 2 == 0 && RI <= N && RJ <= N && T % 32 == 0, "tile");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};
using Tile32 = Tile<5, 4, 4, 512>;
using Tile64 = Tile<6, 4, 8, 512>;

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }

// Sum of the six neighbours, all of the other colour, of four consecutive
// half-indices 4 m .. 4 m + 3 of region row rr; p: the cells' k parity, whose
// shifted own-row neighbour comes from the next or previous lane (the Q4
// lanes of a row are consecutive); E returns the own row's four values.
// Every lane of the warp calls it.
template <class C>
__device__ __forceinline__ float4 nbsum4(const float *oth, int rr, int m, int p, float4 &E)
{
    const float *o = oth + rr * C::HN + 4 * m;
    const float4 A = ld4(o + C::RJ * C::HN), B = ld4(o - C::RJ * C::HN), Cc = ld4(o + C::HN), D = ld4(o - C::HN);
    E = ld4(o);
    const float x = __shfl_sync(0xffffffffu, p ? E.x : E.w, p ? m + 1 : m - 1 + C::Q4, C::Q4);
    const float4 S = p ? make_float4(E.y, E.z, E.w, x) : make_float4(x, E.x, E.y, E.z);
    return make_float4(A.x + B.x + Cc.x + D.x + E.x + S.x, A.y + B.y + Cc.y + D.y + E.y + S.y,
                       A.z + B.z + Cc.z + D.z + E.z + S.z, A.w + B.w + Cc.w + D.w + E.w + S.w);
}

template <int KIND>
__device__ __forceinline__ float4 relax4(float4 nb, float4 F, float4 G, float h2)
{
    const float s6 = 1.0f / 6.0f;
    if (KIND == KPOISSON) G = make_float4(s6, s6, s6, s6);
    return make_float4(__fmaf_rn(-h2, F.x, nb.x) * G.x, __fmaf_rn(-h2, F.y, nb.y) * G.y,
                       __fmaf_rn(-h2, F.z, nb.z) * G.z, __fmaf_rn(-h2, F.w, nb.w) * G.w);
}

// item t of the region's rows shrunk by S on every side -> region row, float4 index and row offset in a half-array
template <class C, int S>
__device__ __forceinline__ bool item(int t, int i0, int j0, int &rr, int &m, int &p, int &off)
{
    constexpr int W = C::RJ - 2 * S, CNT = (C::RI - 2 * S) * W * C::Q4;
    const bool ok = t < CNT;
    if (!ok) t = CNT - C::Q4 + (t & (C::Q4 - 1));  // the last row again: lanes stay in step
    m = t & (C::Q4 - 1);
    const int row = t / C::Q4, a = row / W, ri = a + S, rj = row - a * W + S;
    rr = ri * C::RJ + rj;
    p = (ri + rj) & 1;  // tile origins and the halo are even
    const int gi = (i0 + ri - kHalo) & (C::N - 1), gj = (j0 + rj - kHalo) & (C::N - 1);
    off = ((gi << C::LGN) + gj) * C::HN + 4 * m;
    return ok;
}

// The right-hand sides (and inverse diagonals) of one colour pass on the
// region shrunk by S, in registers.  A kernel fetches those of all its passes
// at its start: a pass takes some 300 cycles and a fetch from L2 twice that, so
// a fetch between two passes would be most of the time.
template <class C, int KIND, int COL, int S>
struct Rhs {
    static constexpr int CNT = (C::RI - 2 * S) * (C::RJ - 2 * S) * C::Q4;
    static constexpr int NIT = (CNT + C::T - 1) / C::T;
    float4 F[NIT], G[KIND == KHELM ? NIT : 1];
    __device__ __forceinline__ void load(const float *__restrict__ r, const float *__restrict__ inv, int i0, int j0)
    {
#pragma unroll
        for (int s = 0; s < NIT; s++) {
            int rr, m, p, off;
            item<C, S>(s * C::T + (int)threadIdx.x, i0, j0, rr, m, p, off);
            F[s] = ld4(r + COL * C::HALF + off);
            if (KIND == KHELM) G[s] = ld4(inv + COL * C::HALF + off);
        }
    }
    // one pass: own from oth; begins with the barrier that ends the pass before
    __device__ __forceinline__ void relax(float *own, const float *oth, float h2, int i0, int j0) const
    {
        __syncthreads();
#pragma unroll
        for (int s = 0; s < NIT; s++) {
            int rr, m, p, off;
            const bool ok = item<C, S>(s * C::T + (int)threadIdx.x, i0, j0, rr, m, p, off);
            float4 E;
            const float4 nb = nbsum4<C>(oth, rr, m, p ^ COL, E);
            const float4 v = relax4<KIND>(nb, F[s], G[KIND == KHELM ? s : 0], h2);
            if (ok) st4(own + rr * C::HN + 4 * m, v);
        }
    }
};

// FROM_R: the first red pass from e = 0 is -h^2 r / 6 (-h^2 r / (6 + h^2 m));
// otherwise e holds the red values.  eb: the black half after the last pass.
// ec (may be null): the coarse correction's start, its first red pass from
// zero when h2c > 0, else zeros.
template <class C, int KIND, bool FROM_R>
__global__ void __launch_bounds__(C::T)
    k_level_down(const float *__restrict__ e, float *__restrict__ eb, const float *__restrict__ r,
                 const float *__restrict__ m_, const float *__restrict__ inv, float h2, float ih2,
                 float *__restrict__ ec, float *__restrict__ rc, const float *__restrict__ cinv, float h2c)
{
    pdl_begin();
    extern __shared__ float sh[];
    float *red = sh, *blk = sh + C::RI * C::RJ * C::HN;
    const int i0 = ((int)blockIdx.x / (C::N / C::TJ)) * C::TI, j0 = ((int)blockIdx.x % (C::N / C::TJ)) * C::TJ;
    constexpr int CNT = C::RI * C::RJ * C::Q4;
    Rhs<C, KIND, 1, 1> b1;
    Rhs<C, KIND, 0, 2> r2;
    Rhs<C, KIND, 1, 3> b3;
    b1.load(r, inv, i0, j0);
    r2.load(r, inv, i0, j0);
    b3.load(r, inv, i0, j0);
#pragma unroll
    for (int t = threadIdx.x; t < CNT; t += C::T) {
        int rr, m, p, off;
        item<C, 0>(t, i0, j0, rr, m, p, off);
        float4 v;
        if (FROM_R) {
            const float4 G = KIND == KHELM ? ld4(inv + off) : make_float4(0, 0, 0, 0);
            v = relax4<KIND>(make_float4(0, 0, 0, 0), ld4(r + off), G, h2);
        } else {
            v = ld4(e + off);
        }
        st4(red + rr * C::HN + 4 * m, v);
    }
    // red residual of the tile's rows; the four rows of a coarse row sit in one
    // warp, W lanes each, and are summed by shuffles
    constexpr int W = C::Q4 < 8 ? C::Q4 : 8, LC = C::LGN - 1, HC = C::HALF / 8;
    constexpr int RCNT = C::TI * C::TJ * C::Q4, RIT = (RCNT + C::T - 1) / C::T;
    static_assert(RCNT % 32 == 0 && 4 * W <= 32 && (C::T % (4 * W)) == 0, "restriction lanes");
    float4 F[RIT], M[RIT];
    int rrs[RIT], ms[RIT];
#pragma unroll
    for (int s = 0; s < RIT; s++) {
        int t = s * C::T + (int)threadIdx.x;
        if (t >= RCNT) t &= 31;  // whole warps: their results are dropped
        const int ml = t % W, ab = (t / W) & 3, g = t / (4 * W);
        const int mh = g % (C::Q4 / W), cr = g / (C::Q4 / W);
        const int ri = kHalo + 2 * (cr / (C::TJ / 2)) + (ab >> 1), rj = kHalo + 2 * (cr % (C::TJ / 2)) + (ab & 1);
        rrs[s] = ri * C::RJ + rj;
        ms[s] = mh * W + ml;
        const int off = (((i0 + ri - kHalo) << C::LGN) + j0 + rj - kHalo) * C::HN + 4 * ms[s];
        F[s] = ld4(r + off);
        M[s] = KIND == KHELM ? ld4(m_ + off) : make_float4(0, 0, 0, 0);
    }
    b1.relax(blk, red, h2, i0, j0);
    r2.relax(red, blk, h2, i0, j0);
    b3.relax(blk, red, h2, i0, j0);
    __syncthreads();
#pragma unroll
    for (int s = 0; s < RIT; s++) {
        const int t = s * C::T + (int)threadIdx.x;
        const bool ok = t < RCNT;
        const int rr = rrs[s], m = ms[s], ri = rr / C::RJ, rj = rr - ri * C::RJ;
        const float *bo = blk + rr * C::HN + 4 * m;
        float4 E;
        // the Q4 lanes of a row are not consecutive here when Q4 > W: the shifted neighbour from shared memory
        const float4 A = ld4(bo + C::RJ * C::HN), B = ld4(bo - C::RJ * C::HN), Cc = ld4(bo + C::HN), D = ld4(bo - C::HN);
        E = ld4(bo);
        const int p = (ri + rj) & 1;
        const float x = blk[rr * C::HN + ((4 * m + (p ? 4 : C::HN - 1)) & (C::HN - 1))];
        const float4 S = p ? make_float4(E.y, E.z, E.w, x) : make_float4(x, E.x, E.y, E.z);
        const float4 u = ld4(red + rr * C::HN + 4 * m);
        const float4 km = p ? E : S, kp = p ? S : E;  // k - 1, k + 1
        auto res = [&](float ia, float ib, float ja, float jb, float ka, float kb, float uc, float mm, float rv) {
            const float nb = ia + ib + ja + jb + ka + kb;
            float lap = (nb - 6.0f * uc) * ih2;
            if (KIND == KHELM) lap -= mm * uc;
            return lap - rv;
        };
        const float4 v = make_float4(res(B.x, A.x, D.x, Cc.x, km.x, kp.x, u.x, M[s].x, F[s].x),
                                     res(B.y, A.y, D.y, Cc.y, km.y, kp.y, u.y, M[s].y, F[s].y),
                                     res(B.z, A.z, D.z, Cc.z, km.z, kp.z, u.z, M[s].z, F[s].z),
                                     res(B.w, A.w, D.w, Cc.w, km.w, kp.w, u.w, M[s].w, F[s].w));
        const int gi = i0 + ri - kHalo, gj = j0 + rj - kHalo;
        if (ok) st4(eb + ((gi << C::LGN) + gj) * C::HN + 4 * m, E);
        float4 q = v;  // rows (0, 0), (0, 1), (1, 0), (1, 1) in this order
#pragma unroll
        for (int o = 1; o < 4; o++) {
            q.x += __shfl_down_sync(0xffffffffu, v.x, o * W);
            q.y += __shfl_down_sync(0xffffffffu, v.y, o * W);
            q.z += __shfl_down_sync(0xffffffffu, v.z, o * W);
            q.w += __shfl_down_sync(0xffffffffu, v.w, o * W);
        }
        if (ok && ((t / W) & 3) == 0) {
            const int I = gi >> 1, J = gj >> 1, c0 = (I + J) & 1;  // colour of the even coarse K
            const int base = (((I << LC) + J) << (LC - 1)) + 2 * m;
            const float2 ev = make_float2(-(0.125f * q.x), -(0.125f * q.z)), od = make_float2(-(0.125f * q.y), -(0.125f * q.w));
            *reinterpret_cast<float2 *>(rc + (c0 ? HC : 0) + base) = ev;
            *reinterpret_cast<float2 *>(rc + (c0 ? 0 : HC) + base) = od;
            if (ec) {
                float2 rv = c0 ? od : ev;  // the red ones
                float2 g = make_float2(1.0f / 6.0f, 1.0f / 6.0f);
                if (KIND == KHELM && h2c > 0.0f) g = *reinterpret_cast<const float2 *>(cinv + base);
                *reinterpret_cast<float2 *>(ec + base) = make_float2(-h2c * rv.x * g.x, -h2c * rv.y * g.y);
                *reinterpret_cast<float2 *>(ec + HC + base) = make_float2(0.0f, 0.0f);
            }
        }
    }
}

// 3/4 own + 1/4 neighbour, summed from the lower to the upper of the two as k_prolong_black4 does
__device__ __forceinline__ float4 lerp4(float4 own, float4 nbr, int upper)
{
    const float w0 = 0.25f, w1 = 0.75f;
    if (upper)
        return make_float4(w1 * own.x + w0 * nbr.x, w1 * own.y + w0 * nbr.y, w1 * own.z + w0 * nbr.z,
                           w1 * own.w + w0 * nbr.w);
    return make_float4(w0 * nbr.x + w1 * own.x, w0 * nbr.y + w1 * own.y, w0 * nbr.z + w1 * own.z,
                       w0 * nbr.w + w1 * own.w);
}

// UPDATE: the result is added to the double-float unknown (uh, ul) instead of
// being written to e.
template <class C, int KIND, bool UPDATE>
__global__ void __launch_bounds__(C::T)
    k_level_up(float *__restrict__ e, const float *__restrict__ eb, const float *__restrict__ r,
               const float *__restrict__ inv, const float *__restrict__ ec, float h2, float *__restrict__ uh,
               float *__restrict__ ul)
{
    pdl_begin();
    extern __shared__ float sh[];
    float *red = sh, *blk = sh + C::RI * C::RJ * C::HN;
    const int i0 = ((int)blockIdx.x / (C::N / C::TJ)) * C::TI, j0 = ((int)blockIdx.x % (C::N / C::TJ)) * C::TJ;
    constexpr int CNT = C::RI * C::RJ * C::Q4;
    constexpr int LC = C::LGN - 1, NC = C::N / 2, HC = C::HALF / 8, HNC = NC / 2;
    const float w0 = 0.25f, w1 = 0.75f;
    Rhs<C, KIND, 0, 1> r1;
    Rhs<C, KIND, 1, 2> b2;
    Rhs<C, KIND, 0, 3> r3;
    Rhs<C, KIND, 1, kHalo> b4;
    r1.load(r, inv, i0, j0);
    b2.load(r, inv, i0, j0);
    r3.load(r, inv, i0, j0);
    b4.load(r, inv, i0, j0);
#pragma unroll
    for (int t = threadIdx.x; t < CNT; t += C::T) {
        int rr, m, p, off;
        item<C, 0>(t, i0, j0, rr, m, p, off);
        const int row = off / C::HN, gi = row >> C::LGN, gj = row & (C::N - 1);
        const float4 old = ld4(eb + off);
        const int I[2] = {gi >> 1, ((gi >> 1) + ((gi & 1) ? 1 : -1)) & (NC - 1)};
        const int J[2] = {gj >> 1, ((gj >> 1) + ((gj & 1) ? 1 : -1)) & (NC - 1)};
        const int pb = p ^ 1;  // k parity of the black cells: the fine cell 2K + pb interpolates K and K - 1 or K + 1
        float4 y[2];
#pragma unroll
        for (int a = 0; a < 2; a++) {
            float4 z[2];
#pragma unroll
            for (int b = 0; b < 2; b++) {
                const int base = ((I[a] << LC) + J[b]) * HNC;
                const int ce = ((I[a] + J[b]) & 1) ? HC : 0, co = HC - ce;
                const float2 ev = *reinterpret_cast<const float2 *>(ec + ce + base + 2 * m);  // K = 4m, 4m + 2
                const float2 od = *reinterpret_cast<const float2 *>(ec + co + base + 2 * m);  // K = 4m + 1, 4m + 3
                const float x = pb ? ec[ce + base + ((2 * m + 2) & (HNC - 1))] : ec[co + base + ((2 * m - 1) & (HNC - 1))];
                z[b] = pb ? make_float4(w1 * ev.x + w0 * od.x, w1 * od.x + w0 * ev.y, w1 * ev.y + w0 * od.y, w1 * od.y + w0 * x)
                          : make_float4(w1 * ev.x + w0 * x, w1 * od.x + w0 * ev.x, w1 * ev.y + w0 * od.x, w1 * od.y + w0 * ev.y);
            }
            y[a] = lerp4(z[0], z[1], gj & 1);
        }
        const float4 v = lerp4(y[0], y[1], gi & 1);
        st4(blk + rr * C::HN + 4 * m, make_float4(old.x + v.x, old.y + v.y, old.z + v.z, old.w + v.w));
    }
    r1.relax(red, blk, h2, i0, j0);
    b2.relax(blk, red, h2, i0, j0);
    r3.relax(red, blk, h2, i0, j0);
    // the last black pass, on the tile itself, straight to memory with the red values
    constexpr int LIT = Rhs<C, KIND, 1, kHalo>::NIT;
    __syncthreads();
#pragma unroll
    for (int s = 0; s < LIT; s++) {
        int rr, m, p, off;
        const bool ok = item<C, kHalo>(s * C::T + (int)threadIdx.x, i0, j0, rr, m, p, off);
        float4 E;
        const float4 nb = nbsum4<C>(red, rr, m, p ^ 1, E);
        const float4 v = relax4<KIND>(nb, b4.F[s], b4.G[KIND == KHELM ? s : 0], h2);
        if (!ok) continue;
        if (!UPDATE) {
            st4(e + off, E);
            st4(e + C::HALF + off, v);
            continue;
        }
#pragma unroll
        for (int c = 0; c < 2; c++) {
            float *H = uh + c * C::HALF + off, *L = ul + c * C::HALF + off;
            const float4 h4 = ld4(H), l4 = ld4(L), d = c ? v : E;
            const df s0 = df_plus_f(h4.x, l4.x, d.x), s1 = df_plus_f(h4.y, l4.y, d.y), s2 = df_plus_f(h4.z, l4.z, d.z),
                     s3 = df_plus_f(h4.w, l4.w, d.w);
            st4(H, make_float4(s0.hi, s1.hi, s2.hi, s3.hi));
            st4(L, make_float4(s0.lo, s1.lo, s2.lo, s3.lo));
        }
    }
}

// the shared-memory opt-in, once per kernel and device.  The carve-out is held to one
// block per SM: left to itself the driver makes room for as many blocks as the
// SM could take, and the kernels that follow (which state no preference) then
// run with what L1 is left, 10% slower over a 512^3 solve.
template <class C, class Kernel>
bool opt_in(Kernel k)
{
    const int pct = ((C::SMEM + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024);
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) == cudaSuccess &&
           cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct) == cudaSuccess;
}

template <class C, int KIND, bool FROM_R>
void down_t(const float *e, float *eb, const float *r, const float *m, const float *inv, double h2, double ih2, float *ec,
            float *rc, const float *cinv, double h2c, cudaStream_t st)
{
    per_device([] { return opt_in<C>(k_level_down<C, KIND, FROM_R>); });
    GR_LAUNCH_SMEM((k_level_down<C, KIND, FROM_R>), C::BLOCKS, C::T, C::SMEM, st, e, eb, r, m, inv, (float)h2, (float)ih2,
                   ec, rc, cinv, (float)h2c);
}

template <class C, int KIND, bool UPDATE>
void up_t(float *e, const float *eb, const float *r, const float *inv, const float *ec, double h2, float *uh, float *ul,
          cudaStream_t st)
{
    per_device([] { return opt_in<C>(k_level_up<C, KIND, UPDATE>); });
    GR_LAUNCH_SMEM((k_level_up<C, KIND, UPDATE>), C::BLOCKS, C::T, C::SMEM, st, e, eb, r, inv, ec, (float)h2, uh, ul);
}

template <class C>
void down_c(int kind, bool from_r, const float *e, float *eb, const float *r, const float *m, const float *inv, double h2,
            double ih2, float *ec, float *rc, const float *cinv, double h2c, cudaStream_t st)
{
    if (kind == KPOISSON) {
        if (from_r) down_t<C, KPOISSON, true>(e, eb, r, m, inv, h2, ih2, ec, rc, cinv, h2c, st);
        else down_t<C, KPOISSON, false>(e, eb, r, m, inv, h2, ih2, ec, rc, cinv, h2c, st);
    } else {
        if (from_r) down_t<C, KHELM, true>(e, eb, r, m, inv, h2, ih2, ec, rc, cinv, h2c, st);
        else down_t<C, KHELM, false>(e, eb, r, m, inv, h2, ih2, ec, rc, cinv, h2c, st);
    }
}

template <class C>
void up_c(int kind, float *e, const float *eb, const float *r, const float *inv, const float *ec, double h2, float *uh,
          float *ul, cudaStream_t st)
{
    if (kind == KPOISSON) {
        if (uh) up_t<C, KPOISSON, true>(e, eb, r, inv, ec, h2, uh, ul, st);
        else up_t<C, KPOISSON, false>(e, eb, r, inv, ec, h2, uh, ul, st);
    } else {
        if (uh) up_t<C, KHELM, true>(e, eb, r, inv, ec, h2, uh, ul, st);
        else up_t<C, KHELM, false>(e, eb, r, inv, ec, h2, uh, ul, st);
    }
}

}  // namespace

bool level_fused_fits(int kind, int n, int nu1, int nu2)
{
    return (kind == KPOISSON || kind == KHELM) && (n == 32 || n == 64) && nu1 == 2 && nu2 == 2;
}

void level_down(int kind, int n, bool from_r, const float *e, float *eb, const float *r, const float *m,
                const float *inv, double h2, double ih2, float *ec, float *rc, const float *cinv, double h2c,
                cudaStream_t st)
{
    if (n == 32) down_c<Tile32>(kind, from_r, e, eb, r, m, inv, h2, ih2, ec, rc, cinv, h2c, st);
    else down_c<Tile64>(kind, from_r, e, eb, r, m, inv, h2, ih2, ec, rc, cinv, h2c, st);
}

void level_up(int kind, int n, float *e, const float *eb, const float *r, const float *inv, const float *ec, double h2,
              float *uh, float *ul, cudaStream_t st)
{
    if (n == 32) up_c<Tile32>(kind, e, eb, r, inv, ec, h2, uh, ul, st);
    else up_c<Tile64>(kind, e, eb, r, inv, ec, h2, uh, ul, st);
}

}  // namespace gr
