// deposit_tiles.cu - the cloud-in-cell deposit over tiles of 8^3 cells, for
// particle sets that fill the grid (field_kernels.cu and particle_kernels.cu
// keep the direct kernels for sparse ones).
//
// The direct kernel adds forty doubles per particle to memory: 5.4e9 FP64
// atomics for 134M particles, which L2 takes at 290e9/s (measured limits: 238e9
// sectors/s, 534e9 elements/s), next to 47 FP64 operations per particle on a
// pipe that issues 2 lanes per cycle.  Here the particles are first put in
// tile order (count with the particle's rank in its tile, scan, scatter of the
// indices), then a block sums up to 1024 particles of one tile (an item) in shared
// memory, over the tile's 9^3 reached cells, and adds each cell's five sums to memory once.
//
// An item's sums are exact integers of 64 bits.  The unit of s0 and s_l is 2^-60 of a bound on the
// item's charges of that kind (its largest component of u gives it), of sigma, whose range is twice as wide,
// 2^-60 of the bound from the particles around the cell; in a cell that more than eight of the item's particles
// reach it is coarser by the bits that their number may need.  Weights are 62-bit integers, products of the
// positions' fractions, which integer operations take from the FP64 positions.
// A 64-bit shared-memory addition is two native 32-bit atomics, the second
// with the first one's carry (measured over tiles: 1300 to 2300e9 additions/s; the
// FP64 atomic is a compare-and-swap loop at 250 to 490e9/s).  Items and neighbouring
// tiles meet in FP64 atomics (cells inside the tile of a single item are stored), so the last bit of such
// a cell depends on the order in which they arrive.
//
// Error: a charge is off by about half a unit and a sum by nothing more.  A sum that is small in those units (its
// cell holds slow particles beside fast ones, grazing clouds or opposite velocities) would have
// few correct bits: below 2^46 times the units it may be off by, the sum is dropped and its charges are
// added in FP64 by k_dt_redo, from a list of particles (of 134M at contrast 5, 4% are listed; what does
// not fit the list is added by the block).  Measured against FP64 sums, 4.2M particles on 128^3, rms contrast 5, in
// units of the sum of the charges' magnitudes in a cell: worst cell 9.2e-15, rms 1.8e-16; the direct kernels'
// double-float products 1.1e-14 and 1.1e-15.  Without the list the worst was 1.3e-9, and
// 2.5e-5 with a velocity of 1 in every 5000th particle and 1e-9 in the others.
//
// Bound: integer multiplies and the additions' bank conflicts (four wavefronts each for clustered
// particles), at 62% occupancy (48 registers; 4 blocks of 60 registers took 4%
// more).  Measured, 134M particles on 512^3, rms contrast 5: 18.8 -> 15.4 ms
// (order 2.2 ms, sums 11.8 ms, list 0.7 ms, zeroing 0.8 ms; without the list and the bounds per cell 12.8).
//
// Items whose charges leave the scaled range (not finite, or 2^200 and more)
// and particles at positions that are not finite are listed with all their charges.
#include <cuda_runtime.h>

#include <cmath>

#include "df64.cuh"
#include "gr_internal.cuh"

namespace gr {
namespace {

constexpr int kTile = 8, kReach = kTile + 1, kReachCells = kReach * kReach * kReach;
constexpr int kSeg = 1024;         // particles per block
constexpr int kSegThreads = 256;
constexpr int kScanThreads = 1024;  // tiles per block of the scan
constexpr int kUnit = 52;          // to_units' scale
constexpr int kBits = 60;          // bits of a block's largest charge in cells of few particles
constexpr unsigned kBad = 512u;     // flag beside a particle's cell in its tile
constexpr int kWords = (10 * kReachCells + 3) / 4 * 4;
constexpr int kPad = kReach + 1;    // a tile's cells with a border below and above, per axis
// A cell's sum of m charges is off by up to kDeviation sqrt(m) units (four standard deviations of m
// roundings to a unit, 0.29 each); it is kept if that is 2^-46 of it or less
constexpr float kDeviation = 1.2f;

typedef unsigned long long u64;

struct Item {
    unsigned tile, first, count;
};

// a particle some of whose charges are added directly after the tiles' sums (deposit_direct's todo)
struct Redo {
    u64 todo;
    unsigned p, pad;
};

// t = the argument times 2^shift: floor(t) and the fraction t - floor(t) in units of 2^-62 (positions below
// 2^-62 of a cell are dropped), by integer operations on t's bits; wide: t is
// beyond 2^30 cells or not finite (no cell, no fraction)
__device__ __forceinline__ int split_cell(double t, u64 &frac, bool &wide, int shift = 0)
{
    const long long b = __double_as_longlong(t);
    const int ex = (int)((b >> 52) & 0x7ff) - 1023 + shift;
    wide = ex >= 30;
    if (wide) {
        frac = 0;
        return 0;
    }
    const u64 m = ((u64)b & 0xfffffffffffffull) | 0x10000000000000ull;
    int c;
    u64 f;  // units of 2^-64
    if (ex >= 0) {
        c = (int)(m >> (52 - ex));
        f = m << (12 + ex);
    } else {
        c = 0;
        f = ex < -64 ? 0ull : (m << 11) >> (-1 - ex);
    }
    if (b < 0) {
        c = f ? -c - 1 : -c;
        f = 0ull - f;
    }
    frac = f >> 2;
    return c;
}

// a b 2^-62 of two 62-bit numbers, to one unit
__device__ __forceinline__ u64 mul62(u64 a, u64 b)
{
    const unsigned ah = (unsigned)(a >> 31), al = (unsigned)a & 0x7fffffffu;
    const unsigned bh = (unsigned)(b >> 31), bl = (unsigned)b & 0x7fffffffu;
    const u64 mid = (u64)ah * bl + (u64)al * bh + (1ull << 30);
    return (u64)ah * bh + (mid >> 31);
}

// x in units of 2^(e - 52); |x| < 2^(e + 4) up to a rounding
__device__ __forceinline__ long long to_units(double x, int e)
{
    const long long b = __double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7ff);
    if (ef == 0) return 0;
    const int sh = e - (ef - 1023) + 8;
    const u64 m = (((u64)b & 0xfffffffffffffull) | 0x10000000000000ull) << 8;
    const long long v = sh > 62 ? 0ll : (long long)((m + (1ull << (sh - 1))) >> sh);
    return b < 0 ? -v : v;
}

// v 2^e rounded to nearest (v != 0, a normal result)
__device__ __forceinline__ double from_units(long long v, int e)
{
    const double d = __ll2double_rn(v);
    return __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

// q w 2^-62 rounded (|q| < 2^57).  The product of the low halves, up to a unit, enters by its
// leading 30 bits: left out, it would be a bias, which a crowd of particles at one place sums up
__device__ __forceinline__ long long scale62(int qh, int ql, int wh, int wl)
{
    const unsigned low = (1u << 30) + 2u * (unsigned)((ql >> 16) * (wl >> 16));
    const long long mid = (long long)qh * wl + ((long long)ql * wh + (long long)low);
    return (long long)qh * wh + (mid >> 31);
}

// v >> s of v >= 0, zero from s = 64 on
__device__ __forceinline__ long long shift_down(long long v, int s)
{
    long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}

struct Grid {
    int lgn;
    double invh;
    int lgh;  // invh = 2^lgh (exactly), or -1
};

// The FP64 form, for coordinates of 2^30 cells and more: wrapped into the grid as the
// direct kernels wrap them.  bad: not finite, the fraction then is no number
struct WideCell {
    int lo;
    bool bad;
    u64 frac;
};
static __device__ __noinline__ WideCell cell_wide(double x, double invh, int m)
{
    const double t = fma(x, invh, -0.5), fl = floor(t), fr = t - fl;
    const bool bad = !(fr < 1.0);
    return {(int)((long long)fl & m), bad, bad ? 0ull : (u64)(fr * 0x1p62)};
}

// cells (to be wrapped into the grid) and fractions of a position: t = x / h - 1/2.  With 1/h a power of two
// (any box whose side is one) the scaling is an exponent and the half is
// taken off the fraction: no FP64 operation.  Every pass calls it, so a particle is summed in the tile it
// was counted in.
__device__ __forceinline__ void cells_of(const Grid &g, const double (&x)[3], int (&c)[3], u64 (&frac)[3], bool &bad)
{
    const u64 half = 1ull << 61;
    unsigned far = 0u;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        bool wide;
        if (g.lgh < 0) {
            c[d] = split_cell(fma(x[d], g.invh, -0.5), frac[d], wide);
        } else {
            c[d] = split_cell(x[d], frac[d], wide, g.lgh);
            if (frac[d] < half) c[d]--;
            frac[d] = (frac[d] - half) & ((1ull << 62) - 1);
        }
        far |= (wide ? 1u : 0u) << d;
    }
    bad = false;
    if (far == 0u) return;
#pragma unroll
    for (int d = 0; d < 3; d++)
        if (far >> d & 1u) {
            const WideCell w = cell_wide(x[d], g.invh, (1 << g.lgn) - 1);
            c[d] = w.lo;
            frac[d] = w.frac;
            bad |= w.bad;
        }
}

__device__ __forceinline__ unsigned tile_of(const Grid &g, const int lo[3])
{
    const int m = (1 << g.lgn) - 1, lt = g.lgn - 3;
    return (unsigned)(((((lo[0] & m) >> 3) << lt) + ((lo[1] & m) >> 3)) << lt) + (unsigned)((lo[2] & m) >> 3);
}

// tile, cell within it (9 bits), whether its position is not finite (bit 9), and rank within the tile (arrival
// order) of every particle; the lanes of a warp that share a tile take one atomic
__global__ void __launch_bounds__(kBlock)
    k_dt_count(Grid g, int64_t np, int64_t stride, const double *__restrict__ x, unsigned *__restrict__ count,
               uint2 *__restrict__ key)
{
    pdl_begin();
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool ok = p < np;
    int lo[3] = {0, 0, 0};
    bool bad = false;
    if (ok) {
        const double xd[3] = {x[p], x[stride + p], x[2 * stride + p]};
        u64 f[3];
        cells_of(g, xd, lo, f, bad);
    }
    const unsigned tile = ok ? tile_of(g, lo) : 0xffffffffu;
    const unsigned same = __match_any_sync(0xffffffffu, tile);
    const int lane = threadIdx.x & 31, leader = __ffs(same) - 1;
    unsigned base = 0;
    if (ok && lane == leader) base = atomicAdd(count + tile, (unsigned)__popc(same));
    base = __shfl_sync(0xffffffffu, base, leader);
    const unsigned cell = (unsigned)((((lo[0] & 7) << 3) | (lo[1] & 7)) << 3 | (lo[2] & 7)) | (bad ? kBad : 0u);
    if (ok) key[p] = make_uint2(tile << 10 | cell, base + __popc(same & ((1u << lane) - 1)));
}

// particles (high half) and items (low half) of tile t
__device__ __forceinline__ u64 tile_load(int ntile, const unsigned *count, int t)
{
    const unsigned c = t < ntile ? count[t] : 0u;
    return ((u64)c << 32) + (c + kSeg - 1) / kSeg;
}

// sum of v over the block (kScanThreads), for every thread
__device__ __forceinline__ u64 block_total(u64 v, u64 *warp)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) warp[w] = v;
    __syncthreads();
    v = warp[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    return v;
}

// totals of kScanThreads tiles per block
__global__ void __launch_bounds__(kScanThreads)
    k_dt_totals(int ntile, const unsigned *__restrict__ count, u64 *__restrict__ total)
{
    pdl_begin();
    __shared__ u64 warp[kScanThreads / 32];
    const u64 v = block_total(tile_load(ntile, count, blockIdx.x * kScanThreads + threadIdx.x), warp);
    if (threadIdx.x == 0) total[blockIdx.x] = v;
}

// exclusive offsets of the tiles and the list of items (at most kSeg particles
// of one tile each); *nitem their number
__global__ void __launch_bounds__(kScanThreads)
    k_dt_scan(int ntile, const unsigned *__restrict__ count, const u64 *__restrict__ total, unsigned *__restrict__ off,
              Item *__restrict__ items, unsigned *__restrict__ nitem)
{
    pdl_begin();
    __shared__ u64 warp[kScanThreads / 32];
    u64 before = 0;  // the blocks before this one
    for (int q = threadIdx.x; q < (int)blockIdx.x; q += kScanThreads) before += total[q];
    before = block_total(before, warp);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int t = blockIdx.x * kScanThreads + threadIdx.x;
    const u64 own = tile_load(ntile, count, t);
    u64 inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u64 v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) warp[w] = inc;
    __syncthreads();
    u64 wsum = lane < w ? warp[lane] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
    const u64 at = before + wsum + inc - own;
    if (t < ntile) {
        const unsigned c = (unsigned)(own >> 32), first = (unsigned)(at >> 32), it = (unsigned)at;
        off[t] = first;
        for (unsigned s = 0; s * kSeg < c; s++) {
            const unsigned left = c - s * kSeg;
            items[it + s] = {(unsigned)t, first + s * kSeg, left < kSeg ? left : (unsigned)kSeg};
        }
        if (t == ntile - 1) *nitem = (unsigned)(at + own);
    }
}

__global__ void __launch_bounds__(kBlock)
    k_dt_scatter(int64_t np, const uint2 *__restrict__ key, const unsigned *__restrict__ off, uint2 *__restrict__ perm)
{
    pdl_begin();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < np; p += (int64_t)gridDim.x * blockDim.x) {
        const uint2 k = key[p];
        perm[off[k.x >> 10] + k.y] = make_uint2((unsigned)p, k.x & 1023u);
    }
}

struct Out {
    double *s[5];
};

// One particle straight to memory in FP64.  (cx, cy, cz), f: its cell and fractions by cell_of, so that it
// adds to no cells but those its tile reaches (cells inside another tile may take that tile's plain
// stores at any time); a coordinate that is not finite has no fraction and spoils its cells.
// todo: five bits per corner (2^(4 a + 2 b + c), lowest first), the charges to be added there
static __device__ __noinline__ void deposit_direct(const Grid g, double q, double x, double y, double z, int cx, int cy,
                                                   int cz, u64 f0, u64 f1, u64 f2, double ux, double uy, double uz,
                                                   const double *psi, u64 todo, const Out out)
{
    const int m = (1 << g.lgn) - 1;
    const double x3[3] = {x, y, z};
    const u64 f[3] = {f0, f1, f2};
    const int lo[3] = {cx, cy, cz};
    double fw[3][2];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const double t = x3[d] * g.invh, fr = (double)f[d] * 0x1p-62 + (t - t);  // + 0, or NaN
        fw[d][0] = 1.0 - fr;
        fw[d][1] = fr;
    }
    auto id = [&](int a, int b, int c) {
        return (((((lo[0] + a) & m) << g.lgn) + ((lo[1] + b) & m)) << g.lgn) + ((lo[2] + c) & m);
    };
    double Q[5] = {0.0, q * ux, q * uy, q * uz, 0.0};
    constexpr u64 kLorentz = 0x11ull * 0x842108421ull;  // s0 and sigma at any corner
    if (todo & kLorentz) {
        double ip4 = 1.0;
        if (psi) {
            double ps = 0.0;
            for (int v = 0; v < 8; v++)
                ps = fma((v & 4 ? fw[0][1] : fw[0][0]) * (v & 2 ? fw[1][1] : fw[1][0]) * (v & 1 ? fw[2][1] : fw[2][0]),
                         psi[id(v >> 2, (v >> 1) & 1, v & 1)], ps);
            const double ip2 = 1.0 / (ps * ps);
            ip4 = ip2 * ip2;
        }
        const double u2 = fma(ux, ux, fma(uy, uy, uz * uz)), w2 = fma(ip4, u2, 1.0), rw = rsqrt(w2);
        Q[0] = q * (w2 * rw);
        Q[4] = (q * u2) * rw;
    }
    for (int v = 0; v < 8; v++) {
        const double w = (v & 4 ? fw[0][1] : fw[0][0]) * (v & 2 ? fw[1][1] : fw[1][0]) * (v & 1 ? fw[2][1] : fw[2][0]);
        const int c = id(v >> 2, (v >> 1) & 1, v & 1);
#pragma unroll
        for (int k = 0; k < 5; k++)
            if (todo >> (5 * v + k) & 1u) atomicAdd(out.s[k] + c, Q[k] * w);
    }
}

// the listed charges of a particle
template <bool METRIC>
__device__ __forceinline__ void redo_one(const Grid &g, int64_t stride, const double *__restrict__ x,
                                         const double *__restrict__ u, double q, const double *__restrict__ psi, Redo e,
                                         const Out &out)
{
    const double xd[3] = {x[e.p], x[stride + e.p], x[2 * stride + e.p]};
    int c[3];
    u64 f[3];
    bool bad;
    cells_of(g, xd, c, f, bad);
    const int m = (1 << g.lgn) - 1;
    deposit_direct(g, q, xd[0], xd[1], xd[2], c[0] & m, c[1] & m, c[2] & m, f[0], f[1], f[2], u[e.p], u[stride + e.p],
                   u[2 * stride + e.p], METRIC ? psi : nullptr, e.todo, out);
}

// sums of one item; q = qm 2^(qe - 62).  METRIC: the Lorentz factor at psi (its values on the
// reached cells are kept in shared memory); add: other launches add to out as well
template <bool METRIC>
__global__ void __launch_bounds__(kSegThreads, 5)
    k_dt_sum(Grid g, int64_t stride, const double *__restrict__ x, const double *__restrict__ u, double q,
             u64 qm, int qe, const double *__restrict__ psi, const uint2 *__restrict__ perm, const Item *__restrict__ items, const unsigned *__restrict__ nitem, const unsigned *__restrict__ count, int add,
             Redo *__restrict__ redo, unsigned *__restrict__ nredo, unsigned room, Out out)
{
    pdl_begin();
    // words of the sums, low and high; before them, per cell of the tile, its particles and the largest high word
    // of their |u|; after them the list of particles to be redone
    __shared__ __align__(16) unsigned acc[kWords];
    unsigned *const acc_lo = acc, *const acc_hi = acc + 5 * kReachCells;
    unsigned *const in_count = acc, *const in_top = acc + kPad * kPad * kPad;
    unsigned short *const list = reinterpret_cast<unsigned short *>(acc);
    __shared__ double ps[METRIC ? kReachCells : 1];
    __shared__ unsigned short from[kReachCells];   // particles that reach a cell, then the charges to be redone there
    __shared__ unsigned short scale[kReachCells];  // a cell's units: bits kept free beyond three, 8 x sigma's bits gained
    __shared__ unsigned top[5];  // largest high words of |u_x|, |u_y|, |u_z|, smallest of psi, largest of psi
    __shared__ unsigned listed;  // particles to be redone
    if (blockIdx.x >= *nitem) return;
    const Item it = items[blockIdx.x];
    const int m = (1 << g.lgn) - 1, lt = g.lgn - 3, mt = (1 << lt) - 1;
    const int base[3] = {(int)(it.tile >> (2 * lt)) << 3, (int)((it.tile >> lt) & mt) << 3, (int)(it.tile & mt) << 3};
    auto cell_id = [&](int r) {  // grid index of reached cell r
        const int a = r / (kReach * kReach), b = (r / kReach) % kReach, c = r % kReach;
        return (((((base[0] + a) & m) << g.lgn) + ((base[1] + b) & m)) << g.lgn) + ((base[2] + c) & m);
    };
    for (int r = threadIdx.x; r < 2 * kPad * kPad * kPad; r += kSegThreads) acc[r] = 0u;
    if (threadIdx.x < 5) top[threadIdx.x] = threadIdx.x == 3 ? 0xffffffffu : 0u;
    if (threadIdx.x == 5) listed = 0u;
    __syncthreads();
    // bounds: the largest exponent of each component of u, the range of psi
    unsigned h[5] = {0u, 0u, 0u, 0xffffffffu, 0u};
    for (unsigned s = threadIdx.x; s < it.count; s += kSegThreads) {
        const uint2 pc = perm[it.first + s];
        const unsigned p = pc.x, c = pc.y & (kBad - 1);
        unsigned own = 0u;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const unsigned v = (unsigned)__double2hiint(u[d * stride + p]) & 0x7fffffffu;
            h[d] = max(h[d], v);
            own = max(own, v);
        }
        const int o = ((int)(c >> 6) * kPad + (int)((c >> 3) & 7u)) * kPad + (int)(c & 7u) + (kPad + 1) * kPad + 1;
        atomicAdd(in_count + o, 1u);
        atomicMax(in_top + o, own);
    }
    if (METRIC)
        for (int r = threadIdx.x; r < kReachCells; r += kSegThreads) {
            const double v = psi[cell_id(r)];
            ps[r] = v;
            h[3] = min(h[3], (unsigned)__double2hiint(v));
            h[4] = max(h[4], (unsigned)__double2hiint(v));  // a negative psi is the largest
        }
#pragma unroll
    for (int d = 0; d < (METRIC ? 5 : 3); d++) {
        const unsigned v = d == 3 ? __reduce_min_sync(0xffffffffu, h[d]) : __reduce_max_sync(0xffffffffu, h[d]);
        if ((threadIdx.x & 31) == 0) {
            if (d == 3) atomicMin(top + d, v);
            else atomicMax(top + d, v);
        }
    }
    __syncthreads();
    // exponents: |u_d| < 2^e[1 + d]; W and u^2 / W from the largest, E
    int e[5], E = -1023;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        e[1 + d] = (int)(top[d] >> 20) - 1022;
        E = max(E, e[1 + d]);
    }
    const int px = METRIC ? (int)(top[3] >> 20) - 1023 : 0;  // psi >= 2^px, psi^-2 |u_d| < 2^(E - 2 px)
    const int Ew = E - 2 * px;
    e[0] = max(1, Ew + 1);  // W^2 < 1 + 3 4^Ew
    // sigma's charge from the largest |u_d|: u^2 / W <= u^2 < 3 4^E, and <= psi^2 |u|
    const int px2 = METRIC ? 2 * ((int)(top[4] >> 20) - 1022) : 0;
    auto sigma_exp = [&](int E1) { return max(min(2 * E1 + 2, E1 + 1 + px2), -400); };
    e[4] = sigma_exp(E);
    const bool scaled = E < 200 && (!METRIC || ((top[4] >> 31) == 0u && (int)(top[4] >> 20) - 1023 < 50 && px > -50));
    // charges that vanish on the whole block, or nearly, need no unit of their own
#pragma unroll
    for (int k = 0; k < 4; k++) e[k] = max(e[k], -400);
    // a cell's units: the sum of n charges below 2^(63 - lg n) units stays below 2^63, and sigma's bound
    // there is that of the particles in the eight cells below it
    for (int r = threadIdx.x; r < kReachCells; r += kSegThreads) {
        const int a = r / (kReach * kReach), b = (r / kReach) % kReach, c = r % kReach;
        const int o = (a * kPad + b) * kPad + c;
        unsigned n = 0, t = 0;
#pragma unroll
        for (int v = 0; v < 8; v++) {
            const int q = o + ((v >> 2) * kPad + ((v >> 1) & 1)) * kPad + (v & 1);
            n += in_count[q];
            t = max(t, in_top[q]);
        }
        from[r] = (unsigned short)n;
        const int more = n > 8u ? 29 - __clz(n - 1u) : 0;  // lg n - 3, rounded up
        scale[r] = (unsigned short)(more | (e[4] - sigma_exp((int)(t >> 20) - 1022)) << 3);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < kWords / 4; r += kSegThreads)
        reinterpret_cast<uint4 *>(acc)[r] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    for (unsigned s = threadIdx.x; scaled && s < it.count; s += kSegThreads) {
        const unsigned p = perm[it.first + s].x;
        const double xd[3] = {x[p], x[stride + p], x[2 * stride + p]};
        const double ud[3] = {u[p], u[stride + p], u[2 * stride + p]};
        int lc[3];
        u64 f[3];
        double fr[3];
        bool bad;
        cells_of(g, xd, lc, f, bad);
#pragma unroll
        for (int d = 0; d < 3; d++) {
            lc[d] &= kTile - 1;
            if (METRIC) fr[d] = f[d] ? from_units((long long)f[d], -62) : 0.0;
        }
        if (bad) continue;
        const int r0 = (lc[0] * kReach + lc[1]) * kReach + lc[2];
        double ip4 = 1.0;
        if (METRIC) {  // psi at the particle
            double v[2][2], y[2];
#pragma unroll
            for (int a = 0; a < 2; a++)
#pragma unroll
                for (int b = 0; b < 2; b++) {
                    const double *o = ps + r0 + (a * kReach + b) * kReach;
                    v[a][b] = fma(fr[2], o[1] - o[0], o[0]);
                }
#pragma unroll
            for (int a = 0; a < 2; a++) y[a] = fma(fr[1], v[a][1] - v[a][0], v[a][0]);
            const double pp = fma(fr[0], y[1] - y[0], y[0]), ip2 = 1.0 / (pp * pp);
            ip4 = ip2 * ip2;
        }
        const double u2 = fma(ud[0], ud[0], fma(ud[1], ud[1], ud[2] * ud[2]));
        const double w2 = METRIC ? fma(ip4, u2, 1.0) : 1.0 + u2, rw = rsqrt64(w2);
        const double Q[4] = {w2 * rw, ud[0], ud[1], ud[2]};
        int qh[5], ql[5];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const long long v = to_units(Q[k], e[k] + kUnit - kBits);
            qh[k] = (int)(v >> 31);
            ql[k] = (int)(v & 0x7fffffffll);
        }
        // sigma goes with its own leading bits, shifted down by sh (less the cell's gain) at the end
        int sh;
        {
            const long long b = __double_as_longlong(u2 * rw);
            const int ex = (int)(b >> 52) - 1023;
            const long long v = ex == -1023 ? 0ll : ((b & 0xfffffffffffffll) | 0x10000000000000ll) << (kBits - 53);
            sh = max(e[4] - ex, 1) - 1;
            qh[4] = (int)(v >> 31);
            ql[4] = (int)(v & 0x7fffffffll);
        }
        u64 w[3][2];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            w[d][1] = f[d];
            w[d][0] = (1ull << 62) - (f[d] ? f[d] : 1ull);
        }
        w[0][0] = mul62(w[0][0], qm);  // the mass: its mantissa here, its exponent in the unit
        w[0][1] = mul62(w[0][1], qm);
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int b = 0; b < 2; b++) {
                const u64 wab = mul62(w[0][a], w[1][b]);
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    const int r = r0 + (a * kReach + b) * kReach + c;
                    const int sc = scale[r], drop = sc & 7;
                    // rounded: a crowd's truncations would add up (6000 particles within 3e-4 cells of a centre: twice the error)
                    const u64 wt = (mul62(wab, w[2][c]) + ((1u << drop) >> 1)) >> drop;
                    const int wh = (int)(wt >> 31), wl = (int)(wt & 0x7fffffffull);
#pragma unroll
                    for (int k = 0; k < 5; k++) {
                        long long v = scale62(qh[k], ql[k], wh, wl);
                        if (k == 4) v = (shift_down(2 * v, sh - (sc >> 3)) + 1) >> 1;
                        const unsigned vl = (unsigned)v;
                        const unsigned old = atomicAdd(acc_lo + k * kReachCells + r, vl);
                        atomicAdd(acc_hi + k * kReachCells + r, (unsigned)((u64)v >> 32) + (old + vl < old ? 1u : 0u));
                    }
                }
            }
    }
    __syncthreads();
    // a cell inside the tile is no other tile's: a plain store if this is the tile's only
    // item (what is redone is added after it, and the sum to be redone not stored)
    const bool alone = !add && count[it.tile] <= kSeg;
    for (int r = threadIdx.x; scaled && r < kReachCells; r += kSegThreads) {
        const int a = r / (kReach * kReach), b = (r / kReach) % kReach, c = r % kReach;
        const bool own = alone && a != 0 && a != kTile && b != 0 && b != kTile && c != 0 && c != kTile;
        const int id = cell_id(r);
        const unsigned n = from[r];
        if (n == 0u) continue;
        const int keep = (int)(kDeviation * 0x1p14f * sqrtf((float)n)) + 1;  // high word of the least |sum| kept
        unsigned redo = 0u;
#pragma unroll
        for (int k = 0; k < 5; k++) {
            const long long v = (long long)(((u64)acc_hi[k * kReachCells + r] << 32) | acc_lo[k * kReachCells + r]);
            const int high = (int)(v >> 32);
            if ((high ^ (high >> 31)) < keep) {
                // nothing to redo where the block has no such charge at all
                if (k == 0 || (k == 4 ? (top[0] | top[1] | top[2]) : top[k - 1]) != 0u) redo |= 1u << k;
                continue;
            }
            const double d = from_units(v, e[k] - (k == 4 ? scale[r] >> 3 : 0) + (scale[r] & 7) - kBits + qe);
            if (own) out.s[k][id] = d;
            else atomicAdd(out.s[k] + id, d);
        }
        from[r] = (unsigned short)redo;
    }
    // the particles that reach a cell with a sum to be redone, and those that were left out
    __syncthreads();
    for (unsigned s = threadIdx.x; s < it.count; s += kSegThreads) {
        const unsigned pc = perm[it.first + s].y, c = pc & (kBad - 1);
        const unsigned short *const o = from + ((c >> 6) * kReach + ((c >> 3) & 7u)) * kReach + (c & 7u);
        unsigned any = !scaled || (pc & kBad) ? 1u : 0u;
#pragma unroll
        for (int v = 0; v < 8; v++) any |= o[((v >> 2) * kReach + ((v >> 1) & 1)) * kReach + (v & 1)];
        if (any) list[atomicAdd(&listed, 1u)] = (unsigned short)s;
    }
    __syncthreads();
    if (listed == 0u) return;
    if (threadIdx.x == 0) top[0] = atomicAdd(nredo, listed);
    __syncthreads();
    const unsigned slot = top[0];
    for (unsigned t = threadIdx.x; t < listed; t += kSegThreads) {
        const uint2 pc = perm[it.first + list[t]];
        const unsigned p = pc.x, c = pc.y & (kBad - 1);
        const unsigned short *const o = from + ((c >> 6) * kReach + ((c >> 3) & 7u)) * kReach + (c & 7u);
        u64 todo = !scaled || (pc.y & kBad) ? ~0ull : 0ull;
#pragma unroll
        for (int v = 0; v < 8; v++) todo |= (u64)o[((v >> 2) * kReach + ((v >> 1) & 1)) * kReach + (v & 1)] << (5 * v);
        if (slot + t < room) redo[slot + t] = {todo, p, 0u};
        else redo_one<METRIC>(g, stride, x, u, q, psi, {todo, p, 0u}, out);
    }
}

template <bool METRIC>
__global__ void __launch_bounds__(kBlock)
    k_dt_redo(Grid g, int64_t stride, const double *__restrict__ x, const double *__restrict__ u, double q,
              const double *__restrict__ psi, const Redo *__restrict__ redo, const unsigned *__restrict__ nredo,
              unsigned room, Out out)
{
    pdl_begin();
    const unsigned n = min(*nredo, room);
    for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
        redo_one<METRIC>(g, stride, x, u, q, psi, redo[t], out);
}

int lg(int n)
{
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

// places in the list of particles to be redone (16 bytes each): one in 8
int64_t redo_room(int64_t np) { return np / 8 + 1; }

// scratch of a chunk of np particles: keys, indices with cells, redo list, per-tile counts and offsets, items
size_t scratch_bytes(int n, int64_t np)
{
    const size_t T = (size_t)n * n * n / (kTile * kTile * kTile);
    return 16 * (size_t)np + sizeof(Redo) * (size_t)redo_room(np) + 8 * T + 8 * (T / kScanThreads + 1) + sizeof(Item) * (T + (size_t)(np / kSeg) + 1) + 1024;
}

}  // namespace

// Measured against the direct kernels at 0.5 to 4 particles per cell, rms density contrast 0.3, 1 and 5 (lattice
// order; direct / tiles, ms).  Plain, 128^3: at 0.75 per cell 0.195 / 0.219, 0.198 / 0.236, 0.240 / 0.266; at one
// 0.250 / 0.256, 0.252 / 0.264, 0.304 / 0.289; at two 0.468 / 0.434, 0.469 / 0.440, 0.541 / 0.487.  256^3: at 0.75
// 1.43 / 1.47, 1.43 / 1.51, 1.79 / 1.61; at one 1.86 / 1.74, 1.86 / 1.77, 2.24 / 1.90.  512^3 at one: 14.7 / 14.0
// (contrast 1), 18.9 / 15.0 (5).  With the gather of psi, 128^3: at two 0.523 / 0.530, 0.528 / 0.541, 0.594 / 0.593;
// 256^3: at 0.75 1.60 / 1.83, 1.62 / 1.86, 1.95 / 1.98; at one 2.07 / 2.14, 2.10 / 2.18, 2.46 / 2.34; at two 4.07 /
// 3.75, 4.09 / 3.80, 4.35 / 4.06.  The tiles' sums are closer to the exact ones (rms error of a cell 1.8e-16 against
// 1.1e-15), so they are taken down to where they cost a little more time.
bool deposit_tiles_fit(int n, double L, int64_t np, double mass, bool metric, size_t scratch)
{
    const int64_t N = (int64_t)n * n * n;
    const double h = L / n, q = mass / (h * h * h);
    const int64_t least = metric && n < 256 ? 2 * N : N - N / 4;
    return n >= 128 && np >= least && q > 1e-100 && q < 1e100 && scratch_bytes(n, N) <= scratch;
}

void deposit_tiles(int n, double L, int64_t np, int64_t stride, const double *x, const double *u, double mass,
                   const double *psi, double *s0, double *sx, double *sy, double *sz, double *sig, void *scratch,
                   size_t bytes, bool add, cudaStream_t st)
{
    const double h = L / n;
    int hx;
    const double invh = 1.0 / h;
    const bool pow2 = std::frexp(invh, &hx) == 0.5 && hx > -900 && hx < 900;
    const Grid g = {lg(n), invh, pow2 && hx >= 1 ? hx - 1 : -1};
    const double q = mass / (h * h * h);
    int qe;
    const u64 qm = (u64)std::ldexp(std::frexp(q, &qe), 62);
    const Out out = {{s0, sx, sy, sz, sig}};
    const size_t T = (size_t)n * n * n / (kTile * kTile * kTile);
    // as many particles at a time as the scratch holds (and as 31-bit indices count)
    int64_t chunk = np;
    while (scratch_bytes(n, chunk) > bytes || chunk > (int64_t)1 << 30) chunk = (chunk + 1) / 2;
    for (int64_t p0 = 0; p0 < np; p0 += chunk) {
        const int64_t c = np - p0 < chunk ? np - p0 : chunk;
        char *b = (char *)scratch;
        const unsigned room = (unsigned)redo_room(c);
        Redo *redo = (Redo *)b;
        b += sizeof(Redo) * (size_t)room;
        uint2 *key = (uint2 *)b, *perm = key + c;
        b += 16 * (size_t)c;
        u64 *total = (u64 *)b;
        const int sb = (int)((T + kScanThreads - 1) / kScanThreads);
        b += 8 * (size_t)sb;
        Item *items = (Item *)b;
        const size_t nit = T + (size_t)(c / kSeg) + 1;
        b += sizeof(Item) * nit;
        unsigned *count = (unsigned *)b, *nredo = count + T, *nitem = nredo + 1, *off = nitem + 1;
        cudaMemsetAsync(count, 0, (T + 1) * sizeof(unsigned), st);
        GR_LAUNCH(k_dt_count, (unsigned)((c + kBlock - 1) / kBlock), kBlock, st, g, c, stride, x + p0, count, key);
        GR_LAUNCH(k_dt_totals, sb, kScanThreads, st, (int)T, count, total);
        GR_LAUNCH(k_dt_scan, sb, kScanThreads, st, (int)T, count, total, off, items, nitem);
        GR_LAUNCH(k_dt_scatter, wave_grid(k_dt_scatter, c), kBlock, st, c, key, off, perm);
        const int more = (add || chunk < np) ? 1 : 0;
        const int gr2 = wave_grid(psi ? k_dt_redo<true> : k_dt_redo<false>, room);
        if (psi) {
            GR_LAUNCH(k_dt_sum<true>, (unsigned)nit, kSegThreads, st, g, stride, x + p0, u + p0, q, qm, qe, psi, perm,
                      items, nitem, count, more, redo, nredo, room, out);
            GR_LAUNCH(k_dt_redo<true>, gr2, kBlock, st, g, stride, x + p0, u + p0, q, psi, redo, nredo, room, out);
        } else {
            GR_LAUNCH(k_dt_sum<false>, (unsigned)nit, kSegThreads, st, g, stride, x + p0, u + p0, q, qm, qe, psi, perm,
                      items, nitem, count, more, redo, nredo, room, out);
            GR_LAUNCH(k_dt_redo<false>, gr2, kBlock, st, g, stride, x + p0, u + p0, q, psi, redo, nredo, room, out);
        }
    }
}

}  // namespace gr
