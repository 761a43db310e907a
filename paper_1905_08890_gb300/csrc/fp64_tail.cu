// fp64_tail.cu - levels 16^3 .. 2^3 of one FP64 V-cycle in one launch: a
// thread-block cluster of 16 CTAs, CTA r holding plane i = r of every level
// of at least r + 1 planes.
//
// Below 32^3 a level's FP64 pass is latency: GB300's FP64 pipe returns a
// dependent operation after 64 cycles (measured), a relaxation is a chain of
// five to six of them, and a launch of its own adds 1.5 to 2 us.  One CTA alone
// would be bound by its two FP64 lanes per cycle (a 16^3 colour pass is 2048
// x 7 operations, 4 us), so the planes are spread over 16 SMs.  A plane's
// result is pushed into the two neighbouring CTAs' halo copies (distributed
// shared memory), so a pass reads local shared memory only, and a cluster
// barrier (0.2 us at 128 threads) takes the place of the kernel boundary.
//
// The operations are those of the per-level kernels: red-black sweeps,
// residual and 8-child restriction (KPSI: full approximation scheme), the 2^3
// level solved in CTA 0, trilinear prolongation.  Sums are paired to shorten
// the chains, reciprocals are Newton's iteration, and after a black pass of a linear
// kind the black residuals, zero up to rounding, are not formed.
// Measured at 32^3: the three levels and the 2^3 solve took 34 launches of 2
// to 5 us each per linear cycle (psi: 240 us for the 2^3 sweeps alone); this
// launch takes 27 us (69 us for psi).  With it, the finer prolongation and the
// red-only restriction (mg_kernels.cu) a 32^3 FP64 solve of the ten equations
// went from 19.1 to 8.8 ms.
#include <cooperative_groups.h>

#include "coarse_tail.cuh"
#include "gr_internal.cuh"

namespace cg = cooperative_groups;

namespace gr {
namespace {

constexpr int kT64Ctas = 16, kT64Threads = 128;

// arrays of levels 2^3 .. 16^3 (index 0 = 2^3); u and f of the top level in, u out
struct T64Args {
    double *u;
    const double *f;
    const double *c0[4], *c1[4];
    double h2[4], ih2[4];
    double rho;
    int top;  // index of the top level, 1 .. 3
};

__host__ __device__ constexpr int plane_off(int l) { return ((4 << (2 * l)) - 4) / 3; }  // planes of levels < l

struct T64Smem {
    double u[3 * 340];   // per level: plane r - 1, plane r, plane r + 1
    double f[340], c0[340], c1[340], ur[340];
    double part[2 * 340], partu[2 * 340];  // 8-child sums from the two fine planes
    double cb[2 * 340];  // coarser level's correction for this CTA's plane: own and neighbouring coarse plane
    double zf[2][2][4], zu[2][2][4];       // the 2^3 level's incoming sums [plane][half][cell]
    double z0[8], z1[8], zb[8];
};

// N(u) at a cell without its right-hand side; nb the neighbour sum
template <int KIND>
__device__ __forceinline__ double op64(double nb, double u, double c0, double c1, double ih2, double rho)
{
    const double lap = fma(-6.0, u, nb) * ih2;
    if (KIND == KPOISSON) return lap;
    if (KIND == KHELM) return fma(-c0, u, lap);
    const double v = 1.0 + u, iv = recip64(v), iv2 = iv * iv, iv4 = iv2 * iv2, v2 = v * v, v4 = v2 * v2;
    const double a = fma(2.0 * kPi * c0, iv, lap), b = (0.125 * c1) * (iv4 * iv2 * iv);
    return (a + b) - (2.0 * kPi * rho) * (v4 * v);
}

// one relaxation; KPSI: a Newton step (Sec. 4.3.2)
template <int KIND>
__device__ __forceinline__ double relax64(double nb, double u, double f, double c0, double c1, double h2, double ih2,
                                          double rho)
{
    if (KIND == KPOISSON) return fma(-h2, f, nb) * (1.0 / 6.0);
    if (KIND == KHELM) return fma(-h2, f, nb) * c1;
    const double v = 1.0 + u, iv = recip64(v), iv2 = iv * iv, iv4 = iv2 * iv2, v2 = v * v, v4 = v2 * v2;
    const double s = 2.0 * kPi * c0, p = 2.0 * kPi * rho;
    const double g = (fma(fma(-6.0, u, nb), ih2, -f) + s * iv) + fma((0.125 * c1) * (iv4 * iv2), iv, -p * (v4 * v));
    const double dg = (fma(-s, iv2, -6.0 * ih2) - (0.875 * c1) * (iv4 * iv4)) - (5.0 * p) * v4;
    return fma(-g, recip64(dg), u);
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

template <int KIND>
struct Tail64 {
    T64Smem &S;
    const T64Args &A;
    const int r;  // this CTA's plane
    cg::cluster_group cl;

    __device__ double *uo(int l) { return S.u + 3 * plane_off(l) + (4 << (2 * l)); }  // own plane

    // write a cell of the own plane and the neighbours' copies of it
    __device__ void put(int l, int id, double v)
    {
        const int n = 2 << l, nn = n * n;
        double *o = uo(l) + id;
        *o = v;
        *cl.map_shared_rank(o - nn, (r + 1) & (n - 1)) = v;
        *cl.map_shared_rank(o + nn, (r - 1) & (n - 1)) = v;
    }
    __device__ double nbsum(int l, int j, int k)
    {
        const int n = 2 << l, m = n - 1, nn = n * n;
        const double *o = uo(l);
        const int id = j * n + k;
        return ((o[id + nn] + o[id - nn]) + (o[((j + 1) & m) * n + k] + o[((j - 1) & m) * n + k])) +
               (o[j * n + ((k + 1) & m)] + o[j * n + ((k - 1) & m)]);
    }
    __device__ void sweep(int l, int color)
    {
        const int n = 2 << l, po = plane_off(l);
        if (r < n)
            for (int t = threadIdx.x; t < n * n / 2; t += kT64Threads) {
                const int j = t >> l, k = 2 * (t & ((1 << l) - 1)) + ((r + j + color) & 1), id = j * n + k;
                put(l, id, relax64<KIND>(nbsum(l, j, k), uo(l)[id], S.f[po + id], S.c0[po + id], S.c1[po + id], A.h2[l],
                                         A.ih2[l], A.rho));
            }
        cluster_barrier();
    }
    // residual of level l and its 8-child sums into level l - 1's owner (the
    // 2^3 level's into CTA 0), then the coarse start and right-hand side
    __device__ void down(int l, bool red_only)
    {
        const int n = 2 << l, nc = n / 2, po = plane_off(l);
        if (r < n)
            for (int t = threadIdx.x; t < nc * nc; t += kT64Threads) {
                const int J = t >> l, K = t & (nc - 1);
                double s = 0.0, su = 0.0;
#pragma unroll
                for (int b = 0; b < 2; b++)
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        const int j = 2 * J + b, k = 2 * K + c, id = j * n + k;
                        if (red_only && ((r + j + k) & 1)) continue;
                        const double u = uo(l)[id];
                        s += op64<KIND>(nbsum(l, j, k), u, S.c0[po + id], S.c1[po + id], A.ih2[l], A.rho) - S.f[po + id];
                        su += u;
                    }
                if (l > 1) {
                    const int w = 2 * plane_off(l - 1) + (r & 1) * nc * nc + t;
                    *cl.map_shared_rank(S.part + w, r >> 1) = s;
                    if (KIND == KPSI) *cl.map_shared_rank(S.partu + w, r >> 1) = su;
                } else {
                    *cl.map_shared_rank(&S.zf[r >> 1][r & 1][t], 0) = s;
                    if (KIND == KPSI) *cl.map_shared_rank(&S.zu[r >> 1][r & 1][t], 0) = su;
                }
            }
        cluster_barrier();
        if (l == 1) return;
        const int pc = plane_off(l - 1);
        if (r < nc)
            for (int t = threadIdx.x; t < nc * nc; t += kT64Threads) {
                const double R = 0.125 * (S.part[2 * pc + t] + S.part[2 * pc + nc * nc + t]);
                if (KIND == KPSI) {
                    const double uc = 0.125 * (S.partu[2 * pc + t] + S.partu[2 * pc + nc * nc + t]);
                    S.f[pc + t] = R;
                    S.ur[pc + t] = uc;
                    put(l - 1, t, uc);
                } else {
                    S.f[pc + t] = -R;  // u is zero since the start
                }
            }
        if (KIND == KPSI) {
            cluster_barrier();  // N(uc) needs the neighbouring planes
            if (r < nc)
                for (int t = threadIdx.x; t < nc * nc; t += kT64Threads)
                    S.f[pc + t] = op64<KIND>(nbsum(l - 1, t / nc, t & (nc - 1)), uo(l - 1)[t], S.c0[pc + t],
                                             S.c1[pc + t], A.ih2[l - 1], A.rho) -
                                  S.f[pc + t];
            cluster_barrier();  // before the next pass changes them
        } else {
            __syncthreads();  // the next pass reads what other threads of this CTA wrote
        }
    }
    // plane r of level l - 1's correction to the fine planes that read it
    __device__ void send(int l, int rc, int t, double v)
    {
        const int n = 2 << l, nc = n / 2;
#pragma unroll
        for (int d = -1; d <= 2; d++) {
            const int fi = (2 * rc + d) & (n - 1), nbr = (fi >> 1) != rc;
            *cl.map_shared_rank(S.cb + 2 * plane_off(l - 1) + nbr * nc * nc + t, fi) = v;
        }
    }
    // trilinear prolongation onto level l (3/4 and 1/4 per axis)
    __device__ void up(int l, bool black_only)
    {
        const int n = 2 << l, nc = n / 2, mc = nc - 1, pc = plane_off(l - 1);
        if (l > 1) {
            if (r < nc)
                for (int t = threadIdx.x; t < nc * nc; t += kT64Threads)
                    send(l, r, t, KIND == KPSI ? uo(l - 1)[t] - S.ur[pc + t] : uo(l - 1)[t]);
        } else if (r == 0 && threadIdx.x < 8) {
            const int p = threadIdx.x >> 2, t = threadIdx.x & 3;
            send(l, p, t, S.zb[threadIdx.x]);
        }
        cluster_barrier();
        if (r < n) {
            const double *own = S.cb + 2 * pc, *nbr = own + nc * nc;
            for (int t = threadIdx.x; t < (black_only ? n * n / 2 : n * n); t += kT64Threads) {
                int j, k;
                if (black_only) {
                    j = t >> l;
                    k = 2 * (t & ((1 << l) - 1)) + ((r + j + 1) & 1);
                } else {
                    j = t >> (l + 1);
                    k = t & (n - 1);
                }
                const int J = j >> 1, J1 = (J + ((j & 1) ? 1 : -1)) & mc, K = k >> 1, K1 = (K + ((k & 1) ? 1 : -1)) & mc;
                auto y = [&](int a, int b) { return fma(3.0, own[a * nc + b], nbr[a * nc + b]); };
                const double z = fma(3.0, fma(3.0, y(J, K), y(J, K1)), fma(3.0, y(J1, K), y(J1, K1)));
                put(l, j * n + k, fma(1.0 / 64.0, z, uo(l)[j * n + k]));
            }
        }
        cluster_barrier();
    }
    // the 2^3 level, by the first warp of CTA 0: lane x < 8 holds cell x = 4i + 2j + k
    __device__ void coarsest()
    {
        if (r != 0 || threadIdx.x >= 32) return;
        const unsigned full = 0xffffffffu;
        const int x = threadIdx.x & 7, p = x >> 2, t = x & 3;
        const double R = 0.125 * (S.zf[p][0][t] + S.zf[p][1][t]);
        const double c0 = S.z0[x], c1 = S.z1[x], h2 = A.h2[0], ih2 = A.ih2[0];
        double e;
        if (KIND != KPSI) {
            e = coarsest_exact<KIND>(-R, c0, h2);
        } else {
            // every neighbour along an axis is the same cell, counted twice
            auto nb = [&](double u) {
                return 2.0 * ((__shfl_xor_sync(full, u, 1) + __shfl_xor_sync(full, u, 2)) + __shfl_xor_sync(full, u, 4));
            };
            const double ur = 0.125 * (S.zu[p][0][t] + S.zu[p][1][t]);
            const double f = op64<KPSI>(nb(ur), ur, c0, c1, ih2, A.rho) - R;
            // Newton's method on the eight cells, each step solved exactly: the
            // coarse start is near the solution and the error squares per step
            // (three to four steps of 3 us; red-black sweeps contract by 9 and take 5 us each)
            double u = ur;
            bool done = false;
            for (int step = 0; step < 8 && !done; step++) {
                const double v = 1.0 + u, iv = recip64(v), iv2 = iv * iv, iv4 = iv2 * iv2, v2 = v * v, v4 = v2 * v2;
                const double m = fma(2.0 * kPi * c0, iv2, (0.875 * c1) * (iv4 * iv4)) + (10.0 * kPi * A.rho) * v4;
                const double d = coarsest_exact<KHELM>(f - op64<KPSI>(nb(u), u, c0, c1, ih2, A.rho), m, h2);
                u += d;
                // a step out of the positive conformal factors may end at a root beyond the pole at zero
                if (__any_sync(full, __double2hiint(1.0 + u) <= 0)) break;
                // the next step would move u by less than its rounding
                done = __all_sync(full, d * d <= 0x1p-56 * fabs(u) || d == 0.0);
            }
            if (!done) {  // far from the solution (one in a thousand of random strong defects): red-black Newton sweeps and the zero-mode shift, as k_coarsest
                const int color = __popc(x) & 1;
                u = ur;
                for (int sweep = 0; sweep < kCoarsestSweeps; sweep++) {
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        const double v = relax64<KPSI>(nb(u), u, f, c0, c1, h2, ih2, A.rho);
                        if (color == c) u = v;
                    }
                    const double v = 1.0 + u, iv = recip64(v), iv2 = iv * iv, iv4 = iv2 * iv2, v2 = v * v, v4 = v2 * v2;
                    double zr = f - op64<KPSI>(nb(u), u, c0, c1, ih2, A.rho);
                    double zm = fma(2.0 * kPi * c0, iv2, (0.875 * c1) * (iv4 * iv4)) + (10.0 * kPi * A.rho) * v4;
#pragma unroll
                    for (int b = 1; b < 8; b <<= 1) {
                        zr += __shfl_xor_sync(full, zr, b);
                        zm += __shfl_xor_sync(full, zm, b);
                    }
                    if (zm > 0.0) u -= zr / zm;
                }
            }
            e = u - ur;
        }
        if (threadIdx.x < 8) S.zb[x] = e;
        __syncwarp();
    }
};

template <int KIND>
__global__ void __launch_bounds__(kT64Threads) k_tail64(const T64Args A, int nu1, int nu2)
{
    pdl_begin();
    __shared__ T64Smem S;
    cg::cluster_group cl = cg::this_cluster();
    Tail64<KIND> T{S, A, (int)cl.block_rank(), cl};
    const int r = T.r;
    // coefficients of this CTA's plane of every level, u (with its halo) and f of the top level
    for (int l = 0; l <= A.top; l++) {
        const int n = 2 << l, nn = n * n, half = nn * n / 2, po = plane_off(l);
        if (r >= n) continue;
        for (int t = threadIdx.x; t < nn; t += kT64Threads) {
            const int j = t >> (l + 1), k = t & (n - 1);
            auto at = [&](int i) { return ((i + j + k) & 1) * half + (i * n + j) * (n / 2) + (k >> 1); };
            const int id = at(r);
            S.c0[po + t] = KIND == KPOISSON ? 0.0 : A.c0[l][id];
            S.c1[po + t] = KIND == KPOISSON ? 0.0 : A.c1[l][id];
            double *o = T.uo(l) + t;
            if (l < A.top) {  // the corrections start from zero (KPSI: from R u, set going down)
                o[0] = o[-nn] = o[nn] = 0.0;
            } else {
                o[0] = A.u[id];
                o[-nn] = A.u[at((r - 1) & (n - 1))];
                o[nn] = A.u[at((r + 1) & (n - 1))];
                S.f[po + t] = A.f[id];
            }
        }
    }
    if (r == 0 && threadIdx.x < 8) {
        const int x = threadIdx.x, i = x >> 2, j = (x >> 1) & 1, k = x & 1, id = 4 * ((i + j + k) & 1) + 2 * i + j;
        S.z0[x] = KIND == KPOISSON ? 0.0 : A.c0[0][id];
        S.z1[x] = KIND == KPSI ? A.c1[0][id] : 0.0;
    }
    cluster_barrier();  // every CTA runs and has read u before anyone's push
    for (int l = A.top; l >= 1; l--) {
        for (int s = 0; s < nu1; s++) {
            T.sweep(l, 0);
            T.sweep(l, 1);
        }
        T.down(l, KIND != KPSI && nu1 > 0);
    }
    T.coarsest();
    for (int l = 1; l <= A.top; l++) {
        T.up(l, KIND != KPSI && nu2 > 0);
        for (int s = 0; s < nu2; s++) {
            T.sweep(l, 0);
            T.sweep(l, 1);
        }
    }
    // the last barrier is behind every push: nothing remote is pending at exit
    const int n = 2 << A.top, nn = n * n, half = nn * n / 2;
    if (r < n)
        for (int t = threadIdx.x; t < nn; t += kT64Threads) {
            const int j = t / n, k = t & (n - 1);
            A.u[((r + j + k) & 1) * half + (r * n + j) * (n / 2) + (k >> 1)] = T.uo(A.top)[t];
        }
}

template <int KIND>
cudaLaunchConfig_t tail64_config(cudaStream_t st, cudaLaunchAttribute *at)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kT64Ctas);
    cfg.blockDim = dim3(kT64Threads);
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kT64Ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cfg;
}

// once per kind and device: the 16-CTA cluster (beyond the portable 8) is allowed and fits the device
template <int KIND>
bool tail64_usable()
{
    return per_device([] {
        auto k = k_tail64<KIND>;
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t cfg = tail64_config<KIND>(nullptr, at);
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&nc, (const void *)k, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        return nc >= 1;
    });
}

template <int KIND>
void launch_tail64(const T64Args &a, int nu1, int nu2, cudaStream_t st)
{
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = tail64_config<KIND>(st, at);
    if (cudaLaunchKernelEx(&cfg, k_tail64<KIND>, a, nu1, nu2) != cudaSuccess) {
        cudaGetLastError();  // without programmatic serialization; an error of this launch stays recorded
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, k_tail64<KIND>, a, nu1, nu2);
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
}

}  // namespace

bool tail64_ok(int kind)
{
    if (kind == KPOISSON) return tail64_usable<KPOISSON>();
    if (kind == KHELM) return tail64_usable<KHELM>();
    return tail64_usable<KPSI>();
}

void tail64(int kind, int top, double *u, const double *f, const double *const *c0, const double *const *c1,
            const double *h2, const double *ih2, double rho, int nu1, int nu2, cudaStream_t st)
{
    T64Args a;
    a.u = u;
    a.f = f;
    for (int l = 0; l <= 3; l++) {
        const int q = l <= top ? l : 0;
        a.c0[l] = c0[q];
        a.c1[l] = c1[q];
        a.h2[l] = h2[q];
        a.ih2[l] = ih2[q];
    }
    a.rho = rho;
    a.top = top;
    if (kind == KPOISSON) launch_tail64<KPOISSON>(a, nu1, nu2, st);
    else if (kind == KHELM) launch_tail64<KHELM>(a, nu1, nu2, st);
    else launch_tail64<KPSI>(a, nu1, nu2, st);
}

}  // namespace gr
