// line3.cuh -- the D1Q3 lattice of the paper's own simulations (Sec. 4): velocities
// v = 0, +1, -1, weights 2/3, 1/6, 1/6, one periodic line of nx sites.
//
// The same timestep as the D2Q9 kernels (Eq. ssLB with the Eq. definef force, Eq. lgf
// potentials, Sec. 3 equilibria, Eqs. ff1-ff3 forcing) with the discrete operators
// built from the D1Q3 weights: grad g = (g(x+1) - g(x-1)) / 2, lap g = g(x+1) + g(x-1)
// - 2 g(x).  Storage: post-collision values f*[(s * 3 + i) * nx + x] (pull scheme: the
// pre-collision population f_i(x) is the value stored at x - v_i), FP64 or FP32.
//
// Two schedules:
//   - k_line3_resident: one CTA owns a whole line (nx <= L3_MAX_SITES, one site per
//     thread) and advances it by K steps in shared memory before writing it back, so a
//     line crosses HBM once per launch instead of once per step.  A batch launches one
//     CTA per line (every line of the same N in one launch).  Three CTA barriers per
//     step, no other waits.  FP64 lines whose N threads per site fit a cluster take
//     k_line3_resident64 instead.
//   - k_line3_tile: one launch per step for longer lines; a CTA pulls L3_TILE sites
//     (252 written, two halo sites on each side for the radius-2 stencil of the force).
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "log64.cuh"
#include "staged.cuh"

namespace mclb {

constexpr int L3_MAX_SITES = 1024;  // longest line the resident kernel holds
constexpr int L3_TILE = 256;        // threads (sites) of a tile CTA, 4 of them halo
constexpr int L3_CHUNK = LINE3_CHUNK;  // most steps one resident launch advances

__host__ __device__ __forceinline__ constexpr int v3(int i) { return i == 0 ? 0 : (i == 1 ? 1 : -1); }

// D1Q3 weights; in FP32 w_+- is one unit in the last place below the float nearest to
// 1/6 (11184810 * 2^-26), so that 2/3 rounded plus twice it is exactly 1 (the nearest
// floats sum to 1 + 3e-8, a mass drift of that size per step).
template <typename C>
__host__ __device__ __forceinline__ constexpr C w3(int i)
{
    return i == 0 ? C(2.0 / 3.0) : C(1.0 / 6.0);
}
template <>
__host__ __device__ __forceinline__ constexpr float w3<float>(int i)
{
    return i == 0 ? float(2.0 / 3.0) : 11184810.0f * 0x1p-26f;
}

__device__ __forceinline__ int wrap1(int a, int n)
{
    a %= n;
    return a < 0 ? a + n : a;
}

// Post-collision populations of one component at one site: f (1 - 1/tau) + (rho^s/tau)
// w_i (1 + 3 v u + 9/2 v^2 u^2 - 3/2 u^2) + w_i (3 rho^s v a + 9 v^2 a j - 3 a j), with
// the constant w_i rho^s/tau carried in the forcing bracket so that 1 - 3/2 u^2 is never
// rounded (that rounding biases the FP32 masses).
template <typename C>
__device__ __forceinline__ void collide3(const StepParams<C>& p, const C (&f)[3], C r, C j, C u,
                                         C a, C (&out)[3])
{
    const C keep = C(1) - p.omega, omr = p.omega * r;
    if constexpr (std::is_same<C, double>::value) {
        // the same polynomial by its even and odd parts, 16 operations instead of 36 (the
        // FP64 pipe bounds these lines): with q = rho^s/tau u^2 + 2 a j,
        //   w_0 [rho^s/tau - 1.5 q],  w_+- [rho^s/tau + 3 q +- 3 (rho^s/tau u + rho^s a)]
        const C ou = omr * u;
        const C q = fma(C(2), a * j, ou * u);
        const C odd = C(0.5) * fma(r, a, ou);
        const C even = fma(C(0.5), q, C(1.0 / 6.0) * omr);
        out[0] = fma(keep, f[0], fma(C(2.0 / 3.0), omr, -q));
        out[1] = fma(keep, f[1], even + odd);
        out[2] = fma(keep, f[2], even - odd);
        return;
    }
    const C base = C(-1.5) * u * u;
    const C uu45 = C(4.5) * u * u;
    const C m3aj = C(-3) * a * j + omr;
    const C e0 = w3<C>(0) * base;
    const C ep = w3<C>(1) * (base + uu45 + C(3) * u);
    const C em = w3<C>(2) * (base + uu45 - C(3) * u);
    const C ar3 = C(3) * r * a, aj9 = C(9) * a * j;
    const C F0 = w3<C>(0) * m3aj;
    const C Fp = w3<C>(1) * (ar3 + aj9 + m3aj);
    const C Fm = w3<C>(2) * (-ar3 + aj9 + m3aj);
    out[0] = keep * f[0] + (omr * e0 + F0);
    out[1] = keep * f[1] + (omr * ep + Fp);
    out[2] = keep * f[2] + (omr * em + Fm);
}

// rho^s of component s at site x (pull of the three populations).
template <typename T>
__device__ __forceinline__ typename Storage<T>::C pull_rho3(const T* __restrict__ f, int nx, int s,
                                                            int x)
{
    using C = typename Storage<T>::C;
    C r = C(0);
#pragma unroll
    for (int i = 0; i < 3; ++i) r += C(f[(long long)(s * 3 + i) * nx + wrap1(x - v3(i), nx)]);
    return r;
}

// nu^s at site x from rho^s at x - 1, x, x + 1 (each rho array holds all N components).
template <typename C, int N>
__device__ __forceinline__ void nu3(const StepParams<C>& p, const C (&rl)[N], const C (&rc)[N],
                                    const C (&rr)[N], C (&nu)[N])
{
    C lap[N];
#pragma unroll
    for (int s = 0; s < N; ++s) lap[s] = (rr[s] + rl[s]) - C(2) * rc[s];
    site_nu<C, N>(p, rc, lap, nu);
}

// Gibbs-Duhem reading of the sum of the component forces (kappa = 0) on D1Q3: every a^s
// shifted by (A_c - A) / rho, A = sum_s rho^s (a^s - g), A_c = (1 - 1/(2 tau)) (1/3) d_x rho.
template <typename C, int N>
__device__ __forceinline__ void gibbs_duhem3(const StepParams<C>& p, const C (&r)[N], C rho,
                                             C grad_rho, C (&a)[N])
{
    C A = C(0);
#pragma unroll
    for (int s = 0; s < N; ++s) A += r[s] * (a[s] - p.gx);
    const C d = (p.fcoef * grad_rho / C(3) - A) / rho;
#pragma unroll
    for (int s = 0; s < N; ++s) a[s] += d;
}

// One instance of a resident launch: buffers and parameters.
template <typename T>
struct Line3Item {
    StepParams<typename Storage<T>::C> p;
    T* f[2];
};

template <typename T, int N>
struct Line3Smem {
    using C = typename Storage<T>::C;
    // per site: 3N post-collision populations, N densities, N potentials
    static constexpr size_t bytes(int nx) { return (size_t)(5 * N) * nx * sizeof(C); }
    // FP64, one thread per site and component: also N momenta, the total density and four
    // per-site terms, and the neighbours' values beyond a piece's ends
    static constexpr size_t bytes64(int n) { return (size_t)((6 * N + 5) * n + 6 * N + 2) * sizeof(C); }
};

// FP32: K steps of one line per CTA, one thread per site.
// Reads items[b].f[parity], writes items[b].f[parity ^ 1].  blockDim.x >= the longest nx of the launch.
template <typename T, int N>
__global__ void __launch_bounds__(L3_MAX_SITES)
k_line3_resident(const Line3Item<T>* __restrict__ items, int parity, int nsteps)
{
    using C = typename Storage<T>::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ StepParams<C> p;
    if (threadIdx.x == 0) p = items[blockIdx.x].p;
    __syncthreads();
    const int nx = p.nx;
    C* A = reinterpret_cast<C*>(smem_raw);  // [3N][nx] post-collision
    C* R = A + 3 * N * nx;                  // [N][nx]
    C* NU = R + N * nx;                     // [N][nx]
    const T* fin = items[blockIdx.x].f[parity];
    T* fout = items[blockIdx.x].f[parity ^ 1];
    for (int k = threadIdx.x; k < 3 * N * nx; k += blockDim.x) A[k] = C(fin[k]);
    __syncthreads();
    const int x = threadIdx.x;
    const bool act = x < nx;
    const int xl = act ? wrap1(x - 1, nx) : 0, xr = act ? wrap1(x + 1, nx) : 0;
    bool bad = false;
    for (int t = 0; t < nsteps; ++t) {
        C f[N][3], r[N], j[N];
        C u = C(0);
        if (act) {
            C rho = C(0), jt = C(0);
#pragma unroll
            for (int s = 0; s < N; ++s) {
                f[s][0] = A[(s * 3 + 0) * nx + x];
                f[s][1] = A[(s * 3 + 1) * nx + xl];
                f[s][2] = A[(s * 3 + 2) * nx + xr];
                r[s] = (f[s][0] + f[s][1]) + f[s][2];
                j[s] = f[s][1] - f[s][2];
                rho += r[s];
                jt += j[s];
                R[s * nx + x] = r[s];
            }
            u = jt / rho;
            bad = bad || !(rho > C(0)) || !isfinite(rho);
        }
        __syncthreads();
        if (act) {
            C rl[N], rc[N], rr[N], nu[N];
#pragma unroll
            for (int s = 0; s < N; ++s) {
                rl[s] = R[s * nx + xl];
                rc[s] = R[s * nx + x];
                rr[s] = R[s * nx + xr];
            }
            nu3<C, N>(p, rl, rc, rr, nu);
#pragma unroll
            for (int s = 0; s < N; ++s) NU[s * nx + x] = nu[s];
        }
        __syncthreads();
        if (act) {
            C a[N], rho = C(0);
#pragma unroll
            for (int s = 0; s < N; ++s) {
                a[s] = -p.fcoef * (C(0.5) * (NU[s * nx + xr] - NU[s * nx + xl])) + p.gx;
                rho += r[s];
            }
            if (p.gd) {
                C rl = C(0), rr = C(0);
#pragma unroll
                for (int s = 0; s < N; ++s) {
                    rl += R[s * nx + xl];
                    rr += R[s * nx + xr];
                }
                gibbs_duhem3<C, N>(p, r, rho, C(0.5) * (rr - rl), a);
            }
#pragma unroll
            for (int s = 0; s < N; ++s) {
                const C jf = p.bary ? r[s] * u : j[s];
                C out[3];
                collide3(p, f[s], r[s], jf, u, a[s], out);
#pragma unroll
                for (int i = 0; i < 3; ++i) A[(s * 3 + i) * nx + x] = out[i];
            }
        }
        __syncthreads();
    }
    if (bad) atomicOr(p.status, STATUS_NONFINITE);
    for (int k = threadIdx.x; k < 3 * N * nx; k += blockDim.x) fout[k] = T(A[k]);
}

// FP64: K steps of one line per CTA or, where SMs would idle, per cluster of CTAs that cut the
// line into pieces; one thread per site and component (thread t: site t mod stride, component
// t / stride).
//
// The FP64 pipe bounds it: one warp instruction per 64 cycles and SM quarter, however many of
// the 32 lanes are active, so a step costs the FP64 instructions of the busiest quarter.  A
// site's step is therefore spread over its N threads and written short: collide3's even and odd
// parts (16 where 36), one reciprocal (two divisions before), log64 (13 for 29), the sums over
// phi formed from rho^s and scaled once, without the constants of nu^s, which have no gradient.  With one thread per site the busiest quarter ran
// about 180 instructions a step (N = 2), now about 50.  60 lines of 128 sites, N = 2:
// 5.71 -> 2.66 us a step (a CTA pair per line); 512 of 600: 98 -> 62; 10 of 600, N = 3: 38.5 -> 5.1.
//
// Arrays carry the neighbouring site's value beyond the ends of a piece; the thread that owns an
// end site also stores there, in the neighbouring piece's shared memory (its own where the
// line is one piece).  A step:
//   pull, rho^s, j^s                       | barrier (CTA; cluster where kappa != 0)
//   ln rho, 1/rho and what follows from it | barrier (CTA)
//   nu^s                                   | barrier (cluster)
//   a^s, collision                         | barrier (cluster)
template <int N>
__global__ void __launch_bounds__(L3_MAX_SITES)
k_line3_resident64(const Line3Item<double>* __restrict__ items, int parity, int nsteps, int stride)
{
    using C = double;
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ StepParams<C> p;
    __shared__ Log64Row tab[LOG64_ROWS];
    const cg::cluster_group cl = cg::this_cluster();
    const int pieces = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const Line3Item<double>& item = items[blockIdx.x / pieces];
    {
        static_assert(sizeof(StepParams<C>) % sizeof(int) == 0, "parameter copy by words");
        const int* src = reinterpret_cast<const int*>(&item.p);
        for (int k = threadIdx.x; k < (int)(sizeof(StepParams<C>) / sizeof(int)); k += blockDim.x)
            reinterpret_cast<int*>(&p)[k] = src[k];
    }
    log64_load(tab);
    __syncthreads();
    const int nx = p.nx;
    const auto start = [&](int k) { return (int)((long long)nx * k / pieces); };
    const int x0 = start(rank), n = start(rank + 1) - x0;
    const bool lap = p.kappa != 0.0;
    // [N]: f*_0 at 0 .. n - 1, f*_+ with the left neighbour's before it, f*_- with the right
    // neighbour's after it; nu^s and rho^s with both; the Gibbs-Duhem form's total density with
    // both; per site j^s, theta/rho, u, ln rho and the components' common part of nu^s
    struct Arrays {
        int n;
        C* a;
        __device__ C* f0(int s) const { return a + s * (3 * n + 2); }
        __device__ C* fp(int s) const { return f0(s) + n + 1; }        // fp(s)[-1]: left neighbour's
        __device__ C* fm(int s) const { return f0(s) + 2 * n + 1; }    // fm(s)[n]: right neighbour's
        __device__ C* nu(int s) const { return a + N * (3 * n + 2) + s * (n + 2) + 1; }
        __device__ C* rho(int s) const { return nu(N + s); }
        __device__ C* total() const { return nu(2 * N); }
        __device__ C* j(int s) const { return a + N * (3 * n + 2) + (2 * N + 1) * (n + 2) + s * n; }
        __device__ C* site(int q) const { return j(N + q); }
    };
    const int rl = rank == 0 ? pieces - 1 : rank - 1, rr = rank == pieces - 1 ? 0 : rank + 1;
    C* base = reinterpret_cast<C*>(smem_raw);
    const Arrays me{n, base}, left{start(rl + 1) - start(rl), cl.map_shared_rank(base, rl)},
        right{start(rr + 1) - start(rr), cl.map_shared_rank(base, rr)};
    const auto sync = [&]() {
        if (pieces == 1)
            __syncthreads();
        else
            cl.sync();
    };
    const int s = (int)threadIdx.x / stride, l = (int)threadIdx.x - s * stride, x = x0 + l;
    const bool act = s < N && l < n, first = act && l == 0, last = act && l == n - 1;
    const C* fin = item.f[parity];
    C* fout = item.f[parity ^ 1];
    if (act) {
        const C* g = fin + (long long)s * 3 * nx;
        me.f0(s)[l] = g[x];
        me.fp(s)[l] = g[nx + x];
        me.fm(s)[l] = g[2 * nx + x];
        if (first) me.fp(s)[-1] = g[nx + wrap1(x - 1, nx)];
        if (last) me.fm(s)[n] = g[2 * nx + wrap1(x + 1, nx)];
    }
    sync();   // (also: every CTA of the cluster runs before the first store to a neighbour)
    bool bad = false;
    const C k05 = -0.5 * p.fcoef;
    const bool own_log = act && ((p.log_mask >> s) & 1u);
    // ln rho by the first component without a logarithm of its own (else the last), the rest of
    // the site's terms by another one
    const int free_s = __ffs(~p.log_mask & ((1u << N) - 1u));
    const int s_log = free_s > 0 ? free_s - 1 : N - 1, s_inv = N == 1 ? 0 : (s_log == N - 1 ? N - 2 : N - 1);
    for (int t = 0; t < nsteps; ++t) {
        C f[3] = {0.0, 0.0, 0.0}, r = 0.0, j = 0.0;
        if (act) {
            f[0] = me.f0(s)[l];
            f[1] = me.fp(s)[l - 1];
            f[2] = me.fm(s)[l + 1];
            r = (f[0] + f[1]) + f[2];
            j = f[1] - f[2];
            me.rho(s)[l] = r;
            me.j(s)[l] = j;
            if (lap) {
                if (first) left.rho(s)[left.n] = r;
                if (last) right.rho(s)[-1] = r;
            }
        }
        if (lap)
            sync();
        else
            __syncthreads();
        C mine = 0.0;   // (theta/m^s - 1/3) ln rho^s
        if (act) {
            C rt[N], rho = 0.0;
#pragma unroll
            for (int q = 0; q < N; ++q) {
                rt[q] = me.rho(q)[l];
                rho += rt[q];
            }
            if (s == s_log) me.site(2)[l] = log64(rho, tab);
            if (s == s_inv) {
                C jt = 0.0, sm = 0.0, quad = 0.0;
#pragma unroll
                for (int q = 0; q < N; ++q) {
                    C c = 0.0;
#pragma unroll
                    for (int w = 0; w < N; ++w) c += p.chi[q * N + w] * rt[w];
                    jt += me.j(q)[l];
                    sm += rt[q] * p.dm[q];
                    quad += rt[q] * c;
                }
                const C inv = 1.0 / rho, ti = p.theta * inv;
                me.site(0)[l] = ti;
                me.site(1)[l] = jt * inv;
                me.site(3)[l] = -ti * fma(0.5 * quad, inv, sm);
                bad = bad || !(rho > 0.0) || !isfinite(rho);
                if (p.gd) {
                    me.total()[l] = rho;
                    if (first) left.total()[left.n] = rho;
                    if (last) right.total()[-1] = rho;
                }
            }
            if (own_log) {
                const C fl = p.log_floor * rho;
                mine = p.logc[s] * log64(r > fl ? r : fl, tab);
            }
        }
        __syncthreads();
        if (act) {
            C c = 0.0;
#pragma unroll
            for (int w = 0; w < N; ++w) c += p.chi[s * N + w] * me.rho(w)[l];
            C nu = fma(-p.th_m[s], me.site(2)[l], fma(me.site(0)[l], c, me.site(3)[l])) + mine;
            if (lap) nu -= p.kappa * ((me.rho(s)[l + 1] + me.rho(s)[l - 1]) - 2.0 * r);
            me.nu(s)[l] = nu;
            if (first) left.nu(s)[left.n] = nu;
            if (last) right.nu(s)[-1] = nu;
        }
        sync();
        if (act) {
            const C u = me.site(1)[l];
            C a = fma(k05, me.nu(s)[l + 1] - me.nu(s)[l - 1], p.gx);
            if (p.gd) {
                // the common shift of gibbs_duhem3: (A_c - A)/rho with A = sum_s rho^s (a^s - g)
                C A = 0.0;
#pragma unroll
                for (int q = 0; q < N; ++q) A += me.rho(q)[l] * (me.nu(q)[l + 1] - me.nu(q)[l - 1]);
                const C k3 = p.fcoef * (0.5 / 3.0);
                a += fma(k3, me.total()[l + 1] - me.total()[l - 1], -k05 * A) / me.total()[l];
            }
            C out[3];
            collide3(p, f, r, p.bary ? r * u : j, u, a, out);
            me.f0(s)[l] = out[0];
            me.fp(s)[l] = out[1];
            me.fm(s)[l] = out[2];
            if (last) right.fp(s)[-1] = out[1];
            if (first) left.fm(s)[left.n] = out[2];
        }
        sync();
    }
    if (bad) atomicOr(p.status, STATUS_NONFINITE);
    if (act) {
        C* g = fout + (long long)s * 3 * nx;
        g[x] = me.f0(s)[l];
        g[nx + x] = me.fp(s)[l];
        g[2 * nx + x] = me.fm(s)[l];
    }
}

// One step of a line of any length: CTA b covers written sites [x0, x0 + L3_TILE - 4),
// thread t the site x0 - 2 + t (indices wrap, so lines shorter than a tile work too).
template <typename T, int N>
__global__ void __launch_bounds__(L3_TILE)
k_line3_tile(const T* __restrict__ fin, T* __restrict__ fout,
             const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    using C = typename Storage<T>::C;
    __shared__ C R[N][L3_TILE];
    __shared__ C NU[N][L3_TILE];
    const int nx = p.nx;
    const int t = threadIdx.x;
    const int x0 = blockIdx.x * (L3_TILE - 4);
    const int x = wrap1(x0 - 2 + t, nx);
    C f[N][3], r[N], j[N];
    C rho = C(0), jt = C(0);
#pragma unroll
    for (int s = 0; s < N; ++s) {
#pragma unroll
        for (int i = 0; i < 3; ++i) f[s][i] = C(fin[(long long)(s * 3 + i) * nx + wrap1(x - v3(i), nx)]);
        r[s] = (f[s][0] + f[s][1]) + f[s][2];
        j[s] = f[s][1] - f[s][2];
        rho += r[s];
        jt += j[s];
        R[s][t] = r[s];
    }
    const C u = jt / rho;
    __syncthreads();
    if (t >= 1 && t < L3_TILE - 1) {
        C rl[N], rc[N], rr[N], nu[N];
#pragma unroll
        for (int s = 0; s < N; ++s) {
            rl[s] = R[s][t - 1];
            rc[s] = r[s];
            rr[s] = R[s][t + 1];
        }
        nu3<C, N>(p, rl, rc, rr, nu);
#pragma unroll
        for (int s = 0; s < N; ++s) NU[s][t] = nu[s];
    }
    __syncthreads();
    const int xo = x0 - 2 + t;
    if (t >= 2 && t < L3_TILE - 2 && xo < nx) {
        if (!(rho > C(0)) || !isfinite(rho)) atomicOr(p.status, STATUS_NONFINITE);
        C a[N];
#pragma unroll
        for (int s = 0; s < N; ++s) a[s] = -p.fcoef * (C(0.5) * (NU[s][t + 1] - NU[s][t - 1])) + p.gx;
        if (p.gd) {
            C rl = C(0), rr = C(0);
#pragma unroll
            for (int s = 0; s < N; ++s) {
                rl += R[s][t - 1];
                rr += R[s][t + 1];
            }
            gibbs_duhem3<C, N>(p, r, rho, C(0.5) * (rr - rl), a);
        }
#pragma unroll
        for (int s = 0; s < N; ++s) {
            const C jf = p.bary ? r[s] * u : j[s];
            C out[3];
            collide3(p, f[s], r[s], jf, u, a[s], out);
#pragma unroll
            for (int i = 0; i < 3; ++i) fout[(long long)(s * 3 + i) * nx + xo] = T(out[i]);
        }
    }
}

// f*_i(x) such that the pull at x + v_i yields f^e_i(rho(x + v_i), u(x + v_i)).
template <typename T, int N>
__global__ void __launch_bounds__(SITE_THREADS)
k_line3_init(const double* __restrict__ rho, const double* __restrict__ u, T* __restrict__ f,
             const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    using C = typename Storage<T>::C;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= p.nx) return;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int xs = wrap1(x + v3(i), p.nx);
        const C uu = u ? C(u[xs]) : C(0);
        const C cu = C(v3(i)) * uu;
#pragma unroll
        for (int s = 0; s < N; ++s)
            f[(long long)(s * 3 + i) * p.nx + x] =
                T(w3<C>(i) * C(rho[(long long)s * p.nx + xs]) *
                  (C(1) + C(3) * cu + C(4.5) * cu * cu - C(1.5) * uu * uu));
    }
}

template <typename T, int N>
__global__ void __launch_bounds__(SITE_THREADS)
k_line3_get_state(const T* __restrict__ f, double* __restrict__ out,
                  const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= p.nx) return;
#pragma unroll
    for (int s = 0; s < N; ++s)
#pragma unroll
        for (int i = 0; i < 3; ++i)
            out[(long long)(s * 3 + i) * p.nx + x] =
                (double)f[(long long)(s * 3 + i) * p.nx + wrap1(x - v3(i), p.nx)];
}

template <typename T, int N>
__global__ void __launch_bounds__(SITE_THREADS)
k_line3_set_state(const double* __restrict__ in, T* __restrict__ f,
                  const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= p.nx) return;
#pragma unroll
    for (int s = 0; s < N; ++s)
#pragma unroll
        for (int i = 0; i < 3; ++i)
            f[(long long)(s * 3 + i) * p.nx + x] =
                T(in[(long long)(s * 3 + i) * p.nx + wrap1(x + v3(i), p.nx)]);
}

// rho^s at x - 2 .. x + 2, nu^s at x - 1 .. x + 1 and the site's own moments.
template <typename T, int N>
struct Line3Site {
    using C = typename Storage<T>::C;
    C r[5][N];
    C nu[3][N];
    C j[N];
    C rho, u;
    __device__ __forceinline__ Line3Site(const T* __restrict__ f, const StepParams<C>& p, int x)
    {
#pragma unroll
        for (int d = 0; d < 5; ++d)
#pragma unroll
            for (int s = 0; s < N; ++s) r[d][s] = pull_rho3(f, p.nx, s, x - 2 + d);
#pragma unroll
        for (int d = 0; d < 3; ++d) nu3<C, N>(p, r[d], r[d + 1], r[d + 2], nu[d]);
        rho = C(0);
        C jt = C(0);
#pragma unroll
        for (int s = 0; s < N; ++s) {
            j[s] = C(f[(long long)(s * 3 + 1) * p.nx + wrap1(x - 1, p.nx)]) -
                   C(f[(long long)(s * 3 + 2) * p.nx + wrap1(x + 1, p.nx)]);
            rho += r[2][s];
            jt += j[s];
        }
        u = jt / rho;
        // Gibbs-Duhem reading: the common shift of every a^s
        shift = C(0);
        if (p.gd) {
            C A = C(0), rl = C(0), rr = C(0);
#pragma unroll
            for (int s = 0; s < N; ++s) {
                A += r[2][s] * (-p.fcoef * (C(0.5) * (nu[2][s] - nu[0][s])));
                rl += r[1][s];
                rr += r[3][s];
            }
            shift = (p.fcoef * (C(0.5) * (rr - rl)) / C(3) - A) / rho;
        }
    }
    C shift;
    __device__ __forceinline__ C accel(const StepParams<C>& p, int s) const
    {
        return -p.fcoef * (C(0.5) * (nu[2][s] - nu[0][s])) + p.gx + shift;
    }
};

// Output fields in the shapes of a D2Q9 lattice with ny = 1: rho^s; U = (u + a/2, 0);
// mu^s/m^s with the gradient term; P = (iso + kappa sum (d_x rho)^2, 0, iso).
template <typename T, int N>
__global__ void __launch_bounds__(SITE_THREADS)
k_line3_moments(const T* __restrict__ f, double* __restrict__ rho_out, double* __restrict__ U,
                double* __restrict__ mu_out, double* __restrict__ P,
                const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    using C = typename Storage<T>::C;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= p.nx) return;
    const Line3Site<T, N> q(f, p, x);
    const int nx = p.nx;
    if (rho_out)
#pragma unroll
        for (int s = 0; s < N; ++s) rho_out[(long long)s * nx + x] = (double)q.r[2][s];
    if (U) {
        C fx = C(0);
#pragma unroll
        for (int s = 0; s < N; ++s) fx += q.r[2][s] * q.accel(p, s);
        U[x] = (double)(q.u + C(0.5) * fx / q.rho);
        U[nx + x] = 0.0;
    }
    if (mu_out || P) {
        C lap[N], mu[N];
#pragma unroll
        for (int s = 0; s < N; ++s) lap[s] = (q.r[3][s] + q.r[1][s]) - C(2) * q.r[2][s];
        site_mu<C, N>(p, q.r[2], lap, mu);
        if (mu_out)
#pragma unroll
            for (int s = 0; s < N; ++s) mu_out[(long long)s * nx + x] = (double)mu[s];
        if (P) {
            const C psi = site_psi<C, N>(p, q.r[2]);
            C rmu = C(0), gg = C(0), pxx = C(0);
#pragma unroll
            for (int s = 0; s < N; ++s) {
                const C gx = C(0.5) * (q.r[3][s] - q.r[1][s]);
                rmu += q.r[2][s] * mu[s];
                gg += C(0.5) * p.kappa * gx * gx;
                pxx += p.kappa * gx * gx;
            }
            const C iso = rmu - (psi + gg);
            P[x] = (double)(iso + pxx);
            P[nx + x] = 0.0;
            P[2 * nx + x] = (double)iso;
        }
    }
}

// Conservation sums (FP64, fixed-grid block partials): mass^s, momentum (x, 0), force (x, 0).
template <typename T, int N>
__global__ void __launch_bounds__(SITE_THREADS)
k_line3_conservation(const T* __restrict__ f, double* __restrict__ partial,
                     const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    constexpr int K = N + 4;
    double acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < p.nx; x += gridDim.x * blockDim.x) {
        const Line3Site<T, N> q(f, p, x);
#pragma unroll
        for (int s = 0; s < N; ++s) {
            acc[s] += (double)q.r[2][s];
            acc[N] += (double)q.j[s];
            acc[N + 2] += (double)q.r[2][s] * (double)q.accel(p, s);
        }
    }
    block_reduce_store<K>(acc, partial);
}

// FP64 compositions and bulk flags (|d_x phi^s| < tol for every s).
template <typename T, int N>
__global__ void __launch_bounds__(SITE_THREADS)
k_line3_compositions(const T* __restrict__ f, double* __restrict__ phi, double* __restrict__ bulk,
                     double tol, const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= p.nx) return;
    double ph[3][N];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double rho = 0.0, r[N];
#pragma unroll
        for (int s = 0; s < N; ++s) {
            r[s] = (double)pull_rho3(f, p.nx, s, x - 1 + d);
            rho += r[s];
        }
#pragma unroll
        for (int s = 0; s < N; ++s) ph[d][s] = r[s] / rho;
    }
    double gmax = 0.0;
#pragma unroll
    for (int s = 0; s < N; ++s) {
        phi[(long long)s * p.nx + x] = ph[1][s];
        const double g = fabs(0.5 * (ph[2][s] - ph[0][s]));
        gmax = g > gmax ? g : gmax;
    }
    bulk[x] = gmax < tol ? 1.0 : 0.0;
}

}  // namespace mclb
