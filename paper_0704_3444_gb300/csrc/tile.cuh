// tile.cuh -- one launch per timestep by small tiles: the schedule of lattices too small to
// fill the GPU with the column march.
//
// A CTA owns TX x TY sites and computes everything their new state needs from the stored
// populations: rho^s on the tile and two rows and columns around it (the pull of Eq. ssLB),
// nu^s on the tile and one around it (Eq. lgf with -kappa lap rho^s and -(1/3) ln rho^s),
// then the collision on the tile (Eq. definef, Eqs. ff1-ff3).  rho^s, j^s, nu^s and u of the
// tile live in shared memory; nothing else is written to memory but the new populations,
// ghost columns included.  Thread t owns site t mod SITES and component t / SITES: one
// component's nine values per thread, so N warps share a site's work and the longest chain
// of a step is short.
//
// What bounds it: on these lattices neither memory nor arithmetic but latency -- one round
// trip to L2 for the pulls, two CTA barriers, one logarithm and one division, the launch.
// The march spends (segment rows + 4) dependent row iterations on the same step and runs on
// few SMs.  FP32 and FP64; the 16-bit formats have tile16.cuh.
#pragma once

#include "log64.cuh"
#include "tma.cuh"

namespace mclb {

// Threads per CTA and registers per thread at most: 56 registers, and 80 in FP64
// up to four components, keep two to three CTAs
// of 16 x 8 sites on an SM (uncapped the compiler takes 72 and 128: 1000 x 333 x 3 FP32
// 31.6 -> 26.9 us, 512 x 512 x 2 FP64 188 -> 171 us).
template <typename T>
constexpr int tile_max_threads() { return sizeof(typename Storage<T>::C) == 8 ? 512 : 768; }
template <typename T>
constexpr int tile_max_regs(int n) { return sizeof(typename Storage<T>::C) == 8 ? (n <= 4 ? 80 : 128) : 56; }

// Components up to which the tiles have the Gibbs-Duhem form (as the march, whose place they take)
constexpr int TILE_GD_NMAX = 3;

// Shared memory of one CTA in values of C: rho^s, nu^s, j^s, u and (Gibbs-Duhem) rho, 1/rho, a^s.
__host__ __device__ constexpr int tile_smem_values(int n, int tx, int ty, bool gd)
{
    return n * (tx + 4) * (ty + 4) + n * (tx + 2) * (ty + 2) + 2 * n * tx * ty + 2 * tx * ty +
           (gd ? (tx + 2) * (ty + 2) + tx * ty + 2 * n * tx * ty : 0);
}

// a mod n, for any a (one conditional step when a is within n of the range)
__device__ __forceinline__ int wrap_any(int a, int n)
{
    a += a < 0 ? n : 0;
    a -= a >= n ? n : 0;
    if (a < 0 || a >= n) {
        a %= n;
        a += a < 0 ? n : 0;
    }
    return a;
}

// The nine pulled values of component s at column x, -2 <= x <= nx + 1 (the ghost columns
// make the columns beyond the lattice plain addresses), and row y of the lattice.  Offsets
// are 32 bits from the nine lines' uniform bases (the buffer holds fewer than 2^31 values).
// Between walls the value of a link that crosses one is the site's own of the opposite
// velocity; the choice is made on the offset, so the nine loads stay independent of it.
template <typename T, typename C>
__device__ __forceinline__ void tile_pull(const T* __restrict__ f, const StepParams<C>& p, int s, int x,
                                          int y, C (&v)[Q])
{
    const unsigned pitch = (unsigned)p.pitch;
    unsigned rl[3];   // rows y - 1, y, y + 1 of the component
    rl[0] = (unsigned)(s * p.ny + (y == 0 ? p.ny - 1 : y - 1));
    rl[1] = (unsigned)(s * p.ny + y);
    rl[2] = (unsigned)(s * p.ny + (y == p.ny - 1 ? 0 : y + 1));
    const unsigned col = (unsigned)(p.hx + x);
    auto value = [&](int i, const T* line, unsigned row, unsigned c) {
        C r = Storage<T>::load(line + (row * (Q * pitch) + c));
        if constexpr (Storage<T>::shifted)
            r = fma(wq<C>(i),
                    __ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(f) + p.rbytes) +
                          (row * pitch + c)),
                    r);
        return r;
    };
    if (!p.walls) {
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = value(i, f + i * pitch, rl[1 - vy(i)], col - vx(i));
    } else {
        const bool lo = y == 0, hi = y == p.ny - 1;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const bool b = vy(i) > 0 ? lo : (vy(i) < 0 ? hi : false);
            v[i] = value(i, f + (b ? opp9(i) : i) * pitch, b ? rl[1] : rl[1 - vy(i)], b ? col : col - vx(i));
        }
    }
}

template <typename C>
__device__ __forceinline__ C sum9(const C (&v)[Q])
{
    return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])) + v[8];
}

// Post-collision values of one component (the polynomial of collide(), physics.cuh, by its
// coefficients): with L = 3 (rho^s u/tau + rho^s a), Cxx = rho^s/tau 4.5 ux^2 + 9 ax jx, Cyy
// alike and Cxy = rho^s/tau 9 ux uy + 9 (ax jy + ay jx),
//   f*_i = (1 - 1/tau) f_i + w_i [rho^s/tau - (Cxx + Cyy)/3 + L.v + C:vv],
// whose parts even and odd in v serve two opposite velocities at once: 57 operations where
// the direction-by-direction form takes 45 plus 36 for the site's e_i, which here every
// component's thread would form again.  The constant w_i rho^s/tau enters last (see eq_weights
// on why it is not rounded together with the velocity terms; summed with them first, 9
// operations fewer, the error of U on 64 x 64 FP64 grew from 2.2e-15 to 3.3e-15).
template <typename C>
__device__ __forceinline__ void collide_poly(const StepParams<C>& p, const C (&f)[Q], C r, C jx, C jy,
                                             C ux, C uy, C ax, C ay, C (&out)[Q])
{
    const C omr = p.omega * r, keep = C(1) - p.omega;
    const C lx = C(3) * fma(omr, ux, r * ax), ly = C(3) * fma(omr, uy, r * ay);
    const C ax9 = C(9) * ax, ay9 = C(9) * ay;
    const C ou = C(4.5) * omr;
    const C cxx = fma(ou * ux, ux, ax9 * jx), cyy = fma(ou * uy, uy, ay9 * jy);
    const C cxy = fma(C(2) * ou * ux, uy, fma(ax9, jy, ay9 * jx));
    const C tr = cxx + cyy, b = C(-1.0 / 3.0) * tr;
    const C w1 = wq<C>(1), w5 = wq<C>(5);
    auto put = [&](int i, C g) { out[i] = fma(keep, f[i], fma(wq<C>(i), omr, g)); };
    put(0, wq<C>(0) * b);
    const C ex = w1 * (b + cxx), ey = w1 * (b + cyy), ox = w1 * lx, oy = w1 * ly;
    put(1, ex + ox);
    put(3, ex - ox);
    put(2, ey + oy);
    put(4, ey - oy);
    const C d = b + tr;
    const C ep = w5 * (d + cxy), em = w5 * (d - cxy), op = w5 * (lx + ly), om = w5 * (lx - ly);
    put(5, ep + op);
    put(7, ep - op);
    put(8, em + om);
    put(6, em - om);
}

__device__ __forceinline__ float tile_log(float x, const Log64Row*) { return dev_log(x); }
__device__ __forceinline__ double tile_log(double x, const Log64Row* tab) { return log64(x, tab); }

// nu^s without its gradient term, as in site_nu with the sums over phi formed from rho^s and
// scaled once, of the components that `part` of `parts` takes; also rho and 1/rho.  Constants
// have no gradient and are left out (theta (1/m^s - 1), and theta/m^0 of theta sum phi^s/m^s: what
// is left of that sum vanishes for equal m), which also leaves less to round.
template <typename C, int N>
__device__ __forceinline__ void tile_nu(const StepParams<C>& p, const C (&r)[N], const Log64Row* tab, int part,
                                        int parts, C (&nu)[N], C& rho, C& inv)
{
    rho = r[0];
#pragma unroll
    for (int s = 1; s < N; ++s) rho += r[s];
    inv = C(1) / rho;
    C acc[N], sm = C(0), quad = C(0);
#pragma unroll
    for (int s = 0; s < N; ++s) {
        C a = C(0);
#pragma unroll
        for (int t = 0; t < N; ++t) a += p.chi[s * N + t] * r[t];
        acc[s] = a;
        sm += r[s] * p.dm[s];
        quad += r[s] * a;
    }
    const C ti = p.theta * inv;
    const C G = -ti * fma(C(0.5) * quad, inv, sm);
    const C lnr = tile_log(rho, tab);
#pragma unroll
    for (int s = 0; s < N; ++s) {
        if (parts > 1 && s % parts != part) continue;
        nu[s] = fma(-p.th_m[s], lnr, fma(ti, acc[s], G));
        if ((p.log_mask >> s) & 1u) {
            const C fl = p.log_floor * rho;
            nu[s] += p.logc[s] * tile_log(r[s] > fl ? r[s] : fl, tab);
        }
    }
}

// rho^s of every site and component (one per thread), for k_tile's rs.
template <typename T>
__global__ void __launch_bounds__(128)
k_tile_rho(const T* __restrict__ f, typename Storage<T>::C* __restrict__ rs,
           const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    using C = typename Storage<T>::C;
    const int site = blockIdx.x * 128 + threadIdx.x, s = blockIdx.y;
    grid_dependency_wait();
    if (site < (int)p.S) {
        const int y = site / p.nx;
        C v[Q];
        tile_pull<T, C>(f, p, s, site - y * p.nx, y, v);
        rs[s * p.S + site] = sum9(v);
    }
    grid_dependents_launch();
}

// One timestep fin -> fout on the tile at column x0, row y0: TX = 1 << lx columns, ty rows.
// blockDim.x = N TX TY, or in FP64 more: threads beyond those pull around the tile while the
// others pull the tile, and parts > 1 spreads a site's potentials over as many threads -- for
// tiles of so few warps that SM quarters would idle.  rs: the rho^s field of fin, read around
// the tile instead of pulling there, or null.  p may live in parameter or shared memory.
template <typename T, int N>
__device__ __forceinline__ void tile_step(const T* __restrict__ fin, T* __restrict__ fout,
                                          const typename Storage<T>::C* __restrict__ rs,
                                          const StepParams<typename Storage<T>::C>& p, const int x0,
                                          const int y0, int lx, int ty, int parts64)
{
    using C = typename Storage<T>::C;
    constexpr bool F64 = sizeof(C) == 8;
    const int parts = F64 ? parts64 : 1;
    __shared__ Log64Row tab[F64 ? LOG64_ROWS : 1];
    extern __shared__ __align__(16) unsigned char tile_raw[];
    const int TX = 1 << lx, SITES = ty << lx;
    const int EX = TX + 4, EY = ty + 4, NX = TX + 2, NY = ty + 2;
    C* R = reinterpret_cast<C*>(tile_raw);   // [N][EY][EX]
    C* NU = R + N * EX * EY;                 // [N][NY][NX]
    C* J = NU + N * NX * NY;                 // [2][N][SITES]
    C* U = J + 2 * N * SITES;                // [2][SITES]
    C* RT = U + 2 * SITES;                   // Gibbs-Duhem: rho [NY][NX], 1/rho [SITES], a [2][N][SITES]
    C* IT = RT + NX * NY;
    C* A = IT + SITES;

    const int tid = threadIdx.x;
    const int s = tid / SITES, site = tid - s * SITES;
    const bool mine = !F64 || s < N;   // (else a thread beyond the tile's)
    const int tx = site & (TX - 1), tyy = site >> lx;
    const int x = x0 + tx, y = y0 + tyy;
    const bool own = x < p.nx && y < p.ny;
    // (lanes beyond the lattice compute some site's values and store nothing)
    const int xlast = p.nx + 1;

    if constexpr (F64) log64_load(tab);
    // the previous step's populations are complete from here on
    grid_dependency_wait();

    // ---- rho^s on the tile and two around it; j^s on the tile
    C f[Q], r = C(0), jx = C(0), jy = C(0);
    if (mine) tile_pull<T, C>(fin, p, s, min(x, xlast), wrap_any(y, p.ny), f);
    const int ring2 = EX * EY - SITES;
    // item k of the surroundings of component c
    auto around = [&](int c, int k) {
        int q = k, ex, ey;
        if (q < 4 * EX) {                      // the two rows above, then the two below
            ey = q / EX;
            ex = q - ey * EX;
            ey += ey >= 2 ? ty : 0;
        } else {                               // two columns left and right of each tile row
            q -= 4 * EX;
            ey = 2 + (q >> 2);
            ex = (q & 3) + ((q & 2) ? TX : 0);
        }
        const int yr = wrap_any(y0 - 2 + ey, p.ny);
        C rv;
        if (rs) {
            rv = rs[c * p.S + yr * p.nx + wrap_any(x0 - 2 + ex, p.nx)];
        } else {
            C v[Q];
            tile_pull<T, C>(fin, p, c, min(x0 - 2 + ex, xlast), yr, v);
            rv = sum9(v);
        }
        R[(c * EY + ey) * EX + ex] = rv;
    };
    const int extra = F64 ? (int)blockDim.x - N * SITES : 0;
    if (extra > 0) {
        for (int k = tid - N * SITES; k >= 0 && k < N * ring2; k += extra) around(k / ring2, k % ring2);
    } else {
        for (int k = site; k < ring2; k += SITES) around(s, k);
    }
    if (mine) {
        r = sum9(f);
        const C a = f[5] - f[7], b = f[6] - f[8];
        jx = (f[1] - f[3]) + (a - b);
        jy = (f[2] - f[4]) + (a + b);
        R[(s * EY + tyy + 2) * EX + tx + 2] = r;
        J[s * SITES + site] = jx;
        J[(N + s) * SITES + site] = jy;
    }
    __syncthreads();
    grid_dependents_launch();

    // ---- nu^s on the tile and one around it; u on the tile
    const int npad = (NX * NY + 31) / 32 * 32;   // (a warp's threads take the same part)
    const int threads = F64 ? (int)blockDim.x : N * SITES;
    for (int it = tid; it < (F64 ? npad * parts : NX * NY); it += threads) {
        const int part = F64 ? it / npad : 0, k = it - part * npad;
        if (F64 && k >= NX * NY) continue;
        int bx, by;
        if (k < SITES) {
            bx = (k & (TX - 1)) + 1;
            by = (k >> lx) + 1;
        } else {
            int q = k - SITES;
            if (q < 2 * NX) {
                by = q >= NX ? NY - 1 : 0;
                bx = q >= NX ? q - NX : q;
            } else {
                q -= 2 * NX;
                by = 1 + (q >> 1);
                bx = (q & 1) ? NX - 1 : 0;
            }
        }
        const int yy = y0 - 1 + by;
        const C* c = R + (by + 1) * EX + bx + 1;
        // rows beyond a wall are the mirror images of those next to it
        const int up = (p.walls && yy <= 0) ? 0 : -EX, dn = (p.walls && yy >= p.ny - 1) ? 0 : EX;
        C rr[N], nu[N], rho, inv;
#pragma unroll
        for (int t = 0; t < N; ++t) rr[t] = c[t * EX * EY];
        tile_nu<C, N>(p, rr, tab, part, parts, nu, rho, inv);
#pragma unroll
        for (int t = 0; t < N; ++t) {
            if (parts > 1 && t % parts != part) continue;
            const C* g = c + t * EX * EY;
            if (p.kappa != C(0)) {
                const C ax = (g[-1] + g[1]) + (g[up] + g[dn]);
                const C di = (g[up - 1] + g[up + 1]) + (g[dn - 1] + g[dn + 1]);
                nu[t] = fma(-p.kappa, fma(C(2.0 / 3.0), ax, fma(C(1.0 / 6.0), di, C(-10.0 / 3.0) * rr[t])), nu[t]);
            }
            NU[(t * NY + by) * NX + bx] = nu[t];
        }
        if (part != parts - 1) continue;
        if (N <= TILE_GD_NMAX && p.gd) RT[by * NX + bx] = rho;
        if (k < SITES) {
            C ux = C(0), uy = C(0);
#pragma unroll
            for (int t = 0; t < N; ++t) {
                ux += J[t * SITES + k];
                uy += J[(N + t) * SITES + k];
            }
            U[k] = ux * inv;
            U[SITES + k] = uy * inv;
            if (N <= TILE_GD_NMAX && p.gd) IT[k] = inv;
            if (x0 + bx - 1 < p.nx && yy < p.ny && (!(rho > C(0)) || !isfinite(rho)))
                atomicOr(p.status, STATUS_NONFINITE);
        }
    }
    __syncthreads();

    // ---- collision: a^s = -(1 - 1/2tau) grad nu^s + g
    const int up = (p.walls && y == 0) ? 0 : -NX, dn = (p.walls && y == p.ny - 1) ? 0 : NX;
    auto grad = [&](const C* g, C& gx, C& gy) {   // 3 sum_i w_i v_i g(r + v_i)
        const C ne = g[dn + 1], nw = g[dn - 1], se = g[up + 1], sw = g[up - 1];
        gx = fma(C(1.0 / 3.0), g[1] - g[-1], C(1.0 / 12.0) * ((ne - nw) + (se - sw)));
        gy = fma(C(1.0 / 3.0), g[dn] - g[up], C(1.0 / 12.0) * ((ne - se) + (nw - sw)));
    };
    C ax = C(0), ay = C(0);
    if (mine) {
        grad(NU + (s * NY + tyy + 1) * NX + tx + 1, ax, ay);
        ax = fma(-p.fcoef, ax, p.gx);
        ay = fma(-p.fcoef, ay, p.gy);
    }
    if (N <= TILE_GD_NMAX && p.gd) {
        // the common shift (A_c - A)/rho of every component (gibbs_duhem_shift)
        if (mine) {
            A[s * SITES + site] = ax - p.gx;
            A[(N + s) * SITES + site] = ay - p.gy;
        }
        __syncthreads();
        if (!mine) return;
        C sx = C(0), sy = C(0), grx, gry;
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const C rt = R[(t * EY + tyy + 2) * EX + tx + 2];
            sx += rt * A[t * SITES + site];
            sy += rt * A[(N + t) * SITES + site];
        }
        grad(RT + (tyy + 1) * NX + tx + 1, grx, gry);
        const C k = p.fcoef * C(1.0 / 3.0), it = IT[site];
        ax += (k * grx - sx) * it;
        ay += (k * gry - sy) * it;
    }
    if (!mine || !own) return;
    const C ux = U[site], uy = U[SITES + site];
    C fjx, fjy, out[Q];
    forcing_momentum(p, r, jx, jy, ux, uy, fjx, fjy);
    collide_poly(p, f, r, fjx, fjy, ux, uy, ax, ay, out);
    // the new values, and their copies in the ghost columns where the tile touches an edge
    const bool edge = x0 < p.hx || x0 + TX > p.nx - p.hx;
    T* row = fout + (unsigned)(s * p.ny + y) * (Q * (unsigned)p.pitch);
    auto put = [&](T* line, C v) {
        if (edge)
            store_row(line, x, p.nx, p.hx, v);
        else
            Storage<T>::store(line + p.hx + x, v);
    };
#pragma unroll
    for (int i = 0; i < Q; ++i) put(row + i * (unsigned)p.pitch, out[i]);
}

// The three rows next to each wall (blockIdx.y: the lower, the upper one), for a lattice whose
// other rows the march steps: tiles of 32 x 3 sites.
constexpr int TILE_WALL_ROWS = 3;
template <typename T, int N>
__global__ void __launch_bounds__(tile_max_threads<T>()) __maxnreg__(tile_max_regs<T>(N))
k_tile_walls(const T* __restrict__ fin, T* __restrict__ fout,
             const __grid_constant__ StepParams<typename Storage<T>::C> p)
{
    tile_step<T, N>(fin, fout, nullptr, p, blockIdx.x * 32, blockIdx.y ? p.ny - TILE_WALL_ROWS : 0, 5,
                    TILE_WALL_ROWS, 1);
}

template <typename T, int N>
__global__ void __launch_bounds__(tile_max_threads<T>()) __maxnreg__(tile_max_regs<T>(N))
k_tile(const T* __restrict__ fin, T* __restrict__ fout, const typename Storage<T>::C* __restrict__ rs,
       const __grid_constant__ StepParams<typename Storage<T>::C> p, int lx, int ty, int parts)
{
    tile_step<T, N>(fin, fout, rs, p, blockIdx.x << lx, blockIdx.y * ty, lx, ty, parts);
}

}  // namespace mclb
