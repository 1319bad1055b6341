// fields.cuh -- the macroscopic output fields of a D2Q9 state in two launches: the density pass
// (k_density, staged.cuh, which also leaves the total momentum in U's place) and one pass over
// tiles that forms nu^s on chip and writes rho^s, U, mu^s and P.
//
// What bounds it: at 8192 x 2048 x 3 the density pass moves 2.1 GB at the copy rate; the tiles
// issue (FP32 output widened to FP64 by moving bits: the conversion instruction runs in the
// FP64 pipe).  Before, nu^s went through memory in a launch of its own, bound by the index
// arithmetic of its neighbour loads, and the output pass pulled every population again for
// the momentum.  The Laplacian is summed from differences of neighbours: by sums that cancel against
// 10/3 rho^s the error of an FP32 mu^s grew by a quarter at kappa = 0.5 (1.13e-7 -> 1.41e-7).
// us a call (rho, U, mu), before / now: 8192 x 2048 x 3 FP32 1386 / 814, 2048^2 x 5 FP32 543 / 329,
// BF16 778 / 401, 64 x 64 x 2 FP64 40 / 18, 2048^2 x 2 FP64 3141 / 2894.
#pragma once

#include "staged.cuh"
#include "tile.cuh"

namespace mclb {

constexpr int FIELDS_X = 28;             // written columns of the 32 a warp holds
constexpr int FIELDS_MAX_WARPS = 8;

// rho^s (two around the tile) and nu^s (one around)
__host__ __device__ constexpr int fields_smem_values(int n, int rows) { return 32 * n * (2 * rows + 6); }

// U holds the stashed total momentum on entry.  Any output may be null.  Tiles of FIELDS_X x rows,
// row by row of the lattice; lane l is column x0 - 2 + l, the warps share the rows of each stage.
template <typename C, int N>
__global__ void __launch_bounds__(32 * FIELDS_MAX_WARPS)
k_fields(const C* __restrict__ rs, double* __restrict__ rho_out, double* __restrict__ U,
         double* __restrict__ mu_out, double* __restrict__ P, const __grid_constant__ StepParams<C> p, int rows)
{
    extern __shared__ __align__(16) unsigned char fields_raw[];
    constexpr bool F64 = sizeof(C) == 8;
    __shared__ Log64Row tab[F64 ? LOG64_ROWS : 1];
    const int EY = rows + 4, NY = rows + 2;
    C* R = reinterpret_cast<C*>(fields_raw);   // [N][EY][32]
    C* NU = R + N * EY * 32;                   // [N][NY][32]
    const int tiles_x = (p.nx + FIELDS_X - 1) / FIELDS_X, tile_y = (int)blockIdx.x / tiles_x;
    const int x0 = ((int)blockIdx.x - tile_y * tiles_x) * FIELDS_X, y0 = tile_y * rows;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int x = x0 - 2 + lane;

    if constexpr (F64) log64_load(tab);
    grid_dependency_wait();
    {
        const int xw = wrap_any(x, p.nx);
        for (int e = warp; e < EY; e += warps) {
            const C* row = rs + (long long)wrap_any(y0 - 2 + e, p.ny) * p.nx + xw;
#pragma unroll
            for (int s = 0; s < N; ++s) R[(s * EY + e) * 32 + lane] = row[s * p.S];
        }
    }
    __syncthreads();

    auto laplacian = [&](const C* g, int up, int dn) {
        return laplacian_of(g[0], [&](int i) { return g[(vy(i) < 0 ? up : vy(i) > 0 ? dn : 0) + vx(i)]; });
    };
    auto gradient = [&](const C* g, int up, int dn, C& gx, C& gy) {   // 3 sum_i w_i v_i g(r + v_i)
        const C ne = g[dn + 1], nw = g[dn - 1], se = g[up + 1], sw = g[up - 1];
        gx = fma(C(1.0 / 3.0), g[1] - g[-1], C(1.0 / 12.0) * ((ne - nw) + (se - sw)));
        gy = fma(C(1.0 / 3.0), g[dn] - g[up], C(1.0 / 12.0) * ((ne - se) + (nw - sw)));
    };
    // offsets to the rows below and above in y; rows beyond a wall are mirror images
    const auto up_of = [&](int y) { return (p.walls && y <= 0) ? 0 : -32; };
    const auto dn_of = [&](int y) { return (p.walls && y >= p.ny - 1) ? 0 : 32; };

    if (U) {
        for (int t = warp; t < NY; t += warps) {
            if (lane < 1 || lane > 30) continue;
            const int y = y0 - 1 + t;
            const C* c = R + (t + 1) * 32 + lane;
            C r[N], nu[N], rho, inv;
#pragma unroll
            for (int s = 0; s < N; ++s) r[s] = c[s * EY * 32];
            tile_nu<C, N>(p, r, tab, 0, 1, nu, rho, inv);
#pragma unroll
            for (int s = 0; s < N; ++s) {
                if (p.kappa != C(0)) nu[s] = fma(-p.kappa, laplacian(c + s * EY * 32, up_of(y), dn_of(y)), nu[s]);
                NU[(s * NY + t) * 32 + lane] = nu[s];
            }
        }
        __syncthreads();
    }
    if (lane < 2 || lane >= 30 || x >= p.nx) return;
    for (int l = warp; l < rows && y0 + l < p.ny; l += warps) {
        const int y = y0 + l;
        const long long site = (long long)y * p.nx + x;
        const C* c = R + (l + 2) * 32 + lane;
        const int up = up_of(y), dn = dn_of(y);
        C r[N], rho = C(0);
#pragma unroll
        for (int s = 0; s < N; ++s) {
            r[s] = c[s * EY * 32];
            rho += r[s];
        }
        if (rho_out)
#pragma unroll
            for (int s = 0; s < N; ++s) rho_out[s * p.S + site] = widen(r[s]);
        if (U) {
            C ax[N], ay[N], fx = C(0), fy = C(0);
#pragma unroll
            for (int s = 0; s < N; ++s) {
                C gx, gy;
                gradient(NU + (s * NY + l + 1) * 32 + lane, up, dn, gx, gy);
                ax[s] = -p.fcoef * gx + p.gx;
                ay[s] = -p.fcoef * gy + p.gy;
            }
            if (p.gd) {
                C grx = C(0), gry = C(0);
#pragma unroll
                for (int s = 0; s < N; ++s) {
                    C gx, gy;
                    gradient(c + s * EY * 32, up, dn, gx, gy);
                    grx += gx;
                    gry += gy;
                }
                gibbs_duhem_shift<C, N>(p, r, rho, grx, gry, ax, ay);
            }
#pragma unroll
            for (int s = 0; s < N; ++s) {
                fx += r[s] * ax[s];
                fy += r[s] * ay[s];
            }
            C jx, jy;
            unstash2(U + site, p.S, jx, jy);
            U[site] = widen(fma(C(0.5), fx, jx) / rho);
            U[p.S + site] = widen(fma(C(0.5), fy, jy) / rho);
        }
        if (mu_out || P) {
            C lap[N], mu[N];
#pragma unroll
            for (int s = 0; s < N; ++s) lap[s] = p.kappa != C(0) ? laplacian(c + s * EY * 32, up, dn) : C(0);
            site_mu<C, N>(p, r, lap, mu);
            if (mu_out)
#pragma unroll
                for (int s = 0; s < N; ++s) mu_out[s * p.S + site] = widen(mu[s]);
            if (P) {
                const C psi = site_psi<C, N>(p, r);
                C rmu = C(0), gg = C(0), pxx = C(0), pxy = C(0), pyy = C(0);
#pragma unroll
                for (int s = 0; s < N; ++s) {
                    C gx, gy;
                    gradient(c + s * EY * 32, up, dn, gx, gy);
                    rmu += r[s] * mu[s];
                    gg += C(0.5) * p.kappa * (gx * gx + gy * gy);
                    pxx += p.kappa * gx * gx;
                    pxy += p.kappa * gx * gy;
                    pyy += p.kappa * gy * gy;
                }
                const C iso = rmu - (psi + gg);
                P[site] = widen(iso + pxx);
                P[p.S + site] = widen(pxy);
                P[2 * p.S + site] = widen(iso + pyy);
            }
        }
    }
}

}  // namespace mclb
