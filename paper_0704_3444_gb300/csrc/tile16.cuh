// tile16.cuh -- small tiles for the 16-bit storage formats: the schedule of tile.cuh in the
// arithmetic of the schedules it stands in for.
//
// A stored deviation has 8 or 11 bits, so one last bit of the FP32 arithmetic before it flips its
// rounding now and then, and after a few dozen steps states that differ by such flips differ by
// 3e-5 in rho and 1e-3 in U (BF16; FP16 an eighth).  Which schedule AUTO picks, by size, or a
// batch, or a slab, must not show in the results: these tiles form every sum in the order and with
// the roundings of the march (SiteSums and the sums along a column, physics.cuh), and on the three
// rows next to a wall those of the staged step, which steps them for the march.  The states are
// equal bit for bit.
//
// What bounds it: latency, as in tile.cuh, so the longer collision costs little.  us a step, with the
// shorter arithmetic of tile.cuh and other values / this: 300 x 170 x 4 10.7 / 11.0, 440^2 x 3 20.4 /
// 20.7, 310^2 x 6 26.4 / 26.7, walls 510^2 x 3 26.0 / 27.9, 360^2 x 6 33.9 / 37.0 (the march 65).
#pragma once

#include "staged.cuh"
#include "tile.cuh"

namespace mclb {

// rho^s and j^s of one site, summed as the march sums them or, WALL, as the staged step does
template <bool WALL>
__device__ __forceinline__ float tile16_density(const float (&f)[Q])
{
    if constexpr (WALL) {
        float r = f[0];
#pragma unroll
        for (int i = 1; i < Q; ++i) r += f[i];
        return r;
    }
    return sum9(f);
}
template <bool WALL>
__device__ __forceinline__ void tile16_momentum(const float (&f)[Q], float& jx, float& jy)
{
    if constexpr (WALL) {
        jx = ((((f[1] - f[3]) + f[5]) - f[6]) - f[7]) + f[8];
        jy = ((((f[2] - f[4]) + f[5]) + f[6]) - f[7]) - f[8];
        return;
    }
    const float a = f[5] - f[7], b = f[6] - f[8];
    jx = (f[1] - f[3]) + (a - b);
    jy = (f[2] - f[4]) + (a + b);
}

// One timestep fin -> fout of the tile at column x0, row y0: TX = 1 << lx columns, ty rows, of which
// those below row yend are written.  Threads beyond N TX ty help with the potentials only.
// WALL: the staged step's arithmetic and walls; otherwise rows that no wall reaches.
template <typename T, int N, bool WALL>
__device__ __forceinline__ void tile16_step(const T* __restrict__ fin, T* __restrict__ fout,
                                            const StepParams<float>& p, const int x0, const int y0, int lx,
                                            int ty, int yend)
{
    extern __shared__ __align__(16) unsigned char tile_raw[];
    const int TX = 1 << lx, SITES = ty << lx;
    const int EX = TX + 4, EY = ty + 4, NX = TX + 2, NY = ty + 2;
    float* R = reinterpret_cast<float*>(tile_raw);   // [N][EY][EX]
    float* NU = R + N * EX * EY;                     // [N][NY][NX]
    float* J = NU + N * NX * NY;                     // [2][N][SITES]
    float* U = J + 2 * N * SITES;                    // [2][SITES]

    const int tid = threadIdx.x;
    const int s = tid / SITES, site = tid - s * SITES;
    const bool mine = s < N;
    const int tx = site & (TX - 1), tyy = site >> lx;
    const int x = x0 + tx, y = y0 + tyy;
    // (lanes beyond the lattice compute some site's values and store nothing)
    const int xlast = p.nx + 1;

    // the previous step's populations are complete from here on
    grid_dependency_wait();

    // ---- rho^s on the tile and two around it; j^s on the tile
    float f[Q], r = 0.0f, jx = 0.0f, jy = 0.0f;
    if (mine) {
        tile_pull<T, float>(fin, p, s, min(x, xlast), wrap_any(y, p.ny), f);
        for (int k = site; k < EX * EY - SITES; k += SITES) {
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
            float v[Q];
            tile_pull<T, float>(fin, p, s, min(x0 - 2 + ex, xlast), wrap_any(y0 - 2 + ey, p.ny), v);
            R[(s * EY + ey) * EX + ex] = tile16_density<WALL>(v);
        }
        r = tile16_density<WALL>(f);
        tile16_momentum<WALL>(f, jx, jy);
        R[(s * EY + tyy + 2) * EX + tx + 2] = r;
        J[s * SITES + site] = jx;
        J[(N + s) * SITES + site] = jy;
    }
    __syncthreads();
    grid_dependents_launch();

    // ---- nu^s on the tile and one around it; u on the tile
    const float k6 = 6.0f * p.kappa;
    for (int k = tid; k < NX * NY; k += blockDim.x) {
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
        const float* c = R + (by + 1) * EX + bx + 1;
        // rows beyond a wall are the mirror images of those next to it
        const int up = WALL && yy <= 0 ? 0 : -EX, dn = WALL && yy >= p.ny - 1 ? 0 : EX;
        float rr[N], rho = 0.0f;
#pragma unroll
        for (int t = 0; t < N; ++t) {
            rr[t] = c[t * EX * EY];
            rho += rr[t];
        }
        const float inv = 1.0f / rho;
        if constexpr (WALL) {
            float lap[N], nu[N];
#pragma unroll
            for (int t = 0; t < N; ++t)
                lap[t] = laplacian_of(rr[t], [&](int i) {
                    return c[t * EX * EY + (vy(i) < 0 ? up : vy(i) > 0 ? dn : 0) + vx(i)];
                });
            site_nu<float, N>(p, rr, lap, nu);
#pragma unroll
            for (int t = 0; t < N; ++t) NU[(t * NY + by) * NX + bx] = nu[t];
        } else {
            const SiteSums<float, N> sums(p, rr, inv);
            const float lnr = dev_log(rho);
#pragma unroll
            for (int t = 0; t < N; ++t) {
                const float* g = c + t * EX * EY;
                auto side = [&](int o) { return lap_side(g[o], g[o - 1] + g[o + 1]); };
                const float part = nu_part(k6, mul_rn(-k6, side(-EX)), sums.nu(p, rr, rho, inv, lnr, t),
                                           lap_mid(g[0], g[-1] + g[1]));
                NU[(t * NY + by) * NX + bx] = nu_whole(k6, part, side(EX));
            }
        }
        if (k < SITES) {
            float ux = 0.0f, uy = 0.0f;
#pragma unroll
            for (int t = 0; t < N; ++t) {
                ux += J[t * SITES + k];
                uy += J[(N + t) * SITES + k];
            }
            U[k] = ux * inv;
            U[SITES + k] = uy * inv;
            if (x0 + bx - 1 < p.nx && yy < yend && (!(rho > 0.0f) || !isfinite(rho)))
                atomicOr(p.status, STATUS_NONFINITE);
        }
    }
    __syncthreads();
    if (!mine || x >= p.nx || y >= yend) return;

    // ---- collision: a^s = -(1 - 1/2tau) grad nu^s + g
    const float* g = NU + (s * NY + tyy + 1) * NX + tx + 1;
    const float ux = U[site], uy = U[SITES + site];
    float ax, ay, fjx, fjy, e[Q], out[Q];
    forcing_momentum(p, r, jx, jy, ux, uy, fjx, fjy);
    if constexpr (WALL) {
        const int up = y == 0 ? 0 : -NX, dn = y == p.ny - 1 ? 0 : NX;
        float gx, gy;
        gradient_of([&](int i) { return g[(vy(i) < 0 ? up : vy(i) > 0 ? dn : 0) + vx(i)]; }, gx, gy);
        ax = fma(-p.fcoef, gx, p.gx);
        ay = fma(-p.fcoef, gy, p.gy);
        eq_weights(ux, uy, fma(ux, ux, uy * uy), e);
        collide(p, f, e, r, fjx, fjy, ax, ay, out);
        store_site(fout, p, s, y, x, out);
    } else {
        auto d = [&](int o) { return g[o + 1] - g[o - 1]; };
        auto rows = [&](int o) { return grad_rows<N>(g[o], g[o + 1] + g[o - 1]); };
        ax = accel_of(p.fcoef, grad_cols(grad_cols_part(d(0), d(-NX)), d(NX)), p.gx);
        ay = accel_of(p.fcoef, rows(NX) - rows(-NX), p.gy);
        eq_weights(ux, uy, speed2(ux, uy), e);
        collide(p, f, e, r, fjx, fjy, ax, ay, out, r);
        // the new values, and their copies in the ghost columns where the tile touches an edge
        const bool edge = x0 < p.hx || x0 + TX > p.nx - p.hx;
        T* row = fout + (unsigned)(s * p.ny + y) * (Q * (unsigned)p.pitch);
        auto put = [&](auto* line, float v) {
            if (edge)
                store_row(line, x, p.nx, p.hx, v);
            else
                Storage<std::remove_pointer_t<decltype(line)>>::store(line + p.hx + x, v);
        };
        float dsum = 0.0f;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const T v = Storage<T>::pack(out[i]);
            dsum = add_wide<T>(dsum, v);
            put(row + i * (unsigned)p.pitch, to_c<T>(v));
        }
        put(rho_line(fout, p, s, y), r - dsum);
    }
}

// Rows next to a wall, in the arithmetic of the staged step
constexpr int TILE16_WALL_ROWS = 3;

// gridDim.y: the row tiles; between walls the rows next to the lower one, those next to the upper one
// (ny > TILE16_WALL_ROWS), then the tiles of the rows between them.
template <typename T, int N, bool WALLS>
__global__ void __launch_bounds__(tile_max_threads<T>()) __maxnreg__(tile_max_regs<T>(N))
k_tile16(const T* __restrict__ fin, T* __restrict__ fout, const __grid_constant__ StepParams<float> p, int lx,
         int ty)
{
    const int x0 = blockIdx.x << lx, by = blockIdx.y;
    if constexpr (WALLS) {
        const int upper = max(TILE16_WALL_ROWS, p.ny - TILE16_WALL_ROWS);
        if (by < 2)
            tile16_step<T, N, true>(fin, fout, p, x0, by ? upper : 0, lx, TILE16_WALL_ROWS,
                                    by ? p.ny : min(p.ny, TILE16_WALL_ROWS));
        else
            tile16_step<T, N, false>(fin, fout, p, x0, TILE16_WALL_ROWS + (by - 2) * ty, lx, ty, upper);
    } else {
        tile16_step<T, N, false>(fin, fout, p, x0, by * ty, lx, ty, p.ny);
    }
}

// The rows next to the walls (blockIdx.y: the lower, the upper one) of a lattice whose other rows
// the march steps: tiles of 32 x 3 sites.
template <typename T, int N>
__global__ void __launch_bounds__(tile_max_threads<T>()) __maxnreg__(tile_max_regs<T>(N))
k_tile16_walls(const T* __restrict__ fin, T* __restrict__ fout, const __grid_constant__ StepParams<float> p)
{
    tile16_step<T, N, true>(fin, fout, p, blockIdx.x * 32, blockIdx.y ? p.ny - TILE16_WALL_ROWS : 0, 5,
                            TILE16_WALL_ROWS, blockIdx.y ? p.ny : TILE16_WALL_ROWS);
}

}  // namespace mclb
