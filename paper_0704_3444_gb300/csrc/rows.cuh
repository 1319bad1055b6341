// rows.cuh -- one launch per timestep by row tiles, FP32 arithmetic: the schedule of lattices
// that fit the caches, where the column march (march.cuh) waits out the latency of its row
// iterations instead of moving bytes.
//
// A CTA owns 28 x 8 sites.  Warp w (0..3) of component s pulls the tile rows 2w and 2w + 1 and
// one of the four halo rows; lane l is column x0 - 2 + l, so every load is one contiguous row
// segment and the two halo columns each side come with it.  The two rows of a lane travel
// as one float2 through the packed FP32x2 instructions: moments and collision of both cost the
// issue slots of one.  As in tile.cuh: rho^s (tile and two around), barrier, nu^s (one
// around) and u, barrier, collision, store with ghost columns.
//
// Populations read per written one: 12 x 32 / (8 x 28) = 1.71, the surplus from L2.  What
// bounds it is the chain of one step (pull from L2, barrier, logarithm and division, barrier,
// store, next launch) and, the more tiles there are, instruction issue: about 740 instructions a
// warp, issue slots 43 % busy at 256^2 x 3 (0.7 of a wave of CTAs), 56 % at 512 x 384 x 3, 64 % at 1000 x 333
// x 3 between walls.  The march needs segment rows + 4 dependent iterations of about 1.2 us for
// the same step.  Eight rows: with
// 10 or 12, which pull 1.4 and 1.33 rows for each written one, CTAs are larger and fewer (us per
// step, 8 / 10 / 12 rows: 256^2 x 3 8.85 / 8.62 / 9.27, 300^2 x 2 8.0 / 8.5 / 8.8, 512 x 384 x 3 14.3 /
// 14.5 / 15.3, 700^2 x 2 18.8 / 20.3 / 19.8; 48 batched instances 153 / - / 184).  (The pulls by
// TMA boxes into shared memory instead: 18 % fewer instructions, but every CTA waits out
// its copies: 48.8 us against 44.1 us at 1024^2 x 2.)
#pragma once

#include "tile.cuh"

namespace mclb {

constexpr int ROWS_X = 28;        // written columns of the 32 a warp holds
constexpr int ROWS_Y = 8;         // written rows
constexpr int ROWS_WPC = 4;       // warps per component, two written rows and one halo row each
constexpr int ROWS_EY = ROWS_Y + 4;
constexpr int ROWS_NY = ROWS_Y + 2;
constexpr int ROWS_MIN_NY = ROWS_EY;   // rows wrap at most once
constexpr int ROWS_NMAX = 5;           // two CTAs of more warps do not fit an SM's registers
// CTAs an SM is to hold: about 36 warps of 48 to 64 registers
__host__ __device__ constexpr int rows_ctas(int n) { return n == 1 ? 8 : n == 2 ? 4 : n == 3 ? 3 : 2; }

// rho^s, nu^s, j^s of N components and u, in floats
__host__ __device__ constexpr int rows_smem_floats(int n)
{
    return 32 * (n * (ROWS_EY + ROWS_NY + 2 * ROWS_Y) + 2 * ROWS_Y);
}

__device__ __forceinline__ int wrap_once(int a, int n)
{
    a += a < 0 ? n : 0;
    return a - (a >= n ? n : 0);
}

// line + i pitch, pitch in bytes: one wide multiply-add
template <typename T>
__device__ __forceinline__ T* line_at(T* line, unsigned pitch_bytes, unsigned i)
{
    return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(line) + (unsigned long long)pitch_bytes * i);
}

// collide_poly (tile.cuh) on two sites of one component
__device__ __forceinline__ void collide_poly2(const StepParams<float>& p, const float2 (&f)[Q], float2 r,
                                              float2 jx, float2 jy, float2 ux, float2 uy, float2 ax,
                                              float2 ay, float2 shift, float2 (&out)[Q])
{
    const float2 mone = pdup(-1.0f), nine = pdup(9.0f), three = pdup(3.0f);
    const float2 omr = pmul(pdup(p.omega), r), keep = pdup(1.0f - p.omega);
    const float2 k0 = pfma(shift, mone, omr);
    const float2 lx = pmul(three, pfma(omr, ux, pmul(r, ax))), ly = pmul(three, pfma(omr, uy, pmul(r, ay)));
    const float2 ax9 = pmul(nine, ax), ay9 = pmul(nine, ay);
    const float2 oux = pmul(pmul(pdup(4.5f), omr), ux), ouy = pmul(pmul(pdup(4.5f), omr), uy);
    const float2 cxx = pfma(oux, ux, pmul(ax9, jx)), cyy = pfma(ouy, uy, pmul(ay9, jy));
    const float2 cxy = pfma(padd(oux, oux), uy, pfma(ax9, jy, pmul(ay9, jx)));
    const float2 tr = padd(cxx, cyy), b = pmul(pdup(-1.0f / 3.0f), tr);
    const float2 w1 = pdup(wq<float>(1)), w5 = pdup(wq<float>(5));
    auto put = [&](int i, float2 g) { out[i] = pfma(keep, f[i], pfma(pdup(wq<float>(i)), k0, g)); };
    put(0, pmul(pdup(wq<float>(0)), b));
    const float2 ex = pmul(w1, padd(b, cxx)), ey = pmul(w1, padd(b, cyy)), ox = pmul(w1, lx), oy = pmul(w1, ly);
    put(1, padd(ex, ox));
    put(3, pfma(ox, mone, ex));
    put(2, padd(ey, oy));
    put(4, pfma(oy, mone, ey));
    const float2 d = padd(b, tr);
    const float2 ep = pmul(w5, padd(d, cxy)), em = pmul(w5, pfma(cxy, mone, d));
    const float2 op = pmul(w5, padd(lx, ly)), om = pmul(w5, pfma(ly, mone, lx));
    put(5, padd(ep, op));
    put(7, pfma(op, mone, ep));
    put(8, padd(em, om));
    put(6, pfma(om, mone, em));
}

// One timestep fin -> fout of the tile at column x0, row y0; CTA of 128 N threads.  p may live in
// parameter or shared memory.  Ends with threads past the collision at different points:
// another tile may follow at once (its first barrier is behind every read of this one's arrays
// that it overwrites).
template <int N, bool WALLS>
__device__ __forceinline__ void rows_tile(const float* __restrict__ fin, float* __restrict__ fout,
                                          const StepParams<float>& p, const int x0, const int y0)
{
    __shared__ float R[N][ROWS_EY][32];
    __shared__ float NU[N][ROWS_NY][32];
    __shared__ float JX[N][ROWS_Y][32], JY[N][ROWS_Y][32];
    __shared__ float U[2][ROWS_Y][32];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = warp / ROWS_WPC, w = warp % ROWS_WPC;
    const int x = x0 - 2 + lane;
    const int ya = y0 + 2 * w;
    const unsigned pb = (unsigned)p.pitch * 4u, rb = Q * pb;   // bytes of a line and of a row

    // column x (clamped: the ghost columns reach nx + 3) of row y of the component
    const float* base = fin + s * p.plane + (p.hx + min(x, p.nx + 1));
    auto row_of = [&](int y) { return line_at(base, rb, (unsigned)wrap_once(y, p.ny)); };
    // velocity i pulled from the rows y - 1, y, y + 1 (r[0..2]); links that cross a wall return
    // the site's own value of the opposite velocity
    auto pull = [&](const float* const* r, int i, bool lo, bool hi) {
        if constexpr (WALLS) {
            if (vy(i) != 0) {
                const bool b = vy(i) > 0 ? lo : hi;
                const float* q = b ? line_at(r[1], pb, (unsigned)opp9(i)) : line_at(r[1 - vy(i)], pb, (unsigned)i) - vx(i);
                return __ldg(q);
            }
        }
        return __ldg(line_at(r[1 - vy(i)], pb, (unsigned)i) - vx(i));
    };

    // the previous step's populations are complete from here on
    grid_dependency_wait();

    // ---- pull rows ya, ya + 1 and a halo row
    const int eh = w < 2 ? w : ROWS_Y + w;   // extended row 0, 1, ROWS_Y + 2 or ROWS_Y + 3
    float2 f[Q];
    float h[Q];
    {
        const float* r[4] = {row_of(ya - 1), row_of(ya), row_of(ya + 1), row_of(ya + 2)};
        const int yh = wrap_once(y0 - 2 + eh, p.ny);
        const float* q[3] = {row_of(yh - 1), row_of(yh), row_of(yh + 1)};
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            f[i].x = pull(r, i, ya == 0, ya == p.ny - 1);
            f[i].y = pull(r + 1, i, false, ya + 1 == p.ny - 1);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) h[i] = pull(q, i, yh == 0, yh == p.ny - 1);
    }
    const float2 mone = pdup(-1.0f);
    const float2 r = padd(padd(padd(padd(f[0], f[1]), padd(f[2], f[3])), padd(padd(f[4], f[5]), padd(f[6], f[7]))), f[8]);
    const float2 da = pfma(f[7], mone, f[5]), db = pfma(f[8], mone, f[6]);
    const float2 jx = padd(pfma(f[3], mone, f[1]), pfma(db, mone, da));
    const float2 jy = padd(pfma(f[4], mone, f[2]), padd(da, db));
    R[s][2 * w + 2][lane] = r.x;
    R[s][2 * w + 3][lane] = r.y;
    R[s][eh][lane] = sum9(h);
    JX[s][2 * w][lane] = jx.x;
    JX[s][2 * w + 1][lane] = jx.y;
    JY[s][2 * w][lane] = jy.x;
    JY[s][2 * w + 1][lane] = jy.y;
    __syncthreads();
    grid_dependents_launch();

    // ---- nu^s of the tile rows and one around them, one row per warp at a time
    for (int t = warp; t < ROWS_NY; t += ROWS_WPC * N) {
        if (lane < 1 || lane > 30) continue;
        const int yy = y0 - 1 + t;
        // rows beyond a wall are the mirror images of those next to it
        const int up = (WALLS && yy <= 0) ? 0 : -32, dn = (WALLS && yy >= p.ny - 1) ? 0 : 32;
        float rr[N], nu[N], rho, inv;
#pragma unroll
        for (int q = 0; q < N; ++q) rr[q] = R[q][t + 1][lane];
        tile_nu<float, N>(p, rr, nullptr, 0, 1, nu, rho, inv);
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const float* g = &R[q][t + 1][lane];
            if (p.kappa != 0.0f) {
                const float ax = (g[-1] + g[1]) + (g[up] + g[dn]);
                const float di = (g[up - 1] + g[up + 1]) + (g[dn - 1] + g[dn + 1]);
                nu[q] = fmaf(-p.kappa, fmaf(2.0f / 3.0f, ax, fmaf(1.0f / 6.0f, di, (-10.0f / 3.0f) * rr[q])), nu[q]);
            }
            NU[q][t][lane] = nu[q];
        }
    }
    // ---- u of the tile rows, from the last warp down (the first have the potentials)
    for (int l = ROWS_WPC * N - 1 - warp; l < ROWS_Y; l += ROWS_WPC * N) {
        float rho = 0.0f, tx = 0.0f, ty = 0.0f;
#pragma unroll
        for (int q = 0; q < N; ++q) {
            rho += R[q][l + 2][lane];
            tx += JX[q][l][lane];
            ty += JY[q][l][lane];
        }
        const float inv = 1.0f / rho;
        U[0][l][lane] = tx * inv;
        U[1][l][lane] = ty * inv;
        if (lane >= 2 && lane < 30 && x < p.nx && y0 + l < p.ny && (!(rho > 0.0f) || !isfinite(rho)))
            atomicOr(p.status, STATUS_NONFINITE);
    }
    __syncthreads();

    // ---- collision of both rows: a^s = -(1 - 1/2tau) grad nu^s + g
    if (lane < 2 || lane >= 30 || x >= p.nx || ya >= p.ny) return;
    float2 ax, ay;
    {
        const float* g = &NU[s][2 * w + 1][lane];
        const int ua = (WALLS && ya == 0) ? 0 : -32, na = (WALLS && ya == p.ny - 1) ? 0 : 32;
        const int nb = (WALLS && ya + 1 == p.ny - 1) ? 32 : 64;   // from row ya; row ya is above ya + 1
        const float2 w3 = pdup(-p.fcoef * (1.0f / 3.0f)), w12 = pdup(-p.fcoef * (1.0f / 12.0f));
        const float2 sw = make_float2(g[ua - 1], g[-1]), se = make_float2(g[ua + 1], g[1]);
        const float2 nw = make_float2(g[na - 1], g[nb - 1]), ne = make_float2(g[na + 1], g[nb + 1]);
        const float2 mid = pfma(make_float2(g[-1], g[31]), mone, make_float2(g[1], g[33]));
        const float2 ver = pfma(make_float2(g[ua], g[0]), mone, make_float2(g[na], g[nb]));
        const float2 e = pfma(sw, mone, ne), o = pfma(nw, mone, se);
        ax = pfma(w3, mid, pfma(w12, padd(e, o), pdup(p.gx)));
        ay = pfma(w3, ver, pfma(w12, pfma(o, mone, e), pdup(p.gy)));
    }
    const float2 ux = make_float2(U[0][2 * w][lane], U[0][2 * w + 1][lane]);
    const float2 uy = make_float2(U[1][2 * w][lane], U[1][2 * w + 1][lane]);
    const float2 fjx = p.bary ? pmul(r, ux) : jx, fjy = p.bary ? pmul(r, uy) : jy;
    float2 out[Q];
    collide_poly2(p, f, r, fjx, fjy, ux, uy, ax, ay, pdup(0.0f), out);

    // the new values, and their copies in the ghost columns where the tile touches an edge
    const bool two = ya + 1 < p.ny;
    float* oa = line_at(fout + s * p.plane + (p.hx + x), rb, (unsigned)ya);
    float* ob = line_at(oa, rb, 1u);
    if (x0 >= p.hx && x0 + ROWS_X <= p.nx - p.hx) {
#pragma unroll
        for (int i = 0; i < Q; ++i) *line_at(oa, pb, (unsigned)i) = out[i].x;
        if (two)
#pragma unroll
            for (int i = 0; i < Q; ++i) *line_at(ob, pb, (unsigned)i) = out[i].y;
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            store_row(line_at(oa, pb, (unsigned)i) - (p.hx + x), x, p.nx, p.hx, out[i].x);
            if (two) store_row(line_at(ob, pb, (unsigned)i) - (p.hx + x), x, p.nx, p.hx, out[i].y);
        }
    }
}

// gridDim = (column tiles, row tiles), blockDim.x = 128 N
template <int N, bool WALLS>
__global__ void __launch_bounds__(32 * ROWS_WPC * N, rows_ctas(N))
k_rows(const float* __restrict__ fin, float* __restrict__ fout, const __grid_constant__ StepParams<float> p)
{
    rows_tile<N, WALLS>(fin, fout, p, blockIdx.x * ROWS_X, blockIdx.y * ROWS_Y);
}

}  // namespace mclb
