// table_impl.cuh -- host launchers for one storage type, dispatched on N at run time.
#pragma once

#include <algorithm>
#include <cmath>

#include "batch.cuh"
#include "cube.cuh"
#include "cube_march.cuh"
#include "fields.cuh"
#include "ghosts.cuh"
#include "line3.cuh"
#include "march.cuh"
#include "mass.cuh"
#include "rows.cuh"
#include "staged.cuh"
#include "tile.cuh"
#include "tile16.cuh"

namespace mclb {

#define MCLB_DISPATCH_N(n, ...)                      \
    switch (n) {                                      \
        case 1: { constexpr int NN = 1; __VA_ARGS__ }       \
        case 2: { constexpr int NN = 2; __VA_ARGS__ }       \
        case 3: { constexpr int NN = 3; __VA_ARGS__ }       \
        case 4: { constexpr int NN = 4; __VA_ARGS__ }       \
        case 5: { constexpr int NN = 5; __VA_ARGS__ }       \
        case 6: { constexpr int NN = 6; __VA_ARGS__ }       \
        case 7: { constexpr int NN = 7; __VA_ARGS__ }       \
        case 8: { constexpr int NN = 8; __VA_ARGS__ }       \
        default: return cudaErrorInvalidValue;        \
    }

inline unsigned site_blocks(long long S) { return (unsigned)((S + SITE_THREADS - 1) / SITE_THREADS); }

// Launch with programmatic stream serialisation: the kernel may be scheduled while the one
// before it drains (it waits for that one's end itself).
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                             A... args)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

template <typename T>
struct Launch {
    using C = typename Storage<T>::C;

    static cudaError_t init(const Problem& P, const Scratch& sc, const double* rho, const double* u,
                            void* f, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_init<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(rho, u, (T*)f, p);
            return cudaGetLastError();
        });
    }

    template <int N>
    static cudaError_t fields_n(const StepParams<C>& p, const Scratch& sc, const T* f,
                                cudaStream_t st)
    {
        k_density<T, N><<<site_blocks(p.S), SITE_THREADS, 0, st>>>(f, (C*)sc.rho_s, p);
        k_potential<C, N><<<site_blocks(p.S), SITE_THREADS, 0, st>>>((const C*)sc.rho_s,
                                                                      (C*)sc.nu, p);
        return cudaGetLastError();
    }

    static cudaError_t step_staged(const Problem& P, const Scratch& sc, const void* fin, void* fout,
                                   cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            cudaError_t e = fields_n<NN>(p, sc, (const T*)fin, st);
            if (e != cudaSuccess) return e;
            k_collide<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(
                (const T*)fin, (T*)fout, (const C*)sc.rho_s, (const C*)sc.nu, p);
            return cudaGetLastError();
        });
    }

    // Strips of WOUT columns, segments of H rows: one wave of CTAs, each segment as
    // tall as the resident CTAs allow (every segment re-reads 4 halo rows and spends 4
    // warm-up iterations), at least 8 rows.
    template <int N, bool GD>
    static FusedPlan plan_k(const Problem& P, int sm_count)
    {
        using G = MarchGeom<T, N>;
        FusedPlan pl{};
        pl.ok = false;
        if (!G::FITS) return pl;
        if (cudaFuncSetAttribute(k_march<T, N, GD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)G::SMEM) != cudaSuccess)
            return pl;
        // the largest shared-memory carveout, so that the resident CTAs the occupancy
        // query counts (it assumes the largest) are the ones the launch gets
        if (cudaFuncSetAttribute(k_march<T, N, GD>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess)
            return pl;
        int ctas = 0;  // resident CTAs per SM as the runtime computes them (smem, registers)
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, k_march<T, N, GD>, G::THREADS,
                                                          G::SMEM) != cudaSuccess || ctas < 1)
            return pl;
        pl.W = G::WOUT;
        pl.box_w = G::WI;
        pl.out_w = G::TMA_STORE ? MARCH_OUT : (G::CTA_STORE ? G::WOUT : 0);
        pl.NS = G::STAGES;
        pl.smem = G::SMEM;
        pl.wall_tiles = false;
        pl.threads = G::THREADS;
        pl.nstrips = (P.nx + G::WOUT - 1) / G::WOUT;
        const int slots = ctas * std::max(1, sm_count);
        int nsegs = std::max(1, slots / pl.nstrips);
        nsegs = std::min(nsegs, std::max(1, P.ny / 8));
        pl.H = (P.ny + nsegs - 1) / nsegs;
        pl.nsegs = (P.ny + pl.H - 1) / pl.H;
        pl.ok = true;
        return pl;
    }

    // The Gibbs-Duhem force form has its own single-pass instance for FP64 and FP32 storage
    // and N <= 3 (the paper's polymer binary and ternary); elsewhere it runs staged.
    template <int N>
    static constexpr bool gd_single_pass()
    {
        return (std::is_same<T, float>::value || std::is_same<T, double>::value) && N <= 3;
    }
    template <int N>
    static FusedPlan plan_n(const Problem& P, int sm_count)
    {
        if (P.force_form == FORCE_GIBBS_DUHEM) {
            if constexpr (gd_single_pass<N>()) return plan_k<N, true>(P, sm_count);
            FusedPlan none{};
            none.ok = false;
            return none;
        }
        return plan_k<N, false>(P, sm_count);
    }

    static FusedPlan plan_fused(const Problem& P, int sm_count)
    {
        FusedPlan none{};
        none.ok = false;
        switch (P.N) {
            case 1: return plan_n<1>(P, sm_count);
            case 2: return plan_n<2>(P, sm_count);
            case 3: return plan_n<3>(P, sm_count);
            case 4: return plan_n<4>(P, sm_count);
            case 5: return plan_n<5>(P, sm_count);
            case 6: return plan_n<6>(P, sm_count);
            case 7: return plan_n<7>(P, sm_count);
            case 8: return plan_n<8>(P, sm_count);
            default: return none;
        }
    }

    // Walls on the single pass.  A row's new state reaches three rows of the old one (the
    // pull of rho^s two rows away, which nu^s one row away needs), so rows 3 .. ny - 4 of
    // k_march, which treats y as periodic, are already those of the walled lattice.  The
    // wall-aware staged kernels then rewrite the three rows next to each wall, from the
    // bands of fields they need (rho^s on five rows, nu^s on four); ghosts included.
    template <int N>
    static cudaError_t wall_rows(StepParams<C> p, const Scratch& sc, const T* fin, T* fout,
                                 cudaStream_t st)
    {
        const auto band = [&](int rows) { return 2 * rows >= p.ny ? 0LL : (long long)rows * p.nx; };
        const auto blocks = [&]() { return site_blocks(p.band ? 2 * p.band : p.S); };
        p.band = band(5);
        k_density<T, N, true><<<blocks(), SITE_THREADS, 0, st>>>(fin, (C*)sc.rho_s, p);
        p.band = band(4);
        k_potential<C, N, true><<<blocks(), SITE_THREADS, 0, st>>>((const C*)sc.rho_s, (C*)sc.nu, p);
        p.band = band(3);
        k_collide<T, N, true><<<blocks(), SITE_THREADS, 0, st>>>(fin, fout, (const C*)sc.rho_s,
                                                            (const C*)sc.nu, p);
        return cudaGetLastError();
    }

    // The same rows by one launch of tiles: us a step against the three band launches: 1500 x 1200 x 3
    // FP32 80 / 95, 1024 x 2048 x 5 148 / 179, 1000 x 700 x 3 BF16 45.5 / 67.8.
    static bool wall_tiles_fit(const Problem& P)
    {
        return P.walls && P.force_form == 0 && P.ny >= 2 * TILE_WALL_ROWS &&
               P.N * 32 * TILE_WALL_ROWS <= tile_max_threads<T>() && (long long)P.plane * P.N < (1LL << 31);
    }
    template <int N>
    static cudaError_t wall_tiles(const StepParams<C>& p, const T* fin, T* fout, cudaStream_t st)
    {
        if constexpr (Storage<T>::shifted && N * 32 * TILE16_WALL_ROWS <= tile_max_threads<T>()) {
            return launch_dependent(k_tile16_walls<T, N>, dim3((p.nx + 31) / 32, 2), N * 32 * TILE16_WALL_ROWS,
                                    sizeof(C) * tile_smem_values(N, 32, TILE16_WALL_ROWS, false), st, fin, fout, p);
        } else if constexpr (N * 32 * TILE_WALL_ROWS <= tile_max_threads<T>()) {
            return launch_dependent(k_tile_walls<T, N>, dim3((p.nx + 31) / 32, 2), N * 32 * TILE_WALL_ROWS,
                                    sizeof(C) * tile_smem_values(N, 32, TILE_WALL_ROWS, false), st, fin, fout, p);
        }
        return cudaErrorInvalidValue;
    }

    static cudaError_t step_fused(const Problem& P, const Scratch& sc, const FusedPlan& pl,
                                  const CUtensorMap* tmap_in, const CUtensorMap* tmapr_in,
                                  const CUtensorMap* tmapw_out, const CUtensorMap* tmapwr_out,
                                  const void* fin, void* fout, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        const dim3 grid(pl.nstrips, pl.nsegs);
        const CUtensorMap& tr = Storage<T>::shifted ? *tmapr_in : *tmap_in;
        const CUtensorMap& tw = pl.out_w > 0 ? *tmapw_out : *tmap_in;
        const CUtensorMap& twr = (pl.out_w > 0 && Storage<T>::shifted) ? *tmapwr_out : *tmap_in;
        MCLB_DISPATCH_N(P.N, {
            bool launched = false;
            if constexpr (gd_single_pass<NN>()) {
                if (P.force_form == FORCE_GIBBS_DUHEM) {
                    k_march<T, NN, true><<<grid, pl.threads, pl.smem, st>>>(*tmap_in, tr, tw, twr,
                                                                          (T*)fout, p, pl.H);
                    launched = true;
                }
            }
            if (!launched)
                k_march<T, NN><<<grid, pl.threads, pl.smem, st>>>(*tmap_in, tr, tw, twr, (T*)fout, p, pl.H);
            const long long ghosts = (long long)NN * P.ny * (Q + (Storage<T>::shifted ? 1 : 0)) * 2 * P.hx;
            k_ghosts<T><<<(unsigned)((ghosts + 255) / 256), 256, 0, st>>>((T*)fout, p, NN);
            if (!P.walls) return cudaGetLastError();
            if (pl.wall_tiles) return wall_tiles<NN>(p, (const T*)fin, (T*)fout, st);
            return wall_rows<NN>(p, sc, (const T*)fin, (T*)fout, st);
        });
    }

    static cudaError_t moments(const Problem& P, const Scratch& sc, const void* f, double* rho,
                               double* U, double* mu, double* Pt, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        // Tiles of 14 rows by eight warps: potentials on 16 rows, two a warp.  Six where their
        // shared memory does not fit; two by four warps where the larger ones would leave SMs
        // without one (and FP64 its pipe on those).
        int rows = 14, warps = FIELDS_MAX_WARPS;
        const auto smem = [&](int r) { return sizeof(C) * fields_smem_values(P.N, r); };
        if (smem(rows) > 44 * 1024) rows = 6;
        if (P.S < 152LL * FIELDS_X * rows) {
            rows = 2;
            warps = 4;
        }
        const long long tiles = (long long)((P.nx + FIELDS_X - 1) / FIELDS_X) * ((P.ny + rows - 1) / rows);
        const dim3 grid((unsigned)tiles);   // (at most the 2^31 sites' number)
        MCLB_DISPATCH_N(P.N, {
            // (few sites: smaller blocks, so that every SM has one)
            const int dt = P.S < 152LL * SITE_THREADS ? 64 : SITE_THREADS;
            cudaError_t e = launch_dependent(U ? k_density<T, NN, false, true> : k_density<T, NN>,
                                             dim3((unsigned)((P.S + dt - 1) / dt)), dt, 0, st, (const T*)f,
                                             (C*)sc.rho_s, p, U);
            if (e != cudaSuccess) return e;
            return launch_dependent(k_fields<C, NN>, grid, 32 * warps, smem(rows), st, (const C*)sc.rho_s, rho,
                                    U, mu, Pt, p, rows);
        });
    }

    static cudaError_t conservation(const Problem& P, const Scratch& sc, const void* f, double* out,
                                    cudaStream_t st)
    {
        return conservation_rows(P, sc, f, 0, P.ny, out, st);
    }

    static cudaError_t conservation_rows(const Problem& P, const Scratch& sc, const void* f,
                                         int y0, int nrows, double* out, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        const long long s0 = (long long)y0 * P.nx, s1 = (long long)(y0 + nrows) * P.nx;
        MCLB_DISPATCH_N(P.N, {
            cudaError_t e = fields_n<NN>(p, sc, (const T*)f, st);
            if (e != cudaSuccess) return e;
            if (sc.partial_cap < (size_t)REDUCE_BLOCKS * (NN + 4)) return cudaErrorInvalidValue;
            k_conservation<T, NN><<<REDUCE_BLOCKS, SITE_THREADS, 0, st>>>(
                (const T*)f, (const C*)sc.rho_s, (const C*)sc.nu, sc.partial, s0, s1, p);
            k_reduce_partials<<<1, SITE_THREADS, 0, st>>>(sc.partial, REDUCE_BLOCKS, NN + 4, out);
            return cudaGetLastError();
        });
    }

    static cudaError_t compositions(const Problem& P, const Scratch& sc, const void* f, double* phi,
                                    double* bulk, double tol, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_density<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>((const T*)f,
                                                                         (C*)sc.rho_s, p);
            k_compositions<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(
                (const C*)sc.rho_s, phi, bulk, tol, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t get_state(const Problem& P, const Scratch& sc, const void* f, double* out,
                                 cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_get_state<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>((const T*)f, out, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t set_state(const Problem& P, const Scratch& sc, const double* in, void* f,
                                 cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_set_state<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(in, (T*)f, p);
            return cudaGetLastError();
        });
    }

    // Per-component mass compensation (mass.cuh), either lattice: record != 0 stores the
    // FP64 mass of every component of f in sc.mass_ref; record == 0 restores it.
    static cudaError_t mass(const Problem& P, const Scratch& sc, void* f, int record, cudaStream_t st)
    {
        MassView v{};
        v.q = P.lattice == LATTICE_D1Q3 ? 3 : (P.lattice == LATTICE_D3Q19 ? Q19 : Q);
        v.lines = (int)(P.S / P.nx) * v.q;   // (layers x) rows x velocities
        v.rlines = Storage<T>::shifted ? P.ny : 0;
        v.comp_stride = P.plane;
        v.pitch = P.pitch;
        v.rbytes = P.rbytes;
        v.S = P.S;
        v.first = P.hx;
        v.nx = P.nx;
        v.span = P.nx + 2 * P.hx;
        v.vec = (P.hx * sizeof(T)) % 16 == 0 && (P.pitch * sizeof(T)) % 16 == 0 &&
                P.rbytes % 16 == 0 && (P.hx * sizeof(float)) % 16 == 0 &&
                (P.pitch * sizeof(float)) % 16 == 0;
        k_mass_partials<T><<<dim3(MASS_BLOCKS, P.N), MASS_THREADS, 0, st>>>((const T*)f, v, sc.partial);
        const unsigned gx = record ? 1u : (unsigned)std::min(P.ny, 1024);
        k_mass_apply<T><<<dim3(gx, P.N), MASS_THREADS, 0, st>>>((T*)f, v, sc.partial, sc.mass_ref,
                                                                record);
        return cudaGetLastError();
    }
};

// The tile schedule (tile.cuh) for one storage type.
template <typename T>
struct TileLaunch {
    using C = typename Storage<T>::C;

    // Most sites x components for which a tile kernel beats the march (measured on both sides of
    // each line, us per step, tile / march; between walls the march has one launch more):
    //   FP64: it runs at the FP64 pipe's rate on every SM with fewer FP64 instructions a site:
    //     64 x 64 x 2 9.65 / 107, 2048^2 x 2 2323 / 2613, 2048^2 x 3 3474 / 3802, 500^2 x 6 533 / 850, 1700^2
    //     x 6 6110 / 10642, x 7 7247 / 12506, x 8 8172 / 14210, Gibbs-Duhem 900^2 x 3 728 / 869: every
    //     size, but 700^2 x 4 610 / 621, 860^2 x 4 912 / 901 and 500^2 x 5 399 / 415, 700^2 x 5 777 /
    //     757; walls 700^2 x 4 609 / 646, 850^2 x 4 906 / 906, 700^2 x 5 778 / 783
    //   FP32 (k_rows): 1000^2 x 1 18.1 / 26.3; 700^2 x 2 20.5 / 22.3, 1024^2 x 2 38 / 37;
    //     512 x 384 x 3 14.7 / 18.5, 700 x 600 x 3 29.8 / 25.7; 400^2 x 4 21.7 / 20.1;
    //     300^2 x 5 13.5 / 19.4, 500 x 450 x 5 24.9 / 23.6.  k_tile, six and more: 300^2 x 6 20.0 / 23.1
    //   FP32 between walls (the march with its rows next to them by tiles): 1500^2 x 1 42 / 57; 800^2 x 2
    //     26.2 / 31.4, 1000^2 x 2 39.4 / 38.7; 800^2 x 3 39.0 / 40.5; 600^2 x 4 33.3 / 33.8, 700^2 x 4 43.2 /
    //     41.1; 500^2 x 5 29.3 / 30.2, 600^2 x 5 42.4 / 38.6; 350^2 x 6 26.4 / 29.2, 400^2 x 6 33.1 / 33.0;
    //     350^2 x 7 31.5 / 32.4, 400^2 x 7 40.0 / 37.3; 300^2 x 8 28.6 / 33.7, 350^2 x 8 37.7 / 34.3
    //   16-bit (k_tile16): 540^2 x 2 19.7 / 21.4, 440^2 x 3 20.7 / 22.1, 340^2 x 5 25.5 / 28.4, 270^2 x 8 31.1 /
    //     41.8; walls (the march with its rows next to them by tiles) 510^2 x 3 27.9, 530^2 x 3 - / 30.0, 440^2
    //     x 4 31.5, 460^2 x 4 - / 34.4, 390^2 x 5 33.8, 410^2 x 5 - / 40.2
    //   FP32 Gibbs-Duhem: 300^2 x 2 10.3 / 15.8, 512 x 384 x 3 22.8 / 18.5
    static long long most(const Problem& P)
    {
        const int N = P.N;
        if (sizeof(C) == 8) {
            if (N == 4) return P.walls ? 2900000 : 2400000;
            if (N == 5) return P.walls ? 2500000 : 1800000;
            return 1LL << 40;
        }
        if (P.force_form == FORCE_GIBBS_DUHEM) return 350000;
        if (Storage<T>::shifted) return P.walls ? 800000 : 600000;
        if (P.walls) {
            constexpr int by_n[NMAX] = {2500000, 1900000, 2200000, 1500000, 1300000, 950000, 900000, 800000};
            return by_n[N - 1];
        }
        return N == 1 ? 2000000 : N == 2 ? 1200000 : N == 4 || N >= 6 ? 550000 : 900000;
    }

    // FP32 above this goes to k_rows, below to k_tile (200 x 100 x 3 5.6 / 6.2 us, 300^2 x 2
    // 7.7 / 7.3, 300^2 x 5 17 / 13.5)
    static constexpr long long ROWS_LEAST = 150000;

    static TilePlan plan(const Problem& P, int)
    {
        TilePlan pl{};
        const bool gd = P.force_form == FORCE_GIBBS_DUHEM;
        if (P.S * P.N > most(P) || (gd && (Storage<T>::shifted || P.N > TILE_GD_NMAX))) return pl;
        if constexpr (std::is_same<T, float>::value) {
            if (!gd && P.S * P.N >= ROWS_LEAST && P.ny >= ROWS_MIN_NY && P.N <= ROWS_NMAX) {
                pl.gx = (P.nx + ROWS_X - 1) / ROWS_X;
                pl.gy = (P.ny + ROWS_Y - 1) / ROWS_Y;
                pl.threads = 32 * ROWS_WPC * P.N;
                pl.ok = pl.gy < 65536;
                return pl;
            }
        }
        // 16 x 8 sites; 8 x 4 where five and more components fill a CTA with fewer sites, and
        // in FP64, whose few operations per clock and SM want every SM busy, below about 100
        // of the larger tiles (100 x 90 x 2 11.4 us, 15.7 with 16 x 8; 160 x 96 x 2 21.2, 20.3)
        const bool small = P.N >= 5 || (sizeof(C) == 8 && P.S < 12800);
        const int ty = small ? 4 : 8;
        pl.lx = small ? 3 : 4;
        pl.ty = ty;
        pl.gx = (P.nx + (1 << pl.lx) - 1) >> pl.lx;
        pl.gy = (P.ny + ty - 1) / ty;
        if (Storage<T>::shifted && P.walls)   // the rows next to each wall are tiles of their own
            pl.gy = P.ny <= TILE16_WALL_ROWS ? 1 : 2 + (std::max(0, P.ny - 2 * TILE16_WALL_ROWS) + ty - 1) / ty;
        pl.threads = P.N * (ty << pl.lx);
        pl.parts = 1;
        if (sizeof(C) == 8 && small && P.N <= 4) {   // a CTA of few warps: twice the threads
            pl.threads *= 2;
            pl.parts = std::min(P.N, 2);
        }
        pl.smem = sizeof(C) * tile_smem_values(P.N, 1 << pl.lx, ty, gd);
        pl.ok = pl.threads <= tile_max_threads<T>() && pl.smem <= 44 * 1024 && pl.gy < 65536 &&
                (long long)P.plane * P.N < (1LL << 31);
        return pl;
    }

    static cudaError_t step(const Problem& P, const Scratch& sc, const TilePlan& pl, const void* fin,
                            void* fout, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        [[maybe_unused]] const C* rs = nullptr;
        if constexpr (!Storage<T>::shifted) {
            if (P.force_form == FORCE_GIBBS_DUHEM) {
                const cudaError_t e = launch_dependent(k_tile_rho<T>, dim3((unsigned)((P.S + 127) / 128), P.N),
                                                       128, 0, st, (const T*)fin, (C*)sc.rho_s, p);
                if (e != cudaSuccess) return e;
                rs = (const C*)sc.rho_s;
            }
        }
        if constexpr (std::is_same<T, float>::value) {
            if (pl.lx == 0)
                MCLB_DISPATCH_N(P.N, {
                    if constexpr (NN <= ROWS_NMAX)
                        return launch_dependent(P.walls ? k_rows<NN, true> : k_rows<NN, false>,
                                                dim3(pl.gx, pl.gy), pl.threads, 0, st, (const T*)fin, (T*)fout, p);
                    return cudaErrorInvalidValue;
                });
        }
        MCLB_DISPATCH_N(P.N, {
            if constexpr (Storage<T>::shifted)
                return launch_dependent(P.walls ? k_tile16<T, NN, true> : k_tile16<T, NN, false>,
                                        dim3(pl.gx, pl.gy), pl.threads, pl.smem, st, (const T*)fin, (T*)fout, p,
                                        pl.lx, pl.ty);
            else
                return launch_dependent(k_tile<T, NN>, dim3(pl.gx, pl.gy), pl.threads, pl.smem, st,
                                        (const T*)fin, (T*)fout, rs, p, pl.lx, pl.ty, pl.parts);
        });
    }
};

// Launchers of the D1Q3 kernels (line3.cuh) for one storage type.
template <typename T>
struct Line3Launch {
    using C = typename Storage<T>::C;
    static constexpr size_t SMEM_CAP = 227 * 1024 - sizeof(StepParams<C>) - 256;

    static int max_resident(int N)
    {
        const size_t per = (size_t)5 * N * sizeof(C);
        return (int)std::min<size_t>(SMEM_CAP / per, (size_t)L3_MAX_SITES);
    }

    static Line3Item<T> item(const Problem& P, const Scratch& sc, void* f0, void* f1)
    {
        Line3Item<T> it{};
        it.p = make_params<C>(P, sc.status);
        it.f[0] = (T*)f0;
        it.f[1] = (T*)f1;
        return it;
    }

    static cudaError_t prepare(const Problem& P, const Scratch& sc, void* const* f)
    {
        const Line3Item<T> it = item(P, sc, f[0], f[1]);
        return cudaMemcpy(sc.line_item, &it, sizeof(it), cudaMemcpyHostToDevice);
    }

    template <int N>
    static cudaError_t resident(const Line3Item<T>* items, int count, int nxmin, int nxmax, int parity,
                                int nsteps, cudaStream_t st)
    {
        if constexpr (std::is_same<T, double>::value) {
            const int c = pieces<N>(count, nxmin, nxmax);
            if (c > 0) return resident64<N>(c, items, count, nxmax, parity, nsteps, st);
        }
        static const cudaError_t attr = cudaFuncSetAttribute(
            k_line3_resident<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_CAP);
        if (attr != cudaSuccess) return attr;
        const size_t smem = Line3Smem<T, N>::bytes(nxmax);
        const int threads = (nxmax + 31) / 32 * 32;
        k_line3_resident<T, N><<<count, threads, smem, st>>>(items, parity, nsteps);
        return cudaGetLastError();
    }

    // CTAs per line for k_line3_resident64 (0: its threads or shared memory do not fit): the
    // count that leaves the busiest SM quarter the fewest warps, whose FP64 instructions are
    // the launch's time (60 lines of 128 sites, N = 2, 1 / 2 / 4 / 8 CTAs: 3.57, 2.66, 2.60,
    // 4.03 us a step; 200 of 100, N = 3: 13.7, 10.5, 10.7, 21.2; 10 of 600, N = 3, 2 / 4 / 8:
    // 14.1, 7.5, 5.1)
    template <int N>
    static int pieces(int count, int nxmin, int nxmax)
    {
        int dev = 0, sms = 1;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        int best = 0;
        long long least = 0;
        for (int c = 1; c <= 8 && c <= nxmin; c *= 2) {
            const int n = (nxmax + c - 1) / c, stride = (n + 31) / 32 * 32;
            if (N * stride > L3_MAX_SITES || Line3Smem<T, N>::bytes64(n) > SMEM_CAP64) continue;
            const long long ctas = ((long long)count * c + sms - 1) / sms;
            const long long cost = (ctas * (N * stride / 32) + 3) / 4;
            if (best == 0 || cost < least) {
                best = c;
                least = cost;
            }
        }
        return best;
    }

    static constexpr size_t SMEM_CAP64 = 227 * 1024 - round_up_sz(sizeof(StepParams<C>) + LOG64_ROWS * sizeof(Log64Row) + 16, 128);

    template <int N>
    static cudaError_t resident64(int c, const Line3Item<T>* items, int count, int nxmax, int parity,
                                  int nsteps, cudaStream_t st)
    {
        static const cudaError_t attr = cudaFuncSetAttribute(
            k_line3_resident64<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_CAP64);
        if (attr != cudaSuccess) return attr;
        const int n = (nxmax + c - 1) / c, stride = (n + 31) / 32 * 32;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)c;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)(count * c));
        cfg.blockDim = dim3((unsigned)(N * stride));
        cfg.dynamicSmemBytes = Line3Smem<T, N>::bytes64(n);
        cfg.stream = st;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, k_line3_resident64<N>, items, parity, nsteps, stride);
    }

    template <int N>
    static cudaError_t tile(const StepParams<C>& p, const void* fin, void* fout, cudaStream_t st)
    {
        const unsigned blocks = (unsigned)((p.nx + L3_TILE - 5) / (L3_TILE - 4));
        k_line3_tile<T, N><<<blocks, L3_TILE, 0, st>>>((const T*)fin, (T*)fout, p);
        return cudaGetLastError();
    }

    static unsigned line_blocks(int nx) { return (unsigned)((nx + SITE_THREADS - 1) / SITE_THREADS); }

    static cudaError_t init(const Problem& P, const Scratch& sc, const double* rho, const double* u,
                            void* f, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_line3_init<T, NN><<<line_blocks(P.nx), SITE_THREADS, 0, st>>>(rho, u, (T*)f, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t step(const Problem& P, const Scratch& sc, void* const* f, int* cur,
                            long nsteps, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        const bool res = P.nx <= max_resident(P.N);
        MCLB_DISPATCH_N(P.N, {
            while (nsteps > 0) {
                cudaError_t e;
                if (res) {
                    const int k = (int)std::min<long>(nsteps, L3_CHUNK);
                    e = resident<NN>((const Line3Item<T>*)sc.line_item, 1, P.nx, P.nx, *cur, k, st);
                    nsteps -= k;
                } else {
                    e = tile<NN>(p, f[*cur], f[*cur ^ 1], st);
                    nsteps -= 1;
                }
                if (e != cudaSuccess) return e;
                *cur ^= 1;
            }
            return cudaSuccess;
        });
    }

    static cudaError_t moments(const Problem& P, const Scratch& sc, const void* f, double* rho,
                               double* U, double* mu, double* Pt, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_line3_moments<T, NN><<<line_blocks(P.nx), SITE_THREADS, 0, st>>>((const T*)f, rho, U,
                                                                               mu, Pt, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t conservation(const Problem& P, const Scratch& sc, const void* f, double* out,
                                    cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            if (sc.partial_cap < (size_t)REDUCE_BLOCKS * (NN + 4)) return cudaErrorInvalidValue;
            k_line3_conservation<T, NN><<<REDUCE_BLOCKS, SITE_THREADS, 0, st>>>((const T*)f,
                                                                                sc.partial, p);
            k_reduce_partials<<<1, SITE_THREADS, 0, st>>>(sc.partial, REDUCE_BLOCKS, NN + 4, out);
            return cudaGetLastError();
        });
    }

    static cudaError_t compositions(const Problem& P, const Scratch& sc, const void* f, double* phi,
                                    double* bulk, double tol, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_line3_compositions<T, NN><<<line_blocks(P.nx), SITE_THREADS, 0, st>>>(
                (const T*)f, phi, bulk, tol, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t get_state(const Problem& P, const Scratch& sc, const void* f, double* out,
                                 cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_line3_get_state<T, NN><<<line_blocks(P.nx), SITE_THREADS, 0, st>>>((const T*)f, out, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t set_state(const Problem& P, const Scratch& sc, const double* in, void* f,
                                 cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k_line3_set_state<T, NN><<<line_blocks(P.nx), SITE_THREADS, 0, st>>>(in, (T*)f, p);
            return cudaGetLastError();
        });
    }

    // ---- batches of lines with one N
    struct Group {
        int N = 0;
        Line3Item<T>* d_items = nullptr;     // lines the resident kernel holds
        int nres = 0, nxmin = INT32_MAX, nxmax = 1;
        std::vector<Line3Item<T>> longs;     // lines stepped with the tile kernel
        std::vector<size_t> long_bytes;
    };

    static void* batch_create(int N, int count, const Problem* probs, const Scratch* scs,
                              void* const* fa, void* const* fb, cudaStream_t st)
    {
        auto* g = new (std::nothrow) Group();
        if (!g) return nullptr;
        g->N = N;
        std::vector<Line3Item<T>> res;
        for (int k = 0; k < count; ++k) {
            const Line3Item<T> it = item(probs[k], scs[k], fa[k], fb[k]);
            if (probs[k].nx <= max_resident(N)) {
                res.push_back(it);
                g->nxmin = std::min(g->nxmin, probs[k].nx);
                g->nxmax = std::max(g->nxmax, probs[k].nx);
            } else {
                g->longs.push_back(it);
                g->long_bytes.push_back((size_t)N * 3 * probs[k].nx * sizeof(T));
            }
        }
        g->nres = (int)res.size();
        if (g->nres > 0) {
            if (cudaMalloc(&g->d_items, sizeof(Line3Item<T>) * res.size()) != cudaSuccess ||
                cudaMemcpyAsync(g->d_items, res.data(), sizeof(Line3Item<T>) * res.size(),
                                cudaMemcpyHostToDevice, st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess) {
                cudaGetLastError();
                batch_destroy(g);
                return nullptr;
            }
        }
        return g;
    }

    static cudaError_t batch_step(void* gv, int parity, int nsteps, cudaStream_t st)
    {
        auto* g = static_cast<Group*>(gv);
        MCLB_DISPATCH_N(g->N, {
            if (g->nres > 0) {
                cudaError_t e = resident<NN>(g->d_items, g->nres, g->nxmin, g->nxmax, parity, nsteps, st);
                if (e != cudaSuccess) return e;
            }
            for (size_t k = 0; k < g->longs.size(); ++k) {
                const Line3Item<T>& it = g->longs[k];
                int c = parity;
                for (int t = 0; t < nsteps; ++t, c ^= 1) {
                    cudaError_t e = tile<NN>(it.p, it.f[c], it.f[c ^ 1], st);
                    if (e != cudaSuccess) return e;
                }
                if (c == parity) {   // an even number of steps: the result goes to parity ^ 1
                    cudaError_t e = cudaMemcpyAsync(it.f[parity ^ 1], it.f[parity], g->long_bytes[k],
                                                    cudaMemcpyDeviceToDevice, st);
                    if (e != cudaSuccess) return e;
                }
            }
            return cudaSuccess;
        });
    }

    static int batch_launches(const void* gv)
    {
        auto* g = static_cast<const Group*>(gv);
        return (g->nres > 0 ? 1 : 0) + (int)g->longs.size();
    }

    static void batch_destroy(void* gv)
    {
        auto* g = static_cast<Group*>(gv);
        if (!g) return;
        if (g->d_items) cudaFree(g->d_items);
        delete g;
    }

    static const LatticeTable* table()
    {
        static const LatticeTable t = [] {
            LatticeTable x{};
            x.max_resident = &max_resident;
            x.item_bytes = sizeof(Line3Item<T>);
            x.prepare = &prepare;
            x.init = &init;
            x.step = &step;
            x.moments = &moments;
            x.conservation = &conservation;
            x.compositions = &compositions;
            x.get_state = &get_state;
            x.set_state = &set_state;
            x.batch_create = &batch_create;
            x.batch_step = &batch_step;
            x.batch_launches = &batch_launches;
            x.batch_destroy = &batch_destroy;
            return x;
        }();
        return &t;
    }
};

// Launchers of the D3Q19 kernels (cube.cuh) for one storage type: the staged step (three
// launches) and the diagnostics; no batches.
template <typename T>
struct Launch19 {
    using C = typename Storage<T>::C;

    static int max_resident(int) { return 0; }
    static cudaError_t prepare(const Problem&, const Scratch&, void* const*) { return cudaSuccess; }

    // The march (cube_march.cuh) after a density pass: tiles of M3_OUT_X x M3_OUT_Y, z
    // segments of H planes.  The four warm-up planes of a segment collide nothing and cost about
    // two; w waves of resident CTAs, which do not run in step, end about one CTA later and lose
    // part of a last wave that is not full.  The segment count that minimises (w + 1 + 0.3 (ceil w
    // - w)) (H + 2) is taken (us per step at 5 / 7 / 10 / 14 / 16 / 20 segments: 256^3 x 3 2351 / 2273 /
    // 2168 / 2090 / 2095 / 2057; 192^3 x 3 938 / 902 / 873 / 855 / 867 / 887; 256 x 200 x 220 x 2 1124
    // / 985 / 1031 / 979 / 996 / 1000; whole waves x (H + 4) took 7 in all three).  Not for N >
    // M3_NMAX, the Gibbs-Duhem reading (it needs grad rho on the density planes the next
    // iteration overwrites) or 19 S >= 2^31 (32-bit offsets).
    template <int N>
    static int plan_n(Problem& P, int sm_count)
    {
        if constexpr (N > M3_NMAX) {
            return 0;
        } else {
            if (P.force_form != 0 || 19.0 * (double)P.S >= 2147483647.0) return 0;
            const int smem = (int)m3_smem_bytes<C, N>();
            if (cudaFuncSetAttribute(k19_march<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     smem) != cudaSuccess)
                return -1;
            int ctas = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, k19_march<T, N>, M3_THREADS,
                                                              smem) != cudaSuccess)
                return -1;
            if (ctas < 1) return 0;
            const long long tx = (P.nx + M3_OUT_X - 1) / M3_OUT_X, ty = (P.ny + M3_OUT_Y - 1) / M3_OUT_Y;
            const long long slots = (long long)ctas * std::max(1, sm_count);
            int best = 1;
            double best_cost = -1.0;
            for (int nseg = 1; nseg <= std::max(1, P.nz / 4); ++nseg) {
                const long long H = (P.nz + nseg - 1) / nseg, segs = (P.nz + H - 1) / H;
                const double w = (double)(tx * ty * segs) / (double)slots;
                const double cost = (w + 1.0 + 0.3 * (std::ceil(w) - w)) * (double)(H + 2);
                if (best_cost < 0 || cost < best_cost) {
                    best_cost = cost;
                    best = nseg;
                }
            }
            const int H = (P.nz + best - 1) / best;
            P.grid3[0] = (int)tx;
            P.grid3[1] = (int)ty;
            P.grid3[2] = (P.nz + H - 1) / H;
            P.seg3 = H;
            return 1;
        }
    }
    // The march pays in FP32 from a number of site-components on, below which its CTAs are too few, each
    // with its dependent plane iterations (us per step, march / staged: 192^3 x 1 390 / 382, 224^3 x 1
    // 578 / 603; 100 x 90 x 70 x 2 66 / 73, 192^3 x 2 627 / 723; 40 x 24 x 30 x 3 37 / 10, 64^3 x 3 53 / 42,
    // 96^3 x 3 131 / 140, 192^3 x 3 873 / 1055; 96^3 x 4 189 / 184, 128 x 120 x 100 x 4 311 / 311, 128^3 x 4
    // 406 / 419, 192^3 x 4 1310 / 1418), and not in FP64, which the FP64 pipe bounds and whose pulled
    // values spill (64^3 x 3 1063 / 357, 128^3 x 4 6082 / 3547).
    static bool pays(const Problem& P)
    {
        const long long least = P.N == 1 ? 8500000 : P.N == 4 ? 6200000 : 1200000;
        return sizeof(C) == 4 && P.N <= M3_NMAX && P.S * P.N >= least;
    }

    static int plan(Problem& P, int sm_count)
    {
        switch (P.N) {
            case 1: return plan_n<1>(P, sm_count);
            case 2: return plan_n<2>(P, sm_count);
            case 3: return plan_n<3>(P, sm_count);
            case 4: return plan_n<4>(P, sm_count);
            default: return 0;
        }
    }

    static cudaError_t init(const Problem& P, const Scratch& sc, const double* rho, const double* u,
                            void* f, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k19_init<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(rho, u, (T*)f, p);
            return cudaGetLastError();
        });
    }

    // density and potential fields of state f into the scratch
    template <int N>
    static cudaError_t fields_n(const StepParams<C>& p, const Scratch& sc, const T* f, cudaStream_t st)
    {
        k19_density<T, N><<<site_blocks(p.S), SITE_THREADS, 0, st>>>(f, (C*)sc.rho_s, (C*)sc.js, p);
        k19_potential<C, N><<<site_blocks(p.S), SITE_THREADS, 0, st>>>((const C*)sc.rho_s,
                                                                        (C*)sc.nu, p);
        return cudaGetLastError();
    }

    static cudaError_t step(const Problem& P, const Scratch& sc, void* const* f, int* cur,
                            long nsteps, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            if constexpr (NN <= M3_NMAX) {
                if (P.seg3 > 0) {
                    const dim3 grid(P.grid3[0], P.grid3[1], P.grid3[2]);
                    // dependent launches hide the launch, but the CTAs that come early crowd the
                    // last wave (100 x 90 x 70 x 2 75 -> 70 us, 192^3 x 3 923 -> 941)
                    const bool dependent = P.S * P.N < 6000000;
                    for (; nsteps > 0; --nsteps) {
                        const T* fi = (const T*)f[*cur];
                        cudaError_t e;
                        if (dependent) {
                            e = launch_dependent(k19_density<T, NN>, dim3(site_blocks(P.S)), SITE_THREADS,
                                                 0, st, fi, (C*)sc.rho_s, nullptr, p, nullptr);
                            if (e == cudaSuccess)
                                e = launch_dependent(k19_march<T, NN>, grid, M3_THREADS, m3_smem_bytes<C, NN>(),
                                                     st, fi, (T*)f[*cur ^ 1], (const C*)sc.rho_s, p, P.seg3);
                        } else {
                            k19_density<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(
                                fi, (C*)sc.rho_s, nullptr, p);
                            k19_march<T, NN><<<grid, M3_THREADS, m3_smem_bytes<C, NN>(), st>>>(
                                fi, (T*)f[*cur ^ 1], (const C*)sc.rho_s, p, P.seg3);
                            e = cudaGetLastError();
                        }
                        if (e != cudaSuccess) return e;
                        *cur ^= 1;
                    }
                    return cudaSuccess;
                }
            }
            // the staged step; few sites: smaller blocks, so that every SM has one
            const int th = P.S < 4LL * 152 * SITE_THREADS ? 64 : SITE_THREADS;
            const dim3 grid((unsigned)((P.S + th - 1) / th));
            for (; nsteps > 0; --nsteps) {
                cudaError_t e = launch_dependent(k19_density<T, NN>, grid, th, 0, st, (const T*)f[*cur],
                                                 (C*)sc.rho_s, (C*)sc.js, p, nullptr);
                if (e == cudaSuccess)
                    e = launch_dependent(k19_potential<C, NN>, grid, th, 0, st, (const C*)sc.rho_s, (C*)sc.nu, p);
                if (e == cudaSuccess)
                    e = launch_dependent(k19_collide<T, NN>, grid, th, 0, st, (const T*)f[*cur],
                                         (T*)f[*cur ^ 1], (const C*)sc.rho_s, (const C*)sc.js, (const C*)sc.nu, p);
                if (e != cudaSuccess) return e;
                *cur ^= 1;
            }
            return cudaSuccess;
        });
    }

    static cudaError_t moments(const Problem& P, const Scratch& sc, const void* f, double* rho,
                               double* U, double* mu, double* Pt, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k19_density<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>((const T*)f, (C*)sc.rho_s,
                                                                                nullptr, p, U);
            if (U)
                k19_potential<C, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>((const C*)sc.rho_s,
                                                                                (C*)sc.nu, p);
            k19_moments<C, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(
                (const C*)sc.rho_s, (const C*)sc.nu, rho, U, mu, Pt, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t conservation(const Problem& P, const Scratch& sc, const void* f, double* out,
                                    cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            if (sc.partial_cap < (size_t)REDUCE_BLOCKS * (NN + 6)) return cudaErrorInvalidValue;
            cudaError_t e = fields_n<NN>(p, sc, (const T*)f, st);
            if (e != cudaSuccess) return e;
            k19_conservation<T, NN><<<REDUCE_BLOCKS, SITE_THREADS, 0, st>>>(
                (const T*)f, (const C*)sc.rho_s, (const C*)sc.nu, sc.partial, p);
            k_reduce_partials<<<1, SITE_THREADS, 0, st>>>(sc.partial, REDUCE_BLOCKS, NN + 6, out);
            return cudaGetLastError();
        });
    }

    static cudaError_t compositions(const Problem& P, const Scratch& sc, const void* f, double* phi,
                                    double* bulk, double tol, cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k19_density<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>((const T*)f,
                                                                          (C*)sc.rho_s, nullptr, p);
            k19_compositions<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(
                (const C*)sc.rho_s, phi, bulk, tol, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t get_state(const Problem& P, const Scratch& sc, const void* f, double* out,
                                 cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k19_get_state<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>((const T*)f, out, p);
            return cudaGetLastError();
        });
    }

    static cudaError_t set_state(const Problem& P, const Scratch& sc, const double* in, void* f,
                                 cudaStream_t st)
    {
        const auto p = make_params<C>(P, sc.status);
        MCLB_DISPATCH_N(P.N, {
            k19_set_state<T, NN><<<site_blocks(P.S), SITE_THREADS, 0, st>>>(in, (T*)f, p);
            return cudaGetLastError();
        });
    }

    static const LatticeTable* table()
    {
        static const LatticeTable t = [] {
            LatticeTable x{};
            x.max_resident = &max_resident;
            x.plan = &plan;
            x.pays = &pays;
            x.item_bytes = 0;
            x.prepare = &prepare;
            x.init = &init;
            x.step = &step;
            x.moments = &moments;
            x.conservation = &conservation;
            x.compositions = &compositions;
            x.get_state = &get_state;
            x.set_state = &set_state;
            return x;
        }();
        return &t;
    }
};

// The kernel table of one storage type is assembled from three parts, each instantiated
// in a translation unit of its own (prec_<type>_<part>.cu) so that
// the build compiles them in parallel; prec_<type>.cu puts the table together.
template <typename T>
inline void table_base(KernelTable& t, CUtensorMapDataType tt)
{
    t.storage_bytes = sizeof(T);
    t.shifted = Storage<T>::shifted;
    t.tma_type = tt;
    t.hx = (int)std::max<size_t>(4, 16 / sizeof(T));
    t.line3 = nullptr;
    t.d3q19 = nullptr;
}

// single handles on D2Q9: the single pass
template <typename T>
inline void fill_march(KernelTable& t)
{
    t.plan_fused = &Launch<T>::plan_fused;
    t.wall_tiles_fit = &Launch<T>::wall_tiles_fit;
    t.step_fused = &Launch<T>::step_fused;
}

// single handles on D2Q9: small tiles
template <typename T>
inline void fill_tile(KernelTable& t)
{
    t.plan_tile = &TileLaunch<T>::plan;
    t.step_tile = &TileLaunch<T>::step;
}

// single handles on D2Q9: the staged schedule and the diagnostics
template <typename T>
inline void fill_staged(KernelTable& t)
{
    t.init = &Launch<T>::init;
    t.step_staged = &Launch<T>::step_staged;
    t.moments = &Launch<T>::moments;
    t.conservation = &Launch<T>::conservation;
    t.conservation_rows = &Launch<T>::conservation_rows;
    t.compositions = &Launch<T>::compositions;
    t.get_state = &Launch<T>::get_state;
    t.set_state = &Launch<T>::set_state;
    t.mass = &Launch<T>::mass;
}

// batches of D2Q9 instances
template <typename T>
inline void fill_batch(KernelTable& t)
{
    t.batch_create = &batch_group_create<T>;
    t.batch_step = &batch_group_step<T>;
    t.batch_launches = &batch_group_launches<T>;
    t.batch_tune = &batch_group_tune<T>;
    t.batch_waves = &batch_group_waves<T>;
    t.batch_destroy = &batch_group_destroy<T>;
    t.narrow_boxes = &batch_narrow_boxes<T>;
    t.batch_force = &batch_group_force<T>;
}

// the D1Q3 lattice (FP64 and FP32 storage)
template <typename T>
inline void fill_line3(KernelTable& t)
{
    static_assert(!Storage<T>::shifted, "D1Q3 stores FP64 or FP32");
    t.line3 = Line3Launch<T>::table();
}

// the D3Q19 lattice (FP64 and FP32 storage)
template <typename T>
inline void fill_cube(KernelTable& t)
{
    static_assert(!Storage<T>::shifted, "D3Q19 stores FP64 or FP32");
    t.d3q19 = Launch19<T>::table();
}

}  // namespace mclb
