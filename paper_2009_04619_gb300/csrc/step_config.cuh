// Launch configuration of the fused step kernel: tile shape, ring depths and
// the z-chunk decomposition.  Everything that decides the kernel's memory
// traffic lives here and in step_kernel.cuh.
#pragma once
#include <cuda.h>

#include <algorithm>

#include "step_kernel.cuh"

namespace sgb {

// Tile configuration (build-time): threads in x (4 points each), threads in y,
// rows per thread, u-ring stages, (u^{n-1}, m, phi)-ring stages, min CTAs/SM.
#ifndef SGB_TXT
#define SGB_TXT 16
#endif
#ifndef SGB_TYT
#define SGB_TYT 8
#endif
#ifndef SGB_TY
#define SGB_TY 2
#endif
#ifndef SGB_NU
#define SGB_NU 9
#endif
#ifndef SGB_NP
#define SGB_NP 4
#endif
#ifndef SGB_MINB
#define SGB_MINB 2
#endif
// L2 promotion of the tensor maps: the u^n box with its x-y halo (the
// halos are shared with neighbouring tiles, so wider L2 fills are reused),
// and the halo-free tiles (u^{n-1}, m, phi, ...), whose rows are whole 32-byte
// sectors that no other tile reads: promoting those fetched sectors nobody
// used (measured on 256^3 + 16-point PML: 14 MB less DRAM read per step
// without promotion, 2% faster on 512^3).
#ifndef SGB_L2PROMO
#define SGB_L2PROMO CU_TENSOR_MAP_L2_PROMOTION_L2_256B
#endif
#ifndef SGB_L2PROMO_P
#define SGB_L2PROMO_P CU_TENSOR_MAP_L2_PROMOTION_NONE
#endif
// Two tile shapes of as many points: 64 x 16, whose rows are whole 256-byte
// lines, and 32 x 32.  choose_decomposition takes one of them per grid.
using Cfg = TileCfg<SGB_TXT, SGB_TYT, SGB_TY, SGB_NU, SGB_NP, SGB_MINB>;
using CfgSq = TileCfg<SGB_TXT / 2, 2 * SGB_TYT, SGB_TY, SGB_NU, SGB_NP, SGB_MINB>;

// How a step of one grid is launched (the tile counts and zc are in StepArgs).
struct StepGrid {
    int ctas = 0;
    bool square = false;  // CfgSq instead of Cfg
};

// f(C{}) with the grid's tile configuration.
template <class F>
auto with_tile(const StepGrid &sg, F f)
{
    return sg.square ? f(CfgSq{}) : f(Cfg{});
}

// Estimated time of one step with tiles C and the z-chunk length that minimises
// it, in planes of an interior tile per CTA slot: waves x (chunk + 4 planes of
// priming) x (1 + 0.2 x the share of tile planes in the PML).  With 16-bit storage
// a partly filled wave after a full one counts half: CTAs of different cost refill
// their slots as they finish (400^3 bf16: 201 us with the 40 planes it then takes,
// 204 with 25; in fp32 a whole wave is the better guess, 343 x 229 x 205: 76 us with
// 21 planes, 77.5 with 35).  Alone in one wave, the dearest CTA decides.  Chunks of 64 x 16
// and 16-bit tiles have at most 40 planes: neighbouring CTAs drift apart in z
// over longer ones and their shared halos fall out of L2 (512^3: 22-40-plane
// chunks move ~10% fewer DRAM bytes than 74-plane ones).  The fp32 32 x 32 tiles
// have twice the row ends per point and lose more to it (512^3: 414 us with 40
// planes, 405 with 24): 30 planes, or 36 in a single wave.
template <class C, class T>
double plan_chunks(const StepArgs &a, int slots, int *zc_out)
{
    constexpr double part = sizeof(T) == 4 ? 1.0 : 0.5;  // a partly filled wave
    constexpr bool short_chunks = C::BX < Cfg::BX && sizeof(T) == 4;
    const int tx = (a.Nx + C::BX - 1) / C::BX, ty = (a.Ny + C::BY - 1) / C::BY;
    const int tiles = tx * ty;
    double pml = 0.0, pml_one = 0.0;  // PML share of all tile planes; of the dearest CTA's
    if (a.nb > 0) {
        const int ix = std::max((a.Nx - a.nb) / C::BX - (a.nb + C::BX - 1) / C::BX, 0);
        const int iy = std::max((a.Ny - a.nb) / C::BY - (a.nb + C::BY - 1) / C::BY, 0);
        const double zshare = std::min(1.0, 2.0 * a.nb / a.Nz);
        const double xy = 1.0 - double(ix) * iy / tiles;
        pml = xy + (1.0 - xy) * zshare;
        pml_one = xy > 0.0 ? 1.0 : zshare;
    }
    const int cmax = std::max(a.Nz / 4, 1);
    double best = 1e300;
    *zc_out = a.Nz;
    int last = 0;
    for (int c = 1; c <= cmax; ++c) {
        const int zc = (a.Nz + c - 1) / c;
        if (zc == last) continue;
        last = zc;
        const int units = tiles * ((a.Nz + zc - 1) / zc);
        const bool one = units <= slots;
        if (zc > (short_chunks ? (one ? 36 : 30) : 40) && c < cmax) continue;
        const double w = double(units) / slots;
        const double waves = one ? 1.0 : w + part * ((units + slots - 1) / slots - w);
        const double cost = waves * (zc + 4) * (1.0 + 0.2 * (one ? pml_one : pml));
        if (cost < best * 0.999) {
            best = cost;
            *zc_out = zc;
        }
    }
    return best;
}

// Tile shape and z-chunks of a step kernel for storage T with occ resident CTAs
// per SM.  Which shape is faster is a matter of how the extents divide: 64 x 16
// spends 22% of its points outside a 200-wide grid, 32 x 32 covers less of a PML
// 16 to 32 points wide with its dearer edge tiles, and either may fit one wave
// where the other needs two.  Where both divide evenly, 32 x 32 costs fp32 4%
// (row ends: 256^3 60.4 -> 62.0 us) and 16-bit storage nothing.  On 23 grids from
// 96^3 to 512^3 the estimate's choice is within 3% of the faster shape at its
// best chunk length, 0.7% on average (PML 10-32, us, 64 x 16 -> 32 x 32: fp32
// 160^3 18.8 -> 16.8, 200^3 39.8 -> 34.7; bf16 200^3 42.9 -> 37.2, 224^3 49.7 ->
// 41.8, 282^3 91.9 -> 81.6, 352^3 145 -> 131, 512^3 376 -> 365).  The fp32
// difference form moves a fifth more bytes, and a single wave of 32 x 32 tiles loses
// more to its row ends there once the chunks are long (64 x 16 -> 32 x 32: 157 x
// 215 x 193 39.3 -> 41.8 us, 144 x 256 x 176 33.0 -> 35.5, 150 x 169 x 309 45.5 ->
// 48.6 with 25 to 31 planes; 224 x 208 x 160 42.1 -> 41.2, the estimate 16% apart;
// 146 x 126 x 135 17.6 -> 14.5 and 129 x 87 x 171 14.9 -> 12.8 with 9): 15% there.
template <class T, bool DIFF = false>
StepGrid choose_decomposition(int sms, int occ, StepArgs &a)
{
    const int slots = sms * occ;
    int zc = 0, zc_sq = 0;
    const double wide = plan_chunks<Cfg, T>(a, slots, &zc);
    double square = plan_chunks<CfgSq, T>(a, slots, &zc_sq);
    const long long units_sq = (long long)((a.Nx + CfgSq::BX - 1) / CfgSq::BX) *
                               ((a.Ny + CfgSq::BY - 1) / CfgSq::BY) * ((a.Nz + zc_sq - 1) / zc_sq);
    const bool long_wave = DIFF && zc_sq > 16 && units_sq <= slots;
    square *= sizeof(T) == 2 ? 1.0 : long_wave ? 1.15 : 1.04;
    StepGrid sg;
    sg.square = square < wide;
    a.zc = sg.square ? zc_sq : zc;
    with_tile(sg, [&](auto c) {
        using C = decltype(c);
        a.tiles_x = (a.Nx + C::BX - 1) / C::BX;
        a.tiles_y = (a.Ny + C::BY - 1) / C::BY;
    });
    sg.ctas = a.tiles_x * a.tiles_y * ((a.Nz + a.zc - 1) / a.zc);
    return sg;
}

}  // namespace sgb
