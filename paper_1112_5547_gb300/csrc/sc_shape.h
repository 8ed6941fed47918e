// Launch shape (tile and z chunk) of the step kernel for a lattice that was
// not tuned: a small model of a step's time, minimised over the candidates.
//
// A CTA marches over its chunk of zc planes and reduces two more to densities,
// so it costs a = zc + extra plane times, `extra` being two planes without
// collision and stores.  The grid starts its CTAs chunk by chunk (the short last chunk
// comes last) on `per_sm` CTAs per SM, and the step ends with the last of them:
// list scheduling of equal items followed by shorter ones.  With the plane time
// of the tile (weight; 1 = a 64x6 FP32 tile, 3.5 - 3.9 us) and the gap between
// two launches this reproduces measured times within about 10 % (GB300, 128^3
// FP32 on 64x6 tiles, us: chunks of 10 planes 173 (45 plane times in the model),
// 13: 168 (43), 16: 194 (52), 20: 173 (42), 28: 220 (58), 43: 193 (44 and the
// one-wave penalty)).  At least 16 planes a chunk on one tile for every lattice,
// the rule before, gave 313 us there, 18.5 ms instead of 7.1 at 512^3, 84 us
// instead of 7.4 at 32^3 and 562 instead of 111 at 48^3 in FP64.
#pragma once

#include "sc_launch.cuh"

namespace lbmsc {

struct StepModel {
    int per_sm;     // CTAs per SM
    double extra;   // cost of a chunk's two density-only planes, in planes
    double weight;  // time of one plane with the SMs full
    double launch;  // from the end of one step to the start of the next
};

// The tiles an untuned lattice may get (-1 ends the list), best first among equals.
//  34 / 41 / 37: 64x6, 48x8 and 32x12 TMA tiles; the one with the least padding
//      of a ragged lattice wins.  18: 32x8, for lattices too low for the others.
//  43 / 42 / 44: the 16-bit TMA tiles with two CTAs per SM (clusters of 1x2, and without),
//      38: the 32x12 one with one.
//  15 / 17 (FP32) and 3: register kernels, for lattices narrower than a TMA tile
//      and for small ones.
inline const int* step_candidates(const Plan& p) {
    static constexpr int f32[] = {34, 41, 37, 18, 15, 17, -1}, f32_any[] = {34, 3, -1}, f16[] = {43, 42, 44, 38, 3, -1},
                         f64[] = {3, -1};
    if (p.precision == 0) return f64;
    if (p.precision != 1) return f16;
    return p.forcing == kForcingShift && p.model == kModelSC ? f32 : f32_any;
}

// Both buffers fit L2 (129 MB).
inline bool in_l2(const Plan& p) {
    return 2.0 * population_planes(p.lattice, p.precision) * (double)p.Np * storage_elem_bytes(p.precision) < 1e8;
}

inline StepModel step_model(const Plan& p, int tile) {
    // FP64 is bound by the FP64 units (two FMA a clock and SM): CTAs on one SM
    // share them, density-only planes are nearly free, and one CTA alone leaves
    // a fifth of the rate unused (48^3 on 32x4 columns in chunks of 2 / 4 / 6 / 8
    // planes: 154 / 144 / 211 / 159 us)
    if (p.precision == 0) return {1, 0.4, 4.5, 0.8};
    const bool l2 = in_l2(p);
    switch (tile) {
        case 34:
        case 41: return {1, 1.2, 1.0, 0.8};
        case 37: return {1, 1.2, 1.03, 0.8};
        case 18: return {1, 1.2, 0.83, 0.8};
        case 42:
        case 43: return {2, 1.2, 0.9, 0.8};
        case 44: return {2, 1.2, 0.93, 0.8};
        case 38: return {1, 1.2, 0.78, 0.8};
        case 15:
        case 17: return {3, 2.0, l2 ? 0.85 : 1.5, 0.8};
        default: break;
    }
    // tiles that only a caller picks, where the model chooses the chunk alone: as their kin
    const TileShape& t = kTiles[tile];
    if (t.kind == 5 || t.kind == 6) return {t.minb, 1.2, t.tx * t.ty / 384.0, 0.8};
    if (t.kind == 4) return {t.stages, 2.0, l2 ? 0.85 : 1.5, 0.8};
    return p.precision == 1 ? StepModel{4, 2.0, l2 ? 0.96 : 1.75, 0.8} : StepModel{4, 2.0, l2 ? 1.3 : 1.8, 0.8};
}

// Time of a step in plane times of the 64x6 tile.
inline double step_cost(const Plan& p, int tile, int zc) {
    TileShape t = kTiles[tile];
    if (p.precision == 0 && tile == 3) f64_tile3(p, t.tx, t.ty);
    const StepModel m = step_model(p, tile);
    const long long xy = (long long)((p.nx + t.tx - 1) / t.tx) * ((p.ny + t.ty - 1) / t.ty);
    const long long slots = (long long)m.per_sm * p.sm_count, full = xy * (p.nz / zc);
    const int last = p.nz % zc;
    const double a = zc + m.extra, b = last + m.extra;
    const long long waves = full / slots, rem = full % slots;
    double end = (double)(waves + (rem ? 1 : 0)) * a;
    if (last) {
        // the xy short items start on the slots that come free first
        const long long early = slots - rem;
        long long left = xy;
        double t0 = (double)waves * a;
        const double t1 = (double)(waves + 1) * a;
        while (left > 0) {
            if (rem == 0 || t0 + b <= t1) {  // another round on the early slots
                t0 += b;
                left -= early;
            } else {  // all slots free at about t1
                t0 = t1 + b * (double)((left + slots - 1) / slots);
                left = 0;
            }
        }
        if (t0 > end) end = t0;
    }
    const double n = (double)(full + (last ? xy : 0)) / (double)slots;  // waves
    double f = m.weight;
    if (p.precision == 0) {
        // CTAs are resident early and share their SM's units: the time is the work
        // of the SM that gets the first CTA of every round (96^3: 24 planes a chunk
        // 803 us, 20 with a short last chunk 1080); one CTA alone on an SM loses a
        // fifth of the rate
        const long long rounds = (full + (last ? xy : 0) + slots - 1) / slots, rfull = (full + slots - 1) / slots;
        end = (double)rfull * a + (double)(rounds - rfull) * b;
        if (n <= 1.0) f *= 1.2;
    } else if (m.per_sm > 1) {
        // fewer CTAs than slots: each runs faster (96^3 Guo, 32x4 tiles, us a
        // plane of all resident CTAs: two per SM 4.15, four 5.9)
        if (n < 1.0) f *= 0.45 + 0.55 * n;
    } else {
        // one wave over HBM starts and ends in step (128^3: 10 - 15 % a plane
        // slower), long chunks lose shared halo rows (192^3: 31 planes 473 us, 14 446)
        if (!in_l2(p)) f *= (1.0 + (n > 1.0 ? 0.3 / n : 0.15)) * (1.0 + 0.003 * zc);
    }
    return end * f + m.launch;
}

constexpr int kMaxGridYZ = 65535;

// Whether the tile rows of a lattice fit the second dimension of a grid.
inline bool rows_fit(int tile, const Plan& p) { return (p.ny + kTiles[tile].ty - 1) / kTiles[tile].ty <= kMaxGridYZ; }

// Whether a launch takes the grid of a tile and z chunk.
inline bool shape_fits_grid(int tile, int zc, const Plan& p) {
    return rows_fit(tile, p) && (p.nz + zc - 1) / zc <= kMaxGridYZ;
}

// Best z chunk of a tile (D3Q19).
inline int best_zchunk(const Plan& p, int tile, double* cost = nullptr) {
    // long chunks let neighbouring tiles drift apart and lose the halo rows they
    // share in L2 (256^3 FP32, chunks of 24 / 43 / 64 planes: 1.05 / 1.14 / 1.19
    // ms; bf16 rest-offset 0.765 / 0.796 / 0.839)
    const int least = (p.nz + kMaxGridYZ - 1) / kMaxGridYZ;  // chunks are a grid's third dimension
    int most = p.precision >= 2 ? 48 : 32;
    if (most < least) most = least;
    int best = least;
    double c = step_cost(p, tile, least);
    for (int z = least + 1; z <= p.nz && z <= most; ++z) {
        const double k = step_cost(p, tile, z);
        if (k < c * (p.precision == 0 ? 1.0 + 1e-9 : 1.0 - 1e-9)) {  // FP64: the longer of equals
            c = k;
            best = z;
        }
    }
    if (cost) *cost = c;
    return best;
}

// Tile and z chunk of an untuned lattice.
inline void pick_step(Plan& p) {
    if (p.lattice == 0) {
        // D2Q9: 32x4 tiles, four to six CTAs per SM (4096^2 FP32 0.461 ms a
        // step against 0.487 with 32x8, 64^2 2.7 us against 3.2); FP64 is
        // bound by its units and 32x8 has the smaller halo (256^2 30.5 / 31.2 us)
        p.step_tile = p.precision == 0 || !rows_fit(kTileD2, p) ? 0 : kTileD2;
        p.step_zchunk = 1;
        return;
    }
    double best = 0.0;
    int tile = -1, zc = 1;
    for (const int* t = step_candidates(p); *t >= 0; ++t) {
        if (!tile_fits(*t, p) || !rows_fit(*t, p)) continue;
        double c;
        const int z = best_zchunk(p, *t, &c);
        if (tile < 0 || c < best * (1.0 - 1e-9)) {
            best = c;
            tile = *t;
            zc = z;
        }
    }
    if (tile < 0) {  // more rows than any candidate's grid holds
        tile = 0;
        zc = best_zchunk(p, 0);
    }
    p.step_tile = tile;
    p.step_zchunk = zc;
}

}  // namespace lbmsc
