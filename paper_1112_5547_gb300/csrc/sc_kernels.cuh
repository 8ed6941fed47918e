// Fused two-component Shan-Chen step on sm_103a: register-pipelined kernel,
// moments / diagnostics kernel, initialisation and the diagnostics fold.
//
// One kernel performs a whole time step of Eq. eq:be with the force of
// Eq. FORCE (paper Sec. 2.1): pull-streaming of both species' populations,
// densities and momenta, the neighbour-density force, the common velocity u',
// the velocity-shifted equilibrium and BGK relaxation, and the store.  The
// per-node arithmetic is in sc_node.cuh.
//
// Storage: structure of arrays, plane (s*Q + i) holds f_is for all N nodes,
// node index x + nx*(y + ny*z).  The buffer holds post-collision values at the
// node where they were produced; pulling f_i(x, t) = f*_i(x - c_i, t - 1) is the
// streaming step, so stores are always aligned and coalesced.
//
// Tiling: a CTA owns a TX x TY tile of (x, y) columns and marches along z over
// a chunk of planes.  The force at plane z needs the densities of planes z-1,
// z, z+1 on the tile plus a one-node ring; they live in a ring of shared
// memory.  Each iteration pulls the populations of plane z+1 (kept in
// registers for the next iteration), writes their densities to the ring,
// computes the densities of the ring's halo nodes (extra pulls served mostly
// by L2, since neighbouring tiles read the same lines at about the same time),
// then collides plane z.  The halo costs 2(TX+TY)+4 extra density pulls per
// TX*TY nodes of a plane, in x and y only: marching removes the z halo.
#pragma once

#include <type_traits>

#include "sc_node.cuh"

namespace lbmsc {

// Pulled populations of node (x, y, z): f_is = f*_is(x - c_i).
// NC: through the non-coherent path (kernels that are not chained only).
template <class L, class S, bool NC = false>
__device__ __forceinline__ void pull_node(const LatticeArgs<S>& a, int x, int y, int z,
                                          typename Codec<S>::C (&f)[2][L::Q]) {
    using C = typename Codec<S>::C;
    const int nz = a.nz;
    int zs[3] = {z, z, z};  // source plane for c_z = -1, 0, +1
    if (L::D == 3) {
        zs[0] = wrap_inc(z, nz);
        zs[2] = wrap_dec(z, nz);
    }
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        // x - c_x and y - c_y lie in [-1, n]: the ghost images make them valid
        const size_t node = cell(a, x - L::c(i, 0), y - L::c(i, 1), zs[L::c(i, 2) + 1]);
        if constexpr (Codec<S>::kRest) {
            const uint32_t v = (a.fin + (size_t)i * (size_t)a.Np + node)->v;
            rest_decode<S>(v, (C)L::w(i), rest_rho<L>(a.fin, a.Np)[node], f[0][i], f[1][i]);
        } else {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const C off = Codec<S>::kOffset ? (C)__fmul_rn((float)L::w(i), (float)(s == 0 ? a.ref_A : a.ref_B)) : (C)0;
                const S* const src = a.fin + (size_t)(s * L::Q + i) * (size_t)a.Np + node;
                if constexpr (NC)
                    f[s][i] = Codec<S>::decode(__ldg(src), off);
                else
                    f[s][i] = Codec<S>::load(src, off);
            }
        }
    }
}

// Store the values of one cell.  base: the offset bases of the rest-offset
// storage (the node's densities rho_A, rho_B; any value works as long as the
// stored one is used, and a node's own density keeps the offsets small);
// ignored by the other storage types.
template <class L, class S>
__device__ __forceinline__ void store_cell(const LatticeArgs<S>& a, size_t c,
                                           const typename Codec<S>::C (&f)[2][L::Q], float2 base) {
    using C = typename Codec<S>::C;
    if constexpr (Codec<S>::kRest) {
        // the bases, kept in FP32 for the nodes that pull from this cell
        const float2 r = base;
        __stcs(rest_rho<L>(a.fout, a.Np) + c, r);
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            __stcs(&(a.fout + (size_t)i * (size_t)a.Np + c)->v, rest_encode<S>(f[0][i], f[1][i], (C)L::w(i), r));
    } else {
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const C off = Codec<S>::kOffset ? (C)__fmul_rn((float)L::w(i), (float)(s == 0 ? a.ref_A : a.ref_B)) : (C)0;
                Codec<S>::store(a.fout + (size_t)(s * L::Q + i) * (size_t)a.Np + c, f[s][i], off);
            }
        }
    }
}

// Post-collision populations of node (x, y, z), x in [0, nx), y in [0, ny), and
// of its periodic images in the ghost columns x in {-2, -1, nx, nx + 1} and
// rows y in {-2, -1, ny, ny + 1}.  Two ghost layers let a node of the halo
// ring itself (x = -1 .. nx) pull without wrapping.
// rA, rB: the node's densities (pre-collision, equal to the post-collision
// sums in exact arithmetic), the offset bases of rest-offset storage.
template <class L, class S>
__device__ __forceinline__ void store_node(const LatticeArgs<S>& a, int x, int y, int z,
                                           const typename Codec<S>::C (&f)[2][L::Q], typename Codec<S>::C rA,
                                           typename Codec<S>::C rB) {
    float2 base = make_float2(0.f, 0.f);
    if constexpr (Codec<S>::kRest) base = make_float2(rA, rB);
    store_cell<L, S>(a, cell(a, x, y, z), f, base);
    const int nx = a.nx, ny = a.ny;
    // x images: the two ghost columns the pulls read, widened to a whole 32-byte
    // sector on each side (columns -GX .. -1 and nx .. nx + GX - 1) when the
    // lattice is at least that wide, so the ghost sectors are written whole: a
    // partly written sector costs a read of the sector from HBM besides its
    // write (measured: 20 % more write traffic on 128-wide rows without it)
    constexpr int kSector = 32 / (int)sizeof(S) > 2 ? 32 / (int)sizeof(S) : 2;
    const int GX = nx >= kSector ? kSector : 2;
    if (nx >= 2 * kSector && ny >= 4) {
        // a node has at most one image along x, one along y and the corner of
        // both: their offsets are formed directly (a walk over all 24 image
        // offsets of a tiny lattice, below, costs the warps at the edges of a
        // tile about as many instructions again as their collision)
        const int ox = x < GX ? nx : (x >= nx - GX ? -nx : 0);
        const int oy = y < 2 ? ny : (y >= ny - 2 ? -ny : 0);
        if ((ox | oy) != 0) {
#pragma unroll 1
            for (int k = 1; k < 4; ++k) {
                if (((k & 1) && ox == 0) || ((k & 2) && oy == 0)) continue;
                store_cell<L, S>(a, cell(a, x + ((k & 1) ? ox : 0), y + ((k & 2) ? oy : 0), z), f, base);
            }
        }
        return;
    }
    if (x < GX || x >= nx - GX || y < 2 || y >= ny - 2) {
#pragma unroll 1
        for (int ix = -2; ix <= 2; ++ix) {
            const int xi = x + ix * nx;
            if (xi < -GX || xi > nx + GX - 1) continue;
#pragma unroll 1
            for (int iy = -2; iy <= 2; ++iy) {
                const int yi = y + iy * ny;
                if ((ix | iy) == 0 || yi < -2 || yi > ny + 1) continue;
                store_cell<L, S>(a, cell(a, xi, yi, z), f, base);
            }
        }
    }
}

// Halo ring cell of thread tid (frame coordinates; frame (1, 1) = tile (0, 0)):
// the top row, the bottom row, the left column, the right column.
template <int TX, int TY> __device__ __forceinline__ void halo_cell(int tid, int& hfx, int& hfy) {
    constexpr int FX = TX + 2, FY = TY + 2;
    if (tid < FX) {
        hfx = tid;
        hfy = 0;
    } else if (tid < 2 * FX) {
        hfx = tid - FX;
        hfy = FY - 1;
    } else if (tid < 2 * FX + TY) {
        hfx = 0;
        hfy = tid - 2 * FX + 1;
    } else {
        hfx = FX - 1;
        hfy = tid - 2 * FX - TY + 1;
    }
}

__device__ __forceinline__ double diag_fold(int k, double a, double b) {
    return (k == kMaxSpeed) ? fmax(a, b) : (k == kMinRhoA || k == kMinRhoB) ? fmin(a, b) : a + b;
}

template <class L, class S, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB) sc_fused_kernel(const LatticeArgs<S> a) {
    using C = typename Codec<S>::C;
    constexpr int Q = L::Q;
    constexpr int FX = TX + 2, FY = TY + 2;
    constexpr int NPL = L::D == 3 ? 3 : 1;
    constexpr int H = 2 * FX + 2 * TY;
    static_assert(H <= TX * TY, "halo ring must fit in the CTA");
    __shared__ Two<C> srho[NPL][FY][FX];  // densities (rho_A, rho_B)
    chain_wait();
    chain_next();

    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const bool owner = (x0 + tx) < nx && (y0 + ty) < ny;
    const int gx = (x0 + tx) % nx, gy = (y0 + ty) % ny;
    const bool halo = tid < H;
    int hfx, hfy;
    halo_cell<TX, TY>(tid, hfx, hfy);
    const int hgx = (x0 - 1 + hfx + nx) % nx;
    const int hgy = (y0 - 1 + hfy + ny) % ny;

    auto density_plane = [&](int slot, int z, C (&f)[2][Q]) {
        pull_node<L, S>(a, gx, gy, z, f);
        srho[slot][ty + 1][tx + 1] = node_densities<L, C>(f);
        if (halo) {
            C h[2][Q];
            pull_node<L, S>(a, hgx, hgy, z, h);
            srho[slot][hfy][hfx] = node_densities<L, C>(h);
        }
    };
    auto collide = [&](C (&f)[2][Q], int sm, int sc, int sp, int z) {
        const Two<C> r = srho[sc][ty + 1][tx + 1];
        auto nbr = [&](int i) -> Two<C> {
            const int slot = L::c(i, 2) == 0 ? sc : (L::c(i, 2) > 0 ? sp : sm);
            return srho[slot][ty + 1 + L::c(i, 1)][tx + 1 + L::c(i, 0)];
        };
        node_update<L, C>(a, gy, nbr, f, r.a, r.b);
        if (owner) store_node<L, S>(a, gx, gy, z, f, r.a, r.b);
    };

    C cur[2][Q];
    if (L::D == 2) {
        density_plane(0, 0, cur);
        __syncthreads();
        collide(cur, 0, 0, 0, 0);
    } else {
        const int z0 = blockIdx.z * a.zchunk;
        const int z1 = min(z0 + a.zchunk, nz);
        {
            C tmp[2][Q];
            density_plane(0, z0 == 0 ? nz - 1 : z0 - 1, tmp);
        }
        density_plane(1, z0, cur);
        int sm = 0, sc = 1, sp = 2;
        for (int z = z0; z < z1; ++z) {
            C nxt[2][Q];
            density_plane(sp, z + 1 == nz ? 0 : z + 1, nxt);
            __syncthreads();
            collide(cur, sm, sc, sp, z);
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int i = 0; i < Q; ++i) cur[s][i] = nxt[s][i];
            const int t = sm;
            sm = sc;
            sc = sp;
            sp = t;
            __syncthreads();
        }
    }
}

// Reported fields and FP64 diagnostics of the current populations.  Marches
// like sc_fused_kernel, but a thread keeps only the momentum of the plane it
// has pulled (3 values instead of 2 Q), so three CTAs share an SM; CTAs take
// tiles and chunks in turn (item = blockIdx.x, + gridDim.x, ...), so that a large
// lattice leaves a few thousand partial sums to fold, not one per tile.
//
// The FP64 sums run on two FP64 lanes a clock and SM and bound the diagnostics:
// per node they take the conversions, one product and sum each for the masses,
// momenta and the energy and one maximum.  The square root of the peak speed is
// taken of the maximum (both are monotone, the rounded result is the same), the
// minima stay in the compute type, a window's distances are formed per column
// and plane, and no window costs nothing.  Measured (GB300): fields 512^3 FP32
// 10.1 -> 5.8 ms, 256^3 1.30 -> 0.75; diagnostics 512^3 FP32 20.9 -> 9.3 ms, 4096^2 4.74 -> 1.04.
template <class L, class S, int TX, int TY, bool DIAG, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB)
    sc_moments_kernel(const LatticeArgs<S> a, const FieldArgs<typename Codec<S>::C> fo, int tiles_x, int tiles_y,
                      int nitems) {
    using C = typename Codec<S>::C;
    using A = Ar<C>;
    constexpr int Q = L::Q;
    constexpr int FX = TX + 2, FY = TY + 2;
    constexpr int NPL = L::D == 3 ? 3 : 1;
    constexpr int H = 2 * FX + 2 * TY;
    static_assert(H <= TX * TY, "halo ring must fit in the CTA");
    __shared__ Two<C> srho[NPL][FY][FX];

    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const bool halo = tid < H;
    int hfx, hfy;
    halo_cell<TX, TY>(tid, hfx, hfy);
    const bool win_in = DIAG && fo.r_in2 > 0.0, win_out = DIAG && fo.r_out2 < 1e300;

    // FP64 sums: masses, momenta, energy; with a window its densities and pressures
    enum { kA, kB, kX, kY, kZ, kE, kIA, kIP, kOA, kOP, kSums };
    double acc[kSums];
    double uu_max = 0.0;
    C minA = (C)INFINITY, minB = (C)INFINITY;
    int nonfinite = 0, drop = 0, n_in = 0, n_out = 0;
    if (DIAG) {
#pragma unroll
        for (int k = 0; k < kSums; ++k) acc[k] = 0.0;
    }

#pragma unroll 1
    for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
        const int bx = item % tiles_x, by = (item / tiles_x) % tiles_y, bz = item / (tiles_x * tiles_y);
        const int x0 = bx * TX, y0 = by * TY;
        const bool owner = (x0 + tx) < nx && (y0 + ty) < ny;
        const int gx = (x0 + tx) % nx, gy = (y0 + ty) % ny;
        const int hgx = (x0 - 1 + hfx + nx) % nx;
        const int hgy = (y0 - 1 + hfy + ny) % ny;
        double rxy2 = 0.0;  // squared periodic minimum-image distance of the column from the window's centre
        if (win_in || win_out) {
            double dx = fabs((double)gx - fo.win_c[0]), dy = fabs((double)gy - fo.win_c[1]);
            dx = fmin(dx, (double)nx - dx);
            dy = fmin(dy, (double)ny - dy);
            rxy2 = dx * dx + dy * dy;
        }

        // densities of plane z into a ring slot, and the node's momentum
        auto density_plane = [&](int slot, int z, C (&j)[3]) {
            {
                C f[2][Q];
                pull_node<L, S>(a, gx, gy, z, f);
                srho[slot][ty + 1][tx + 1] = node_densities<L, C>(f);
                Two<C> js[3];
                node_momenta<L, C>(f, js);
                // FE: u = sum_i f_i c_i / rho, from the first population alone
#pragma unroll
                for (int d = 0; d < 3; ++d) j[d] = a.model == kModelFE ? js[d].a : A::add(js[d].a, js[d].b);
            }
            if (halo) {
                C h[2][Q];
                pull_node<L, S>(a, hgx, hgy, z, h);
                srho[slot][hfy][hfx] = node_densities<L, C>(h);
            }
        };

        auto process = [&](const C (&j)[3], int sm, int sc, int sp, int z) {
            const Two<C> r01 = srho[sc][ty + 1][tx + 1];
            const C r0 = r01.a, r1 = r01.b;
            auto nbr = [&](int i) -> Two<C> {
                const int slot = L::c(i, 2) == 0 ? sc : (L::c(i, 2) > 0 ? sp : sm);
                return srho[slot][ty + 1 + L::c(i, 1)][tx + 1 + L::c(i, 0)];
            };
            const size_t node = (size_t)gx + (size_t)nx * ((size_t)gy + (size_t)ny * z);
            // SC: physical velocity u = (j_A + j_B + (F_A + F_B) / 2) / rho (F dt/2
            // shift, Sec. 2.3).  FE (Sec. 2.2): u = sum_i f_i c_i / rho, and the
            // reported densities are rho_A = (rho + phi)/2, rho_B = (rho - phi)/2.
            const bool fe = a.model == kModelFE;
            C gA[3] = {(C)0, (C)0, (C)0}, gB[3] = {(C)0, (C)0, (C)0};
            if (!fe) {
                node_force<L, C>(nbr, a.G, gA, gB);
                node_body_force<C>(a.body_A, gy, a.ny, gA, gB);
            }
            const C rA = fe ? A::mul((C)0.5, A::add(r0, r1)) : r0;
            const C rB = fe ? A::mul((C)0.5, A::sub(r0, r1)) : r1;
            const C rho = fe ? r0 : A::add(rA, rB);
            const C inv_rho = A::rcp(rho);
            C u[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const C half_force = A::mul((C)0.5, A::fma(rA, gA[d], A::mul(rB, gB[d])));
                u[d] = A::mul(A::add(j[d], half_force), inv_rho);
            }
            const C p = A::mul(A::fma(A::mul(a.G, rA), rB, rho), (C)(1.0 / 3.0));
            if (!owner) return;
            if (!DIAG) {
                if (fo.rhoA) fo.rhoA[node] = rA;
                if (fo.rhoB) fo.rhoB[node] = rB;
                if (fo.u)
#pragma unroll
                    for (int d = 0; d < L::D; ++d) fo.u[(size_t)d * (size_t)a.N + node] = u[d];
                if (fo.p) fo.p[node] = p;
            } else {
                const double dA = (double)rA, dB = (double)rB, drho = dA + dB;
                double ud[3], uu = 0.0;
#pragma unroll
                for (int d = 0; d < L::D; ++d) {
                    ud[d] = (double)u[d];
                    uu += ud[d] * ud[d];
                }
                const bool finite = isfinite(dA) && isfinite(dB) && isfinite(uu) && isfinite(p);
                if (finite) {
                    acc[kA] += dA;
                    acc[kB] += dB;
                    acc[kX] += ud[0] * drho;
                    acc[kY] += ud[1] * drho;
                    if (L::D == 3) acc[kZ] += ud[L::D - 1] * drho;
                    acc[kE] += (0.5 * drho) * uu;
                    uu_max = fmax(uu_max, uu);
                    minA = rA < minA ? rA : minA;
                    minB = rB < minB ? rB : minB;
                } else {
                    ++nonfinite;
                }
                if (win_in || win_out) {
                    double dz = 0.0;
                    if (L::D == 3) {
                        dz = fabs((double)z - fo.win_c[2]);
                        dz = fmin(dz, (double)nz - dz);
                    }
                    const double r2 = rxy2 + dz * dz;
                    if (r2 < fo.r_in2) {
                        ++n_in;
                        acc[kIA] += dA;
                        acc[kIP] += (double)p;
                    }
                    if (r2 > fo.r_out2) {
                        ++n_out;
                        acc[kOA] += dA;
                        acc[kOP] += (double)p;
                    }
                }
                // inside the drop: phi = rho_A - rho_B >= 0, compared in the compute type (Sec. 4.2)
                if (rA >= rB) ++drop;
            }
        };

        C cur[3];
        if (L::D == 2) {
            density_plane(0, 0, cur);
            __syncthreads();
            process(cur, 0, 0, 0, 0);
            __syncthreads();
        } else {
            const int z0 = a.zbase + bz * a.zchunk;
            const int z1 = min(z0 + a.zchunk, a.zend);
            density_plane(0, z0 == 0 ? nz - 1 : z0 - 1, cur);
            density_plane(1, z0, cur);
            int sm = 0, sc = 1, sp = 2;
#pragma unroll 1
            for (int z = z0; z < z1; ++z) {
                C nxt[3];
                density_plane(sp, z + 1 == nz ? 0 : z + 1, nxt);
                __syncthreads();
                process(cur, sm, sc, sp, z);
#pragma unroll
                for (int d = 0; d < 3; ++d) cur[d] = nxt[d];
                const int t = sm;
                sm = sc;
                sc = sp;
                sp = t;
                __syncthreads();
            }
        }
    }

    if (DIAG) {
        // CTA reduction: one warp per FP64 sum over the threads' values in shared
        // memory (13 additions a lane; shuffling every sum through every warp took
        // eight times as many on the few FP64 lanes, 6 us a CTA), whole numbers by
        // the warp reductions, maximum and minima by shuffles
        constexpr int NW = TX * TY / 32, NT = TX * TY;
        static_assert(NW >= 6, "a warp per sum");
        __shared__ double sums[6][NT];
        __shared__ int counts[NW][4];
        __shared__ double ext[NW][3];
        const int lane = tid & 31, warp = tid >> 5;
        double* const out = fo.partials + (size_t)blockIdx.x * kNumDiag;
        const int cnt[4] = {nonfinite, drop, n_in, n_out};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int v = __reduce_add_sync(0xffffffffu, cnt[k]);
            if (lane == 0) counts[warp][k] = v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double m = __shfl_xor_sync(0xffffffffu, uu_max, o);
            uu_max = m > uu_max ? m : uu_max;
            const C p = __shfl_xor_sync(0xffffffffu, minA, o), q = __shfl_xor_sync(0xffffffffu, minB, o);
            minA = p < minA ? p : minA;
            minB = q < minB ? q : minB;
        }
        if (lane == 0) {
            ext[warp][0] = uu_max;
            ext[warp][1] = (double)minA;
            ext[warp][2] = (double)minB;
        }
        // sums k0 .. k0 + n - 1 into the record's slots
        auto fold_sums = [&](auto k0, int n) {
            __syncthreads();
#pragma unroll
            for (int k = 0; k < 6; ++k)
                if (k0 + k < kSums) sums[k][tid] = acc[k0 + k];
            __syncthreads();
            if (warp < n) {
                double v = sums[warp][lane];
#pragma unroll
                for (int t = 1; t < NW; ++t) v += sums[warp][lane + 32 * t];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                constexpr int slot[12] = {kMassA, kMassB, kMomX, kMomY, kMomZ, kKE, kInRhoA, kInP, kOutRhoA, kOutP, 0, 0};
                if (lane == 0) out[slot[k0 + warp]] = v;
            }
        };
        fold_sums(std::integral_constant<int, 0>(), 6);
        if (win_in || win_out)
            fold_sums(std::integral_constant<int, 6>(), 4);
        else if (tid == 0)
            out[kInRhoA] = out[kInP] = out[kOutRhoA] = out[kOutP] = 0.0;
        if (tid == 0) {
            int c[4] = {0, 0, 0, 0};
            double m[3] = {0.0, INFINITY, INFINITY};
            for (int w = 0; w < NW; ++w) {
                for (int k = 0; k < 4; ++k) c[k] += counts[w][k];
                m[0] = ext[w][0] > m[0] ? ext[w][0] : m[0];
                m[1] = ext[w][1] < m[1] ? ext[w][1] : m[1];
                m[2] = ext[w][2] < m[2] ? ext[w][2] : m[2];
            }
            out[kMaxSpeed] = sqrt(m[0]);
            out[kMinRhoA] = m[1] < 1e300 ? m[1] : 1e300;  // 1e300: no finite node
            out[kMinRhoB] = m[2] < 1e300 ? m[2] : 1e300;
            out[kNonFinite] = c[0];
            out[kDropNodes] = c[1];
            out[kInCount] = c[2];
            out[kOutCount] = c[3];
        }
    }
}

// Low-register variant of the step: the populations of plane z are not kept
// in registers while plane z+1 is reduced to densities; they are pulled a
// second time for the collision, one iteration after their first load, when
// they are normally still in L1.  Holding only one plane of pulls lets more
// CTAs share an SM (more loads in flight), and the four-slot density ring
// needs one __syncthreads per plane.  Arithmetic and order as sc_fused_kernel.
// Reference-offset 16-bit storage on tile 14 (D3Q19, 128 registers a thread): the pulls go
// through the non-coherent path, which lets the compiler move them across the
// plane's barrier (48^3, 16 planes a chunk: 70 us a step with plain loads, 55 so); such
// a kernel is not chained (sc_common.cuh).  In the other storages and tiles plain loads
// are as fast or faster (rest-offset by up to 14 %).
template <class L, class S, int TX, int TY, int MINB> constexpr bool reload_nc() {
    return L::D == 3 && Codec<S>::kOffset && TX * TY * MINB <= 512;
}
template <class L, class S, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB) sc_step_reload_kernel(const LatticeArgs<S> a) {
    using C = typename Codec<S>::C;
    constexpr int Q = L::Q;
    constexpr int FX = TX + 2, FY = TY + 2;
    constexpr int NPL = L::D == 3 ? 4 : 1;
    constexpr int H = 2 * FX + 2 * TY;
    static_assert(H <= TX * TY, "halo ring must fit in the CTA");
    constexpr bool NC = reload_nc<L, S, TX, TY, MINB>();
    __shared__ Two<C> ring[NPL][FY][FX];
    if (!NC) {
        chain_wait();
        chain_next();
    }

    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const bool owner = (x0 + tx) < nx && (y0 + ty) < ny;
    const int gx = (x0 + tx) % nx, gy = (y0 + ty) % ny;
    const bool halo = tid < H;
    int hfx, hfy;
    halo_cell<TX, TY>(tid, hfx, hfy);
    const int hgx = (x0 - 1 + hfx + nx) % nx;
    const int hgy = (y0 - 1 + hfy + ny) % ny;

    auto density_plane = [&](int slot, int z) {
        C f[2][Q];
        pull_node<L, S, NC>(a, gx, gy, z, f);
        ring[slot][ty + 1][tx + 1] = node_densities<L, C>(f);
        if (halo) {
            pull_node<L, S, NC>(a, hgx, hgy, z, f);
            ring[slot][hfy][hfx] = node_densities<L, C>(f);
        }
    };
    // (kept == nullptr: pull here)
    auto collide = [&](C (*kept)[2][Q], int sm, int sc, int sp, int z) {
        C f[2][Q];
        if (kept) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                f[0][i] = (*kept)[0][i];
                f[1][i] = (*kept)[1][i];
            }
        } else {
            pull_node<L, S, NC>(a, gx, gy, z, f);
        }
        const Two<C> r = ring[sc][ty + 1][tx + 1];
        const C rA = r.a, rB = r.b;
        auto nbr = [&](int i) -> Two<C> {
            const int sl = L::c(i, 2) == 0 ? sc : (L::c(i, 2) > 0 ? sp : sm);
            return ring[sl][ty + 1 + L::c(i, 1)][tx + 1 + L::c(i, 0)];
        };
        node_update<L, C>(a, gy, nbr, f, rA, rB);
        if (owner) store_node<L, S>(a, gx, gy, z, f, rA, rB);
    };

    if (L::D == 2) {
        // one plane: its pulls stay in registers (pulled again, 2000 x 2100 bf16
        // rest-offset on tile 11 takes 160 us a step instead of 106)
        C f[2][Q];
        pull_node<L, S>(a, gx, gy, 0, f);
        ring[0][ty + 1][tx + 1] = node_densities<L, C>(f);
        if (halo) {
            C h[2][Q];
            pull_node<L, S>(a, hgx, hgy, 0, h);
            ring[0][hfy][hfx] = node_densities<L, C>(h);
        }
        __syncthreads();
        collide(&f, 0, 0, 0, 0);
        return;
    }
    const int z0 = blockIdx.z * a.zchunk;
    const int z1 = min(z0 + a.zchunk, nz);
    // ring slot of plane z is (z - z0 + 1) & 3
    density_plane(0, z0 == 0 ? nz - 1 : z0 - 1);
    density_plane(1, z0);
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        const int k = z - z0 + 1;
        density_plane((k + 1) & 3, z + 1 == nz ? 0 : z + 1);
        __syncthreads();
        collide(nullptr, (k - 1) & 3, k & 3, (k + 1) & 3, z);
    }
}

// Second pass of the diagnostics: CTA k folds slot k of the partial records
// (one CTA for all slots spent its time on one SM's FP64 lanes: 22 us with
// 1024 threads, whatever the lattice).
template <int NT>
__global__ void __launch_bounds__(NT) sc_diag_finish_kernel(const double* __restrict__ partials,
                                                            long long nparts, double* __restrict__ out) {
    __shared__ double red[NT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = blockIdx.x;
    double v = (k == kMinRhoA || k == kMinRhoB) ? 1e300 : 0.0;
    for (long long b = tid; b < nparts; b += NT) v = diag_fold(k, v, partials[b * kNumDiag + k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = diag_fold(k, v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < NT / 32; ++w) v = diag_fold(k, v, red[w]);
        out[k] = v;
    }
}

// Populations of the rest / moving equilibrium (planes [zlo, zhi)): the buffer slot of direction i
// at node x holds f^eq_i(rho_s(x + c_i), u(x + c_i)), so pulling it at x + c_i
// gives f_i(x + c_i, 0) = f^eq_i of that node.  The ghost columns and rows get
// the values of their periodic images.
// One thread per cell, row after row.  Wide rows hold whole 32-byte sectors (the x images
// fill one on either side, as in store_node), and their lanes begin on one, so that no warp's
// stores leave a partly written sector, each of which reads HBM; 16-bit rows begin on a
// cache line.  Narrow rows, where the images would be a good part of the work, take the
// two images that a step reads.  Whether the fluid moves is a template argument: a branch
// around the velocity's loads in each of the Q directions serialises them.  Measured
// (GB300, us at rest / moving; rows walked by blocks of 64 lanes, with that branch, and
// now): FP32 512^3 5214 / 9294 -> 3407 / 6175, 128^3 77 / 124 -> 59 / 119; FP64 160^3
// 1261 / 3120 -> 627 / 2337, 171 x 217 x 4 529 / 1289 -> 102 / 172; bf16 rest-offset 256^3
// 535 / 901 -> 453 / 697.
struct InitRow {
    int images;   // cells x in [-images, nx + images) are written
    int lead;     // lane 0 is the cell x = -lead
    int lanes;    // of a row
    int threads;  // of a block
};
template <class S> __host__ __device__ __forceinline__ InitRow init_row(int nx) {
    constexpr int kSector = 32 / (int)sizeof(S) > 2 ? 32 / (int)sizeof(S) : 2;
    // rows of less than 12 sectors (FP32 185 x 158 x 78: 153 us with whole sectors, 145 without)
    if (nx < 12 * kSector) return InitRow{2, 2, nx + 4, Codec<S>::kRest ? 64 : 256};
    if (sizeof(S) == 2) return InitRow{kSector, 32, (nx + 32 + kSector + 31) / 32 * 32, 256};
    return InitRow{kSector, kSector, (nx + 2 * kSector + kSector - 1) / kSector * kSector, 64};
}
template <class L, class S, bool MOVING>
__global__ void __launch_bounds__(256)
    sc_init_kernel(const LatticeArgs<S> a, const typename Codec<S>::C* __restrict__ rhoA,
                   const typename Codec<S>::C* __restrict__ rhoB, const typename Codec<S>::C* __restrict__ u, int zlo,
                   int zhi) {
    using C = typename Codec<S>::C;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const InitRow rw = init_row<S>(nx);
    const int ey = ny + 4;  // cells y in [-2, ny + 2)
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    auto quotient = [](long long v, int d) { return v <= 0xffffffffLL ? (long long)((unsigned)v / (unsigned)d) : v / d; };
    const long long row = quotient(k, rw.lanes), plane = quotient(row, ey);
    const int cx = (int)(k - row * rw.lanes) - rw.lead;
    const int cy = (int)(row - plane * ey) - 2;
    // the cells of planes [zlo, zhi); they read the fields of planes zlo - 1 .. zhi (periodic)
    if (cx < -rw.images || cx >= nx + rw.images || plane >= zhi - zlo) return;
    const int z = zlo + (int)plane;
    const size_t n = cell(a, cx, cy, z);
    const int x = ((cx % nx) + nx) % nx, y = ((cy % ny) + ny) % ny;
    const int xs[3] = {wrap_dec(x, nx), x, wrap_inc(x, nx)};
    const int ys[3] = {wrap_dec(y, ny), y, wrap_inc(y, ny)};
    const int zs[3] = {L::D == 3 ? wrap_dec(z, nz) : 0, L::D == 3 ? z : 0, L::D == 3 ? wrap_inc(z, nz) : 0};
    C fr[2][L::Q];  // rest-offset storage: the cell's values, stored together
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const size_t m = (size_t)xs[L::c(i, 0) + 1] +
                         (size_t)nx * ((size_t)ys[L::c(i, 1) + 1] + (size_t)ny * zs[L::c(i, 2) + 1]);
        C shape = (C)1;
        if (MOVING) {
            C uv[3] = {0, 0, 0};
            for (int d = 0; d < L::D; ++d) uv[d] = u[(size_t)d * (size_t)a.N + m];
            C uu = uv[0] * uv[0] + uv[1] * uv[1] + uv[2] * uv[2];
            C cu = (C)0;
            for (int d = 0; d < L::D; ++d) cu += (C)L::c(i, d) * uv[d];
            shape = (C)1 - (C)1.5 * uu + cu * ((C)3 + (C)4.5 * cu);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            // SC: species densities; FE: f from rho = rho_A + rho_B, g from phi = rho_A - rho_B
            const C rho = a.model == kModelFE ? (s == 0 ? rhoA[m] + rhoB[m] : rhoA[m] - rhoB[m])
                                              : (s == 0 ? rhoA[m] : rhoB[m]);
            const C f = (C)L::w(i) * rho * shape;
            if constexpr (Codec<S>::kRest) {
                fr[s][i] = f;
            } else {
                const C off = Codec<S>::kOffset ? (C)__fmul_rn((float)L::w(i), (float)(s == 0 ? a.ref_A : a.ref_B)) : (C)0;
                Codec<S>::store(a.fout + (size_t)(s * L::Q + i) * (size_t)a.Np + n, f, off);
            }
        }
    }
    if constexpr (Codec<S>::kRest) {
        // rest-offset bases: the sums of the cell's stored values, in a fixed order
        float2 r = make_float2(fr[0][0], fr[1][0]);
#pragma unroll
        for (int i = 1; i < L::Q; ++i) {
            r.x = __fadd_rn(r.x, fr[0][i]);
            r.y = __fadd_rn(r.y, fr[1][i]);
        }
        store_cell<L, S>(a, n, fr, r);
    }
}

}  // namespace lbmsc
