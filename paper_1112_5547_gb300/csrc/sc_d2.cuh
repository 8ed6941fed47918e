// Several D2Q9 time steps per launch (FP32 storage), bit-identical to single
// steps: the arithmetic of a node is sc_node.cuh's, only where the populations
// live between two steps changes.
//
// sc_d2_pair_kernel: two steps of a 32x16 tile.  A single step reads and writes
// 144 bytes a node and is bound by HBM on large lattices and by latency (one
// dependent chain of pulls, densities, collision and store per launch) on
// middling ones.  Here a CTA pulls its tile and a halo of three nodes, keeps the
// first step's populations of the tile and a halo of two in shared memory, and
// runs the second step from there: half the traffic and half the launches for
// 20 % more collisions (36 x 20 + 32 x 16 for 2 x 512) and 1.6 times the pulls,
// most of which hit L2.  What bounds it now is the chain of its four phases with
// two CTAs per SM (DRAM at 48 % of the copy peak at 4096^2).  Measured, us a step
// before and now: 4096^2 461 / 367, 1024^2 34 / 26, 256^2 3.8 / 3.1, eight 256^2
// lattices in a batch of 300 steps 19 / 13.7.  Three CTAs of 256 threads that pass
// every pulled value through shared memory (45 % of the issue slots at 2048^2) take
// 352, 26 and 3.2, but 434 x 149 3.43 against 3.09: 4 % less at 4096^2 for 11 % more
// on the middling sizes, so this form serves them all.
//
// sc_d2_resident_kernel: all the steps of a call in one launch for a lattice
// that fits the shared memory of one thread-block cluster.  Each CTA owns a band
// of rows (both buffers in shared memory), writes its outermost two rows into
// its neighbours' halo rows (distributed shared memory) and meets them at a
// cluster barrier once a step (64^2: 2.7 us a step in single launches, 1.5 here,
// of which about 1 is the barrier and the phases' latency).
#pragma once

#include <cooperative_groups.h>

#include "sc_batch.cuh"

namespace lbmsc {

struct PairSmem {
    static constexpr int PX = kPairTX + 6, PY = kPairTY + 6;  // first step's densities
    static constexpr int AX = kPairTX + 4, AY = kPairTY + 4;  // first step's collisions
    static constexpr int BX = kPairTX + 2, BY = kPairTY + 2;  // second step's densities
    Two<float> f[D2Q9::Q][AX * AY];
    Two<float> rho1[PX * PY];
    Two<float> rho2[BX * BY];
};

__device__ __forceinline__ int wrap_once(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Two steps of the tile at (x0, y0); nx > 34, ny > 18 (a coordinate of the
// tile's frame wraps at most once).  A thread keeps the populations it pulled in
// registers until their densities are complete (two nodes at a time in either
// step), so shared memory, whose bandwidth bounds the kernel next, carries only
// the first step's results and the densities.
__device__ __forceinline__ void d2_pair_tile(const LatticeArgs<float>& a, int x0, int y0, PairSmem& sm) {
    using L = D2Q9;
    using S = PairSmem;
    constexpr int NT = kPairThreads, A = S::AX * S::AY, B = kPairTX * kPairTY;
    constexpr int RING1 = S::PX * S::PY - A, RING2 = S::BX * S::BY - B;
    static_assert(A <= 2 * NT && B <= 2 * NT && RING1 <= NT && RING2 <= NT, "two nodes per thread, one of each ring");
    const int tid = threadIdx.x;
    const int nx = a.nx, ny = a.ny;
    float f[2][2][L::Q];

    // first step: pulls and densities of the frame, the outermost ring by the last threads
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int k = tid + s * NT;
        if (k < A) {
            const int fy = k / S::AX, fx = k - fy * S::AX;
            pull_node<L, float>(a, wrap_once(x0 - 2 + fx, nx), wrap_once(y0 - 2 + fy, ny), 0, f[s]);
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int k = tid + s * NT;
        if (k < A) {
            const int fy = k / S::AX, fx = k - fy * S::AX;
            sm.rho1[(fy + 1) * S::PX + fx + 1] = node_densities<L, float>(f[s]);
        }
    }
    if (tid >= NT - RING1) {
        int fx, fy;
        halo_cell<S::AX, S::AY>(tid - (NT - RING1), fx, fy);
        float h[2][L::Q];
        pull_node<L, float>(a, wrap_once(x0 - 3 + fx, nx), wrap_once(y0 - 3 + fy, ny), 0, h);
        sm.rho1[fy * S::PX + fx] = node_densities<L, float>(h);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int k = tid + s * NT;
        if (k < A) {
            const int fy = k / S::AX, fx = k - fy * S::AX;
            const Two<float>* c = sm.rho1 + (fy + 1) * S::PX + fx + 1;
            const Two<float> r = *c;
            auto nbr = [&](int i) -> Two<float> { return c[L::c(i, 1) * S::PX + L::c(i, 0)]; };
            node_update<L, float>(a, wrap_once(y0 - 2 + fy, ny), nbr, f[s], r.a, r.b);
#pragma unroll
            for (int i = 0; i < L::Q; ++i) sm.f[i][k] = Two<float>{f[s][0][i], f[s][1][i]};
        }
    }
    __syncthreads();

    // second step
    auto pull = [&](int n, float (&g)[2][L::Q]) {  // n: node in the frame of sm.f
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            const Two<float> v = sm.f[i][n - L::c(i, 1) * S::AX - L::c(i, 0)];
            g[0][i] = v.a;
            g[1][i] = v.b;
        }
    };
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int k = tid + s * NT;
        if (k < B) {
            const int ty = k / kPairTX, tx = k - ty * kPairTX;
            pull((ty + 2) * S::AX + tx + 2, f[s]);
            sm.rho2[(ty + 1) * S::BX + tx + 1] = node_densities<L, float>(f[s]);
        }
    }
    if (tid >= NT - RING2) {
        int fx, fy;
        halo_cell<kPairTX, kPairTY>(tid - (NT - RING2), fx, fy);
        float h[2][L::Q];
        pull((fy + 1) * S::AX + fx + 1, h);
        sm.rho2[fy * S::BX + fx] = node_densities<L, float>(h);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int k = tid + s * NT;
        const int ty = k / kPairTX, tx = k - ty * kPairTX;
        const int x = x0 + tx, y = y0 + ty;
        if (k >= B || x >= nx || y >= ny) continue;
        const Two<float>* c = sm.rho2 + (ty + 1) * S::BX + tx + 1;
        const Two<float> r = *c;
        auto nbr = [&](int i) -> Two<float> { return c[L::c(i, 1) * S::BX + L::c(i, 0)]; };
        node_update<L, float>(a, y, nbr, f[s], r.a, r.b);
        store_node<L, float>(a, x, y, 0, f[s], r.a, r.b);
    }
}

template <int NT>
__global__ void __launch_bounds__(NT, 2) sc_d2_pair_kernel(const LatticeArgs<float> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_wait();
    chain_next();
    d2_pair_tile(a, blockIdx.x * kPairTX, blockIdx.y * kPairTY, *reinterpret_cast<PairSmem*>(smem_raw));
}

// The same over the work list of a batch with 32x8 or 32x4 tiles: the CTA of
// every second (fourth) item of a column takes the two-step tile, the others
// have nothing to do.
template <int NT>
__global__ void __launch_bounds__(NT, 2)
    sc_d2_pair_batch_kernel(const BatchLattice<float>* __restrict__ lats, const BatchItem* __restrict__ items, int parity) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const BatchItem w = items[blockIdx.x];
    chain_wait();
    chain_next();
    if (w.y0 % kPairTY != 0) return;
    const LatticeArgs<float> a = lats[w.lat].a[parity];
    d2_pair_tile(a, w.x0, w.y0, *reinterpret_cast<PairSmem*>(smem_raw));
}

// ---- all steps of a call in one cluster ------------------------------------------

// Above about 110^2 nodes the 16 SMs of a cluster are no faster than all of
// them with two steps a launch (us a step: 96^2 2.1 against 3.0, 128^2 3.0 both).
constexpr int kResidentCtas = 16, kResidentThreads = 512;
constexpr long long kResidentNodes = 12288;

// Bands of a lattice's rows: CTA r of n owns rows [ny r / n, ny (r + 1) / n).
__host__ __device__ inline int d2_resident_rows(int ny, int ctas) { return (ny + ctas - 1) / ctas; }
inline size_t d2_resident_smem(int nx, int ny, int ctas) {
    const size_t rows = (size_t)d2_resident_rows(ny, ctas);
    return ((rows + 4) * 2 * D2Q9::Q + (rows + 2)) * (size_t)nx * sizeof(Two<float>);
}

template <int NT>
__global__ void __launch_bounds__(NT, 1) sc_d2_resident_kernel(const LatticeArgs<float> a, int nsteps) {
    namespace cg = cooperative_groups;
    using L = D2Q9;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const cg::cluster_group cluster = cg::this_cluster();
    const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int nx = a.nx, ny = a.ny;
    auto first_row = [&](int r) { return (int)((long long)ny * r / ctas); };
    const int r0 = first_row(rank), rows = first_row(rank + 1) - r0;
    const int up = rank == 0 ? ctas - 1 : rank - 1, down = rank == ctas - 1 ? 0 : rank + 1;
    const int up_rows = first_row(up + 1) - first_row(up);
    const int plane = (d2_resident_rows(ny, ctas) + 4) * nx;  // values per direction and buffer
    Two<float>* const buf = reinterpret_cast<Two<float>*>(smem_raw);  // [2][Q][plane], row l = global row r0 - 2 + l
    Two<float>* const rho = buf + 2 * L::Q * plane;                   // [rows + 2][nx], row l = global row r0 - 1 + l
    Two<float>* const buf_up = cluster.map_shared_rank(buf, up);
    Two<float>* const buf_down = cluster.map_shared_rank(buf, down);
    const int x = threadIdx.x, ty = threadIdx.y, BY = blockDim.y;
    const bool on = x < nx;
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    auto col = [&](int cx) { return cx == 0 ? x : (cx > 0 ? xp : xm); };

    chain_wait();
    chain_next();
    if (on)
        for (int l = ty; l < rows + 4; l += BY) {
            int gy = r0 - 2 + l;
            gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
            const size_t n = cell(a, x, gy, 0);
#pragma unroll
            for (int i = 0; i < L::Q; ++i)
                buf[i * plane + l * nx + x] = Two<float>{a.fin[(size_t)i * (size_t)a.Np + n],
                                                         a.fin[(size_t)(L::Q + i) * (size_t)a.Np + n]};
        }
    cluster.sync();  // every CTA of the cluster runs and holds its rows
#pragma unroll 1
    for (int t = 0; t < nsteps; ++t) {
        const int cur = (t & 1) * L::Q * plane, nxt = L::Q * plane - cur;
        auto pull = [&](int l, float (&f)[2][L::Q]) {
#pragma unroll
            for (int i = 0; i < L::Q; ++i) {
                const Two<float> v = buf[cur + i * plane + (l - L::c(i, 1)) * nx + col(-L::c(i, 0))];
                f[0][i] = v.a;
                f[1][i] = v.b;
            }
        };
        // the pulls of the thread's last row stay in registers for its collision
        float f[2][L::Q];
        int held = -1;
        if (on)
#pragma unroll 1
            for (int l = 1 + ty; l < rows + 3; l += BY) {
                pull(l, f);
                held = l;
                rho[(l - 1) * nx + x] = node_densities<L, float>(f);
            }
        __syncthreads();
        if (on)
#pragma unroll 1
            for (int l = held; l >= 2; l -= BY) {
                if (l >= rows + 2) continue;
                if (l != held) pull(l, f);
                const Two<float> r = rho[(l - 1) * nx + x];
                auto nbr = [&](int i) -> Two<float> { return rho[(l - 1 + L::c(i, 1)) * nx + col(L::c(i, 0))]; };
                const int gy = r0 - 2 + l;
                node_update<L, float>(a, gy, nbr, f, r.a, r.b);
                if (t == nsteps - 1) {
                    store_node<L, float>(a, x, gy, 0, f, r.a, r.b);
                    continue;
                }
                const int to_up = l < 4 ? up_rows + l : -1;             // the upper neighbour's last two rows
                const int to_down = l >= rows ? l - rows : -1;          // the lower neighbour's first two
#pragma unroll
                for (int i = 0; i < L::Q; ++i) {
                    const Two<float> v{f[0][i], f[1][i]};
                    buf[nxt + i * plane + l * nx + x] = v;
                    if (to_up >= 0) buf_up[nxt + i * plane + to_up * nx + x] = v;
                    if (to_down >= 0) buf_down[nxt + i * plane + to_down * nx + x] = v;
                }
            }
        // the neighbours' rows have arrived, and every CTA has read the buffer
        // that the next step writes; after the last step: nobody leaves while a
        // neighbour may still write here
        cluster.sync();
    }
}

}  // namespace lbmsc
