// Host-side launchers of the Shan-Chen kernels, one instantiation per lattice
// (sc_d2q9.cu, sc_d3q19.cu) so the two compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include "sc_common.cuh"

namespace lbmsc {

// Everything a launcher needs to know about one lattice.
struct Plan {
    int lattice;    // 0 D2Q9, 1 D3Q19
    int precision;  // lbm_precision (4, 5: rest-offset 16-bit storage)
    int nx, ny, nz;
    long long N;
    int step_tile;  // index into kTiles for the step kernel
    int step_zchunk;
    int sm_count;   // multiprocessors of the device (persistent grids)
    double tau_A, tau_B, G, ref_A, ref_B;
    double body_A;         // Kolmogorov forcing amplitude (Eq. kolmo); 0 = none
    int forcing;           // kForcingShift or kForcingGuo
    int model;             // kModelSC or kModelFE
    double kappa, gamma;   // FE: gradient coefficient, Gamma
    int px, py, gxo, gyo;  // ghost-padded storage geometry (see LatticeArgs)
    long long Np;          // values per population plane
    int* err;              // device error word (set by a kernel whose bounded wait expired)
    int wait_probe;        // failure-detection test hook (lbm_sc_set_wait_probe); 0 = off
};

// Bytes of one stored element for a precision (lbm_precision): FP64 8, FP32 4,
// reference-offset 16-bit 2, paired rest-offset 16-bit 4 (both species of one
// direction in one word); 0 for an unknown precision.
inline int storage_elem_bytes(int precision) {
    switch (precision) {
        case 0: return 8;
        case 1: return 4;
        case 2:
        case 3: return 2;
        case 4:
        case 5: return 4;
    }
    return 0;
}
inline bool rest_precision(int precision) { return precision == 4 || precision == 5; }
// Population planes of one buffer: 2 Q (a plane per species and direction), or
// Q paired planes for the rest-offset precisions (which add one plane of float2
// densities after them).
inline int population_planes(int lattice, int precision) {
    const int q = lattice == 0 ? 9 : 19;
    return rest_precision(precision) ? q : 2 * q;
}

// Ghost-padded storage geometry for a lattice.  Node x = 0 sits 128 bytes into
// each row and the row pitch is a multiple of 128 bytes, so every warp's row
// segment of a tile starting at a multiple of 32 nodes is whole cache lines
// (a misaligned store would leave partial sectors shared with the next CTA's
// tile).  The ghost columns x = -2, -1, nx, nx+1 and rows y = -2, -1, ny, ny+1
// hold periodic images; on lattices at least a sector wide the images fill the
// whole 32-byte sector on each side of the row (store_node), and the row has
// room for it, which also keeps 16-byte-aligned TMA boxes of x0 - 16 bytes ..
// x0 + TX + 16 bytes inside the row.
inline void storage_geometry(int nx, int ny, int nz, int elem_bytes, int& px, int& py, int& gxo, int& gyo,
                             long long& Np) {
    const int line = 128 / elem_bytes;  // values per 128 bytes
    // right margin: the 32-byte sector of ghost images beyond column nx - 1
    // (store_node), which also covers the 16-byte pad of the TMA boxes
    const int margin = 32 / elem_bytes;
    gxo = line;
    gyo = 2;
    px = (nx + gxo + margin + line - 1) / line * line;
    py = ny + 2 * gyo;
    Np = (long long)px * py * nz;
}

// Tile of one CTA (threads = TX * TY, one (x, y) column each) for the moments
// kernel, and the tiles the step kernel can be launched with (autotuned).
constexpr int kTX = 32;
constexpr int kTY = 8;
// kind 0: register-pipelined kernel (every lattice and precision);
// kind 3: low-register kernel that re-pulls a plane for its collision, with
//         `stages` = CTAs per SM requested from the register allocator;
// kind 4: register-pipelined kernel with three planes of pulls in registers
//         (D3Q19, 32-bit and 16-bit storage), `stages` = CTAs per SM;
// kind 5: TMA-fed kernel with `stages` shared-memory stages (D3Q19, FP32
//         storage, lattices at least one tile wide in x and y), launched as
//         clusters of cx x cy neighbouring tiles (co-scheduled on one GPC, so
//         the halo lines the tiles share are fetched into one die's L2);
// kind 6: the TMA-fed kernel for 16-bit storage (D3Q19; the rest-offset
//         modes also stage boxes of the FP32 node densities).
// Retired ids (kind kRetired) keep their slot so that the other ids stay
// stable; every call that names one is rejected.  They were measured slower
// than the kinds above at every size and removed: 5-7, a persistent kernel
// copying every pull with cp.async into thread-private stages; 8-10, a
// software-pipelined kernel holding two planes in registers and shared memory;
// 26-29, 64x4 / 32x8 TMA tiles with 128-byte or no L2 promotion (no change
// against the 256-byte promotion every kept tile uses).
constexpr int kRetired = -1;
// promo: L2 promotion of the tensor copies (3: 256 bytes fetched per L2 miss);
// minb: CTAs per SM the register allocation is made for (TMA kinds; two
// CTAs per SM let one CTA's per-plane barrier overlap the other's work).
struct TileShape { int tx, ty, kind, stages, cx = 1, cy = 1, promo = 3, minb = 1; };
constexpr int kNumTiles = 45;
constexpr TileShape kTiles[kNumTiles] = {
    {32, 8, 0, 0},       {32, 16, 0, 0},      {64, 8, 0, 0},       {32, 4, 0, 0},       {64, 4, 0, 0},
    {32, 8, kRetired, 0}, {32, 8, kRetired, 0}, {64, 4, kRetired, 0}, {32, 8, kRetired, 0}, {64, 4, kRetired, 0},
    {32, 4, kRetired, 0}, {32, 4, 3, 6},       {32, 8, 3, 3},       {64, 4, 3, 3},       {32, 4, 3, 4},
    {32, 4, 4, 3},       {32, 8, 4, 1},       {16, 8, 4, 3},       {32, 8, 5, 3},       {64, 4, 5, 3},
    {32, 4, 5, 4},       {32, 4, 5, 2},       {64, 4, 5, 3, 1, 2}, {64, 4, 5, 3, 1, 4}, {64, 4, 5, 3, 2, 2},
    {32, 8, 5, 3, 2, 2}, {64, 4, kRetired, 0}, {64, 4, kRetired, 0}, {32, 8, kRetired, 0},
    {32, 8, kRetired, 0}, {64, 4, 6, 3, 1, 2}, {64, 4, 6, 4, 1, 2}, {32, 8, 6, 3},
    {64, 6, 5, 2, 1, 2}, {64, 6, 5, 2},       {64, 6, 6, 3, 1, 2}, {32, 12, 5, 2, 1, 2}, {32, 12, 5, 2},
    {32, 12, 6, 3, 1, 2}, {64, 8, 6, 2, 1, 2}, {48, 8, 5, 2, 1, 2}, {48, 8, 5, 2},
    {64, 4, 6, 2, 1, 2, 3, 2}, {32, 8, 6, 2, 1, 2, 3, 2}, {64, 4, 6, 2, 1, 1, 3, 2}};

// forcing = kForcingGuo or model = kModelFE: the kernels that choose the
// collision at run time (kinds 0 and 3) and the 64x6 TMA tile (34), which has
// a Guo and an FE instantiation.
inline bool tile_supported(int tile, int lattice, int precision, int forcing = kForcingShift, int model = kModelSC) {
    if (tile < 0 || tile >= kNumTiles) return false;
    if ((forcing == kForcingGuo || model == kModelFE) && kTiles[tile].kind != 0 && kTiles[tile].kind != 3 &&
        tile != 34)
        return false;
    switch (kTiles[tile].kind) {
        case 0: return true;
        case 3: return true;
        case 4: return lattice == 1 && precision >= 1 && precision <= 3;
        case 5: return lattice == 1 && precision == 1;
        case 6: return lattice == 1 && precision >= 2 && precision <= 5;
    }
    return false;
}

// Size rules beyond the lattice kind and precision: the TMA boxes need the
// lattice to span at least one tile in x and y.
inline bool tile_fits(int tile, const Plan& p) {
    if (!tile_supported(tile, p.lattice, p.precision, p.forcing, p.model)) return false;
    const TileShape& t = kTiles[tile];
    if (t.kind == 5 || t.kind == 6) {
        const int tiles_x = (p.nx + t.tx - 1) / t.tx, tiles_y = (p.ny + t.ty - 1) / t.ty;
        return p.nx >= t.tx && p.ny >= t.ty && tiles_x % t.cx == 0 && tiles_y % t.cy == 0;
    }
    return true;
}

// Launch of a kernel that begins with chain_wait (sc_common.cuh), as clusters of
// cx x cy CTAs: it may start before the kernel ahead of it in the stream has
// ended.  Steps come out 2 - 3 us shorter (us a step without and with: D2Q9
// 64^2 6.2 / 2.7, 256^2 6.2 / 3.8; D3Q19 FP32 32^3 10.3 / 7.4, 64^3 30.9 / 28.7).
template <class... KA, class... A>
cudaError_t launch_step_kernel(bool chained, void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                               int cx, int cy, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = 0;
    if (chained) {
        cudaLaunchAttribute& a = attr[cfg.numAttrs++];
        a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        a.val.programmaticStreamSerializationAllowed = 1;
    }
    if (cx > 1 || cy > 1) {
        cudaLaunchAttribute& a = attr[cfg.numAttrs++];
        a.id = cudaLaunchAttributeClusterDimension;
        a.val.clusterDim.x = cx;
        a.val.clusterDim.y = cy;
        a.val.clusterDim.z = 1;
    }
    return cudaLaunchKernelEx(&cfg, kern, args...);
}
template <class... KA, class... A>
cudaError_t launch_chained(void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cx, int cy,
                           const A&... args) {
    return launch_step_kernel(true, kern, grid, block, smem, st, cx, cy, args...);
}

// Whether the register kernels (several CTAs per SM) of a D3Q19 lattice are chained.  The next
// step's CTAs are placed while this step's hold their slots, on the SMs that hold
// fewest, and stay there: where the grid leaves slots free but is larger than the
// SMs, some SMs then get two or three of them and others none.  Steps of some
// microseconds gain more from the early launch; the others lose (GB300, us a step,
// chained / not): FP64 56^3, 168 CTAs 371 / 232; FP64 tile 11 96^3 1172 / 805; FP32
// tiles 13, 15 and 3 at 96^3 138 / 109, 122 / 91, 96 / 87; but FP32 30^3 - 48^3 10 - 20 % gained.
// A grid of at most one CTA per SM stays even (FP64 16^3 - 32^3 2 - 8 % gained), and so do
// the kernels with one CTA per SM and the small CTAs of D2Q9.
inline bool chain_pays(const Plan& p, dim3 grid) {
    if (p.lattice == 0 || (long long)grid.x * grid.y * grid.z <= p.sm_count) return true;
    return p.N <= (p.precision == 0 || kTiles[p.step_tile].kind == 3 ? 32768 : 131072);
}
template <class... KA, class... A>
cudaError_t launch_register_kernel(const Plan& p, void (*kern)(KA...), dim3 grid, dim3 block, cudaStream_t st, const A&... args) {
    return launch_step_kernel(chain_pays(p, grid), kern, grid, block, 0, st, 1, 1, args...);
}

struct MomentsOut {
    void* rhoA;
    void* rhoB;
    void* u;
    void* p;
    double* partials;       // per-CTA diagnostics, or null
    double win[5];          // cx, cy, cz, r_in, r_out (r_in < 0: no inner window)
    int zlo = 0, zhi = 0;   // zhi > 0: fields of planes [zlo, zhi) only (D3Q19, no partials)
};

// Grid of the moments kernel over `planes` planes: items of one tile and one z
// chunk, the chunk chosen for the shortest time on 152 SMs with three CTAs each
// (a chunk of zc planes pulls two more), and the CTAs of a diagnostics launch,
// which take the items in turn and leave one record of partial sums each.  In FP64
// an SM's CTAs share its FP64 units, so it counts as one (three a SM gave shorter
// chunks: fields of 5 x 93 x 270 96 us and of 48^3 84, now 86 and 72).  The shape, and with it
// the records' place in a workspace, does not depend on the device.
struct MomentsShape {
    int tiles_x, tiles_y, zchunk, items, ctas;
};
constexpr int kDiagCtas = 152 * 16;
inline MomentsShape moments_shape(const Plan& p, int planes) {
    MomentsShape m;
    m.tiles_x = (p.nx + kTX - 1) / kTX;
    m.tiles_y = (p.ny + kTY - 1) / kTY;
    m.zchunk = 1;
    const long long xy = (long long)m.tiles_x * m.tiles_y, slots = p.precision == 0 ? 152 : 3 * 152;
    long long best = -1;
    if (p.lattice == 1)
        for (int zc = 1; zc <= planes && zc <= 32; ++zc) {
            const long long n = xy * ((planes + zc - 1) / zc), cost = ((n + slots - 1) / slots) * (zc + 2);
            if (best < 0 || cost < best) {
                best = cost;
                m.zchunk = zc;
            }
        }
    m.items = (int)(xy * (p.lattice == 1 ? (planes + m.zchunk - 1) / m.zchunk : 1));
    m.ctas = m.items < kDiagCtas ? m.items : kDiagCtas;
    return m;
}

// Columns of tile 3 in FP64 on a D3Q19 lattice: 16x8 where that covers fewer
// columns outside the lattice than 32x4.
inline void f64_tile3(const Plan& p, int& tx, int& ty) {
    const long long wide = (long long)((p.nx + 31) / 32 * 32) * ((p.ny + 3) / 4 * 4);
    const long long high = (long long)((p.nx + 15) / 16 * 16) * ((p.ny + 7) / 8 * 8);
    tx = high < wide ? 16 : 32;
    ty = high < wide ? 8 : 4;
}

inline dim3 step_grid(const Plan& p) {
    const TileShape t = kTiles[p.step_tile];
    return dim3((unsigned)((p.nx + t.tx - 1) / t.tx), (unsigned)((p.ny + t.ty - 1) / t.ty),
                (unsigned)(p.lattice == 1 ? (p.nz + p.step_zchunk - 1) / p.step_zchunk : 1));
}

// Records of partial sums a diagnostics launch leaves.
inline long long diag_parts(const Plan& p) { return moments_shape(p, p.nz).ctas; }

cudaError_t d2q9_step(const Plan& p, const void* fin, void* fout, cudaStream_t st);
// The tile of an untuned D2Q9 lattice in 32- and 16-bit storage.
constexpr int kTileD2 = 3;
// Several D2Q9 FP32 steps per launch (sc_d2.cuh).  Two steps: lattices at least
// as wide and high as the tile's frame.  nsteps steps (fout may be fin): lattices
// that fit a cluster's shared memory and are small enough to be better off on
// its 16 SMs.
constexpr int kPairTX = 32, kPairTY = 16, kPairThreads = 384;
inline bool d2_pair_fits(const Plan& p) {
    return p.lattice == 0 && p.precision == 1 && p.nx >= kPairTX + 6 && p.ny >= kPairTY + 6;
}
cudaError_t d2q9_pair(const Plan& p, const void* fin, void* fout, cudaStream_t st);
bool d2q9_resident_fits(const Plan& p);
cudaError_t d2q9_resident(const Plan& p, const void* fin, void* fout, int nsteps, cudaStream_t st);
// init of planes [zlo, zhi) (zhi = 0: all planes)
cudaError_t d2q9_init(const Plan& p, const void* rA, const void* rB, const void* u, void* fout,
                      cudaStream_t st, int zlo = 0, int zhi = 0);
cudaError_t d2q9_moments(const Plan& p, const void* fin, const MomentsOut& o, cudaStream_t st);
cudaError_t d3q19_step(const Plan& p, const void* fin, void* fout, cudaStream_t st);
// the step of each storage precision (sc_d3q19_step_*.cu)
cudaError_t d3q19_step_f64(const Plan& p, const void* fin, void* fout, cudaStream_t st);
cudaError_t d3q19_step_f32(const Plan& p, const void* fin, void* fout, cudaStream_t st);
cudaError_t d3q19_step_bf16(const Plan& p, const void* fin, void* fout, cudaStream_t st);
cudaError_t d3q19_step_f16(const Plan& p, const void* fin, void* fout, cudaStream_t st);
cudaError_t d3q19_step_bf16_rest(const Plan& p, const void* fin, void* fout, cudaStream_t st);
cudaError_t d3q19_step_f16_rest(const Plan& p, const void* fin, void* fout, cudaStream_t st);
cudaError_t d3q19_init(const Plan& p, const void* rA, const void* rB, const void* u, void* fout,
                       cudaStream_t st, int zlo = 0, int zhi = 0);
cudaError_t d3q19_moments(const Plan& p, const void* fin, const MomentsOut& o, cudaStream_t st);
cudaError_t diag_finish(const double* partials, long long nparts, double* out, cudaStream_t st);

}  // namespace lbmsc
