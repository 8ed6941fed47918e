// D2Q9 instantiations of the fused Shan-Chen kernels.
#include <atomic>

#include "sc_instantiate.cuh"
#include "sc_d2.cuh"

namespace lbmsc {
cudaError_t d2q9_step(const Plan& p, const void* fin, void* fout, cudaStream_t st) {
    return step_any<D2Q9>(p, fin, fout, st);
}
cudaError_t d2q9_pair(const Plan& p, const void* fin, void* fout, cudaStream_t st) {
    const cudaError_t e =
        cudaFuncSetAttribute(sc_d2_pair_kernel<kPairThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PairSmem));
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((p.nx + kPairTX - 1) / kPairTX), (unsigned)((p.ny + kPairTY - 1) / kPairTY));
    return launch_chained(sc_d2_pair_kernel<kPairThreads>, grid, dim3(kPairThreads), sizeof(PairSmem), st, 1, 1,
                          make_args<float>(p, fin, fout));
}

namespace {

constexpr size_t kSmemPerCta = 227 * 1024;

// Clusters of 16 CTAs with a whole SM each are opt-in: asked once per device.
bool resident_allowed() {
    static std::atomic<int> known[64];  // 0 unknown, 1 yes, 2 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    const int k = known[dev].load(std::memory_order_acquire);
    if (k != 0) return k == 1;
    bool ok = cudaFuncSetAttribute(sc_d2_resident_kernel<kResidentThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kSmemPerCta) == cudaSuccess &&
              cudaFuncSetAttribute(sc_d2_resident_kernel<kResidentThreads>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    if (ok) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kResidentCtas);
        cfg.blockDim = dim3(kResidentThreads);
        cfg.dynamicSmemBytes = kSmemPerCta;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kResidentCtas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        ok = cudaOccupancyMaxActiveClusters(&n, sc_d2_resident_kernel<kResidentThreads>, &cfg) == cudaSuccess && n >= 1;
    }
    if (!ok) cudaGetLastError();
    known[dev].store(ok ? 1 : 2, std::memory_order_release);
    return ok;
}

int resident_ctas(const Plan& p) { return p.ny / 2 < kResidentCtas ? p.ny / 2 : kResidentCtas; }

// Threads of a CTA: a row of warps along x, as many rows as fit (no more than the band and its halo).
dim3 resident_block(const Plan& p, int ctas) {
    const int bx = (p.nx + 31) / 32 * 32, rows = d2_resident_rows(p.ny, ctas) + 2;
    const int by = kResidentThreads / bx;
    return dim3(bx, by < rows ? by : rows);
}

// Passes of a CTA over its band's rows in a step, at most.  One pass costs about 1.5 us, so
// tall narrow lattices, a warp per row, are better off on all SMs: us for 3 / 5 / 100
// steps, 400 x 30 (two passes) 13 / 18 / 249 and 9 / 15 / 271 on all SMs, 300 x 40 (three) 15 / 21 /
// 325 and 9 / 15 / 295, 1000 x 8 (five) 23 / 32 / 451 and 11 / 18 / 354 (one launch a step
// before chained launches: 19 / 31 / 615).
constexpr int kResidentPasses = 3;

}  // namespace

bool d2q9_resident_fits(const Plan& p) {
    const int ctas = resident_ctas(p);
    if (p.lattice != 0 || p.precision != 1 || p.nx > kResidentThreads || ctas < 1 || p.N > kResidentNodes) return false;
    const int by = (int)resident_block(p, ctas).y;
    return (d2_resident_rows(p.ny, ctas) + 2 + by - 1) / by <= kResidentPasses &&
           d2_resident_smem(p.nx, p.ny, ctas) <= kSmemPerCta && resident_allowed();
}

cudaError_t d2q9_resident(const Plan& p, const void* fin, void* fout, int nsteps, cudaStream_t st) {
    const int ctas = resident_ctas(p);
    return launch_chained(sc_d2_resident_kernel<kResidentThreads>, dim3((unsigned)ctas), resident_block(p, ctas),
                          d2_resident_smem(p.nx, p.ny, ctas), st, ctas, 1, make_args<float>(p, fin, fout), nsteps);
}

cudaError_t d2q9_init(const Plan& p, const void* rA, const void* rB, const void* u, void* fout, cudaStream_t st,
                      int zlo, int zhi) {
    return init_any<D2Q9>(p, rA, rB, u, fout, st, zlo, zhi);
}
cudaError_t d2q9_moments(const Plan& p, const void* fin, const MomentsOut& o, cudaStream_t st) {
    return moments_any<D2Q9>(p, fin, o, st);
}
cudaError_t diag_finish(const double* partials, long long nparts, double* out, cudaStream_t st) {
    sc_diag_finish_kernel<256><<<kNumDiag, 256, 0, st>>>(partials, nparts, out);
    return cudaGetLastError();
}
}  // namespace lbmsc
