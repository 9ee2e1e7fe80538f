// Choice and launch of the phase kernel with thread-private r (phase_reg_impl.cuh).
#include <algorithm>

#include "csc_internal.cuh"
#include "phase_reg.cuh"

namespace csc {

namespace {

RegKernel reg_kernel(const PhaseConfig &cfg, bool dense)
{
    static RegKernel (*const by_nq[])(int, int, bool) = {
        phase_reg_nq1, phase_reg_nq2, phase_reg_nq3, phase_reg_nq4,
        phase_reg_nq5, phase_reg_nq6, phase_reg_nq7, phase_reg_nq8};
    return by_nq[cfg.reg_nq - 1](cfg.block, cfg.reg_cb, dense);
}

// Blocks per SM of the form with more registers (96 a thread).  Launches of no more
// blocks run it: nothing spills in the chain of updates (K = 25, P = 1, L = 200: T = 7396,
// 18 segments, 21.3 -> 17.6 ms a solve; T = 93,992, 2.47 -> 2.20 ms).  Launches of more,
// and those that drain a queue, run the one with more blocks per SM (T = 5,000,000: 26.7 ms
// with one block per SM, 21.0 with two).
int roomy_blocks(int block)
{
    return block <= 160 ? 4 : block <= 288 ? 2 : 1;
}

int sm_count()
{
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return nsm;
}

}  // namespace

// Groups of at most 8 quads of atoms (one group where K <= 32), cb threads each: at
// least the window, and half the segment where that is more, so that a thread has
// at most two columns (10 segments of 199 columns, L = 16: 1.8x, 2.2x and 2.1x the
// speed of visit_segment with 4, 2 and 1 columns per thread).  Refused where a
// block would need more than 16 column warps or its columns do not fit.
bool phase_reg_config(int K, int L, int w_max, PhaseConfig *cfg)
{
    const int KQ = (K + 3) / 4, W2 = 2 * L - 1;
    const int one = KQ <= 8 ? KQ : 8;
    for (int nq : {one, 4}) {
        const int groups = (KQ + nq - 1) / nq;
        const int cb = std::max((W2 + 31) & ~31, std::min(512 / groups & ~31,
                                                          ((w_max + 1) / 2 + 31) & ~31));
        // (16 column warps; the key's index word holds 5 bits of slot, 10 of class;
        // two bits of the changed mask are the halo's)
        const int ns = (w_max + cb - 1) / cb;
        const size_t smem = phase_reg_smem(nq, groups, L, w_max);
        if (groups * cb > 512 || ns > 30 || groups * nq * 4 > kRegAtoms ||
            smem > (size_t)kPhaseRegSmem)
            continue;
        cfg->reg_nq = nq;
        cfg->reg_ns = ns;
        cfg->reg_cb = cb;
        cfg->block = groups * cb + 32;
        cfg->smem = smem;
        cfg->tile_in_smem = true;
        return true;
    }
    return false;
}

cudaError_t launch_phase_reg(const PhaseParams &pp, const PhaseConfig &cfg, int grid, bool drain,
                             cudaStream_t s)
{
    // (all blocks resident with more registers: the form with more registers)
    RegKernel kern = reg_kernel(cfg, drain || grid > roomy_blocks(cfg.block) * sm_count());
    if (!kern || cfg.reg_cb < 2 * pp.L - 1 || pp.w_max > cfg.reg_ns * cfg.reg_cb ||
        (cfg.block - 32) / cfg.reg_cb * cfg.reg_nq * 4 < pp.K)
        return cudaErrorInvalidConfiguration;
    const cudaError_t e = allow_smem(kern, kPhaseRegSmem);
    if (e != cudaSuccess)
        return e;
    kern<<<grid, cfg.block, cfg.smem, s>>>(pp, cfg.reg_cb, drain ? 1 : 0);
    return cudaGetLastError();
}

int phase_reg_blocks_per_sm(const PhaseConfig &cfg)
{
    int per_sm = 1;
    RegKernel kern = reg_kernel(cfg, true);
    if (kern) {
        allow_smem(kern, kPhaseRegSmem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, cfg.block, cfg.smem);
    }
    return per_sm;
}

}  // namespace csc
