// The phase kernel with thread-private r in shared memory (phase_reg_impl.cuh), chosen
// by phase_config (kernel_phase.cu) and launched through launch_phase and
// launch_phase_drain.
#pragma once

#include "csc_internal.cuh"

namespace csc {

// Fills cfg (reg_nq > 0) when a block's threads and shared memory hold a segment of
// w_max columns; false where phase_kernel must run.
bool phase_reg_config(int K, int L, int w_max, PhaseConfig *cfg);
cudaError_t launch_phase_reg(const PhaseParams &pp, const PhaseConfig &cfg, int grid, bool drain,
                             cudaStream_t s);
int phase_reg_blocks_per_sm(const PhaseConfig &cfg);

// The kernel for nq = 1 .. 8 float4 groups of atoms per thread, blocks of `block`
// threads and cb threads per group of atoms (kernel_phase_reg_*.cu).
using RegKernel = void (*)(PhaseParams, int, int);
RegKernel phase_reg_nq1(int block, int cb, bool dense);
RegKernel phase_reg_nq2(int block, int cb, bool dense);
RegKernel phase_reg_nq3(int block, int cb, bool dense);
RegKernel phase_reg_nq4(int block, int cb, bool dense);
RegKernel phase_reg_nq5(int block, int cb, bool dense);
RegKernel phase_reg_nq6(int block, int cb, bool dense);
RegKernel phase_reg_nq7(int block, int cb, bool dense);
RegKernel phase_reg_nq8(int block, int cb, bool dense);

constexpr int kPhaseRegSmem = kMaxSmem - 8192;  // dynamic shared memory at most (static: 5 KB)
constexpr int kRegAtoms = 256;  // atoms of all groups at most, padded to whole groups
// Shared memory (bytes) per group of atoms: the halo of 2 (L-1) columns, the own
// columns, and per own column a key and the bits of its listed and unlisted
// nonzeros.  A column takes NQ | 1 quads (an odd stride: 128-bit accesses without
// bank conflicts).
__host__ __device__ constexpr size_t phase_reg_smem(int nq, int groups, int L, int w)
{
    const size_t col = 16 * (size_t)(nq | 1);
    return groups * ((2 * (size_t)(L - 1) + w) * col + 16 * (size_t)w);
}

}  // namespace csc
