// phase_reg_kernel for NQ = 8 float4 groups of atoms per thread.
#include "phase_reg_impl.cuh"

namespace csc {

RegKernel phase_reg_nq8(int block, int cb, bool dense)
{
    return by_form<8>(block, cb, dense);
}

}  // namespace csc
