// phase_reg_kernel for NQ = 4 float4 groups of atoms per thread.
#include "phase_reg_impl.cuh"

namespace csc {

RegKernel phase_reg_nq4(int block, int cb, bool dense)
{
    return by_form<4>(block, cb, dense);
}

}  // namespace csc
