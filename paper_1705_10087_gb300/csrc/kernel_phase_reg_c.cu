// phase_reg_kernel for NQ = 5, 6 float4 groups of atoms per thread.
#include "phase_reg_impl.cuh"

namespace csc {

RegKernel phase_reg_nq5(int block, int cb, bool dense)
{
    return by_form<5>(block, cb, dense);
}

RegKernel phase_reg_nq6(int block, int cb, bool dense)
{
    return by_form<6>(block, cb, dense);
}

}  // namespace csc
