// phase_reg_kernel for NQ = 1, 2, 3 float4 groups of atoms per thread.
#include "phase_reg_impl.cuh"

namespace csc {

RegKernel phase_reg_nq1(int block, int cb, bool dense)
{
    return by_form<1>(block, cb, dense);
}

RegKernel phase_reg_nq2(int block, int cb, bool dense)
{
    return by_form<2>(block, cb, dense);
}

RegKernel phase_reg_nq3(int block, int cb, bool dense)
{
    return by_form<3>(block, cb, dense);
}

}  // namespace csc
